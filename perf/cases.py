"""What the library's performance is measured on: searches, cost evaluations, batches
and served requests through the package's public calls, from the smallest call
to the largest launch that the benchmark workloads make.

A case is a dict of plain values.  ``kind`` says which entry point it takes:

* ``search``  one instance: ``Instance.search_async`` into device buffers that
              the caller keeps (``blocking``: ``Instance.search``, host results)
* ``batch``   many instances of uneven n: ``Batch.search_async``
* ``cost``    ``Instance.cost`` of many permutations (host data)
* ``serve``   a burst of requests through ``Server.submit`` and ``Server.wait``

Instances come from ``paper_2307_11248_gb300.instances`` (the generators that
the benchmark and the tests use) and from one with values beyond the narrow
element paths.  Tabu tenures: ``periodic`` is [0.9 n, 1.1 n] redrawn every 2n
iterations, ``paper`` is [0.1 n, 0.33 n] redrawn at every move.
"""
import numpy as np
import torch

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

FIELDS = ("best_p", "best_cost", "final_cost", "best_iter", "iters_done", "status",
          "descent_moves", "hash", "descent_hash")

SEARCH = dict(kind="search", family="asym", n=50, walks=256, iters=5000, descend=False,
              tenure="periodic", criterion=0, penalty=0, blocking=False)


def _search(name, **kw):
    return dict(SEARCH, name=name, **kw)


def listed():
    return [
        # The latency case: 2opt from 32 starts on a tiny instance (the
        # benchmark's sym12 workload), where launch and set-up count.
        _search("descend_sym12", family="sym", n=12, walks=32, iters=0, descend=True),
        # A small odd instance solved by one blocking call with host results,
        # the paper's own tenure rule: what a script calls in a loop.
        _search("paper_asym23_blocking", n=23, walks=100, iters=1000, tenure="paper",
                blocking=True),
        # The benchmark's asym50 workload: asymmetric uniform values, 256 walks.
        _search("tabu_asym50"),
        # The benchmark's grid100 workload: 2opt, then tabu, 1024 walks of a
        # sparse symmetric facility layout; the many-walk throughput case.
        _search("grid100", family="grid", n=100, walks=1024, iters=10000, descend=True),
        # An odd size past 128 with about one walk for each SM.
        _search("tabu_asym139", n=139, walks=150, iters=2000),
        # The largest instances the library takes, few walks, one long
        # request: a symmetric layout and a ragged asymmetric one.
        _search("grid256", family="grid", n=256, walks=64, iters=1000, descend=True),
        _search("tabu_asym203", n=203, walks=48, iters=1000, tenure="paper"),
        # Values beyond int16 and int8: the int64 element path.
        _search("tabu_wide61", family="wide", n=61, walks=160, iters=1000),
        # The other tabu criterion with the frequency penalty.
        _search("rules_sym47", family="sym", n=47, walks=160, iters=2000, tenure="paper",
                criterion=1, penalty=3),
        # A cut of the benchmark's batch512 workload: skewed flows, sizes
        # uniform in [20, 150], int64 costs, 64 walks each.
        dict(name="batch_lognormal", kind="batch", count=96, nmin=20, nmax=150, walks=64,
             iters=1000, tenure="periodic"),
        # Eq. 1 for many candidate permutations, host to host.
        dict(name="cost_n100", kind="cost", family="sym", n=100, perms=20000),
        # The request stream of the serving workload as one burst: n uniform
        # in [12, 256], three families, 32 walks each.
        dict(name="serve_burst", kind="serve", count=24, nmin=12, nmax=256, walks=32, iters=500),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["search"] * 7 + ["batch", "cost", "serve"])
    if kind == "batch":
        nmin = rng.randint(12, 60)
        return dict(kind="batch", count=_log_int(rng, 4, 96), nmin=nmin,
                    nmax=rng.randint(nmin + 1, 150), walks=rng.randint(8, 64),
                    iters=_log_int(rng, 100, 1000), tenure=rng.choice(["periodic", "paper"]))
    if kind == "cost":
        return dict(kind="cost", family=rng.choice(["sym", "asym", "grid"]),
                    n=_log_int(rng, 8, 256), perms=_log_int(rng, 100, 20000))
    if kind == "serve":
        nmin = rng.randint(12, 100)
        return dict(kind="serve", count=rng.randint(6, 24), nmin=nmin,
                    nmax=rng.randint(nmin + 1, 256), walks=32, iters=_log_int(rng, 100, 500))
    family = rng.choice(["sym", "asym", "grid", "sym", "asym", "grid", "lognormal", "wide"])
    n = _log_int(rng, 8, 256 if family not in ("lognormal", "wide") else 120)
    walks = _log_int(rng, 8, 1024)
    # no more evaluations than the largest listed case: 1024 walks of n = 100
    # make 10^4 iterations; the slower paths get less
    most = 2.0e10 / (walks * n * (n - 1) / 2)
    if family in ("lognormal", "wide") or n > 181:
        most /= 30
    iters = max(20, min(int(most), _log_int(rng, 100, 5000)))
    crit = rng.choice([0, 0, 0, 0, 0, 1, 2])
    return dict(SEARCH, family=family, n=n, walks=walks, iters=iters,
                descend=rng.random() < 0.4, tenure=rng.choice(["periodic", "paper"]),
                criterion=crit, penalty=rng.choice([0, 2]) if crit else 0,
                blocking=rng.random() < 0.3)


def _instance(family, n, seed):
    if family == "sym":
        return instances.uniform_instance(n, seed, True)
    if family == "asym":
        return instances.uniform_instance(n, seed, False)
    if family == "grid":
        return instances.grid_instance(n, seed)
    if family == "lognormal":
        return instances.lognormal_instance(n, seed, seed % 2 == 0)
    F, _ = instances.uniform_instance(n, seed, False, 0, 1_000_000)
    _, D = instances.uniform_instance(n, seed + 1, False, 0, 10_000)
    return F, D


def _tenure(rule, n):
    return instances.periodic_tenure(n) if rule == "periodic" else instances.paper_tenure(n)


def _per_n(rule):
    return (90, 110, 200) if rule == "periodic" else (10, 33, 0)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        F, D = _instance(case["family"], case["n"], seed)
        inst = q.Instance(F, D)
        prm = q.make_params(case["walks"], seed=seed + 1000, iters=case["iters"],
                            tenure=_tenure(case["tenure"], case["n"]), descend=case["descend"],
                            criterion=case["criterion"], freq_penalty=case["penalty"])
        outs = None if case["blocking"] else inst.device_outputs(case["walks"])
        return dict(kind=kind, inst=inst, prm=prm, outs=outs)
    if kind == "batch":
        # as instances.batch_instances, alternately symmetric and asymmetric
        pairs = [instances.lognormal_instance(n, seed * 1_000_003 + k + 1, k % 2 == 0)
                 for k, n in enumerate(_sizes(case))]
        batch = q.Batch([F for F, _ in pairs], [D for _, D in pairs])
        prm = q.make_params(case["walks"], seed=seed + 1000, iters=case["iters"],
                            tenure=_per_n(case["tenure"]), tenure_per_n=True)
        return dict(kind=kind, batch=batch, prm=prm, outs=batch.device_outputs(case["walks"]))
    if kind == "cost":
        F, D, perms = _cost_data(case, seed)
        return dict(kind=kind, inst=q.Instance(F, D), perms=perms)
    # as instances.poisson_requests: the three families in turn
    work = []
    for k, n in enumerate(_sizes(case)):
        F, D = _instance(("sym", "asym", "grid")[k % 3], n, seed * 1_000_003 + k + 1)
        work.append((F, D, q.make_params(case["walks"], seed=seed + k, iters=case["iters"],
                                         tenure=instances.periodic_tenure(n))))
    return dict(kind=kind, server=q.Server(slots=64, mem_bytes=1 << 28), work=work)


def _sizes(case):
    """Sizes of a batch's or a burst's instances: the case's own, whatever the seed."""
    lo, hi, count = case["nmin"], case["nmax"], case["count"]
    rng = np.random.default_rng([count, lo, hi])
    return [int(n) for n in rng.integers(lo, hi + 1, size=count)]


def _cost_data(case, seed):
    F, D = _instance(case["family"], case["n"], seed)
    rng = np.random.default_rng(seed)
    perms = rng.permuted(np.tile(np.arange(case["n"], dtype=np.int32), (case["perms"], 1)), axis=1)
    return F, D, perms


def run(state):
    kind = state["kind"]
    if kind == "search":
        if state["outs"] is None:
            return state["inst"].search(state["prm"])
        state["inst"].search_async(state["prm"], state["outs"])
        return state["outs"]
    if kind == "batch":
        state["batch"].search_async(state["prm"], state["outs"])
        return state["outs"]
    if kind == "cost":
        return state["inst"].cost(state["perms"])
    server = state["server"]
    tickets = [server.submit(F, D, prm) for F, D, prm in state["work"]]
    results = [server.wait(t)[0] for t in tickets]
    return {k: np.concatenate([r[k].reshape(-1) for r in results]) for k in FIELDS}


def _search_work(n, walks, iters, descend, elem):
    # instance in, per-walk results out; one O(1) delta update (two products
    # of differences and their sum, 8 operations) per pair and iteration; a
    # 2opt descent makes about n moves
    moves = iters + (n if descend else 0)
    return 2 * n * n * elem + walks * (4 * n + 48), 8.0 * walks * moves * n * (n - 1) / 2


def work(case):
    kind = case["kind"]
    if kind == "search":
        elem = {"lognormal": 1.5, "wide": 8}.get(case["family"], 1)
        by, fl = _search_work(case["n"], case["walks"], case["iters"], case["descend"], elem)
    elif kind in ("batch", "serve"):
        per = [_search_work(n, case["walks"], case["iters"], False, 1.5 if kind == "batch" else 1)
               for n in _sizes(case)]
        by, fl = sum(p[0] for p in per), sum(p[1] for p in per)
    else:
        n = case["n"]
        by = 2 * n * n + case["perms"] * (4 * n + 8)
        fl = 2.0 * case["perms"] * n * n
    return {"bytes": by, "flops": fl}


def exact(case, seed):
    # Every output is a whole number.  Costs have a plain numpy value; the
    # searches' are trajectories, which no short expression gives.
    if case["kind"] != "cost":
        return None
    F, D, perms = _cost_data(case, seed)
    return np.array([int((F * D[p[:, None], p[None, :]]).sum()) for p in perms], dtype=np.int64)
