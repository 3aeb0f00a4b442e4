"""GPU parity of the wide path at the edges of its 32-bit elements: values and
differences that just fit and just do not, sizes with P in and out of shared
memory, every tabu criterion, forced thread counts, batches that mix widths."""
import numpy as np
import pytest

import oracle
import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu

FIELDS = ["best_p", "best_cost", "final_cost", "best_iter", "iters_done", "status", "hash",
          "descent_hash", "descent_moves"]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    oracle.build()
    q.lib()
    return torch


def check(F, D, W, threads=0, penalty=0, **kw):
    with q.Instance(F, D) as inst:
        assert inst.info["flow_bytes"] == 8 and inst.info["dist_bytes"] == 8
        g = inst.search(q.make_params(W, threads_per_walk=threads, freq_penalty=penalty, **kw))
        P = np.stack([np.random.default_rng(k).permutation(len(F)).astype(np.int32)
                      for k in range(5)])
        costs = inst.cost(P)
    o = oracle.run_walks(F, D, W, penalty=penalty, **kw)
    for f in FIELDS:
        assert np.array_equal(g[f].astype(np.int64), o[f].astype(np.int64)), f
    assert np.array_equal(costs, [(F * D[np.ix_(p, p)]).sum() for p in P])


# the span of the values: just inside 30 bits, just beyond, at int32's ends
@pytest.mark.parametrize("lo,hi", [(0, 2 ** 30 - 1), (0, 2 ** 30), (-2 ** 29, 2 ** 29 - 1),
                                   (2 ** 31 - 2 ** 20, 2 ** 31 - 1), (2 ** 31 - 5, 2 ** 31),
                                   (-2 ** 31 + 1, -2 ** 31 + 2 ** 20), (-2 ** 31, -2 ** 31 + 9)])
@pytest.mark.parametrize("sym", [False, True])
def test_values_at_the_edges(lo, hi, sym):
    n = 23
    rng = np.random.default_rng(abs(lo) % 1000 + sym)
    F = rng.integers(lo, hi + 1, size=(n, n))
    D = rng.integers(0, 2000, size=(n, n))
    F[0, 1], F[1, 2] = lo, hi
    if sym:
        F, D = np.triu(F) + np.triu(F, 1).T, np.triu(D) + np.triu(D, 1).T
    check(F, D, 3, seed=3, iters=120, tenure=(2, 9, 0), descend=True)
    check(D, F, 3, seed=4, iters=120, tenure=instances.periodic_tenure(n))


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 31, 33, 61, 64, 65, 100, 119, 120, 127, 129, 160, 181,
                               182, 225, 256])
def test_sizes(n, sym):
    F, _ = instances.uniform_instance(n, 4000 + n, sym, 0, 1_000_000)
    _, D = instances.uniform_instance(n, 4100 + n, sym, 0, 10_000)
    crit = n % 3
    check(F, D, 2, seed=5, iters=60, tenure=instances.paper_tenure(n), descend=n % 2 == 0,
          max_descent=20, criterion=crit, penalty=2 if crit == 1 else 0)


@pytest.mark.parametrize("threads", [128, 256, 512, 1024])
def test_thread_counts(threads):
    F, _ = instances.uniform_instance(41, 4200, False, 0, 1_000_000)
    _, D = instances.uniform_instance(41, 4201, False, -5_000, 10_000)
    check(F, D, 3, threads=threads, seed=6, iters=100, tenure=(3, 9, 0))


def test_batch_of_several_widths():
    """One width for the whole batch: int32 only when every instance fits."""
    for top in (10_000, 2 ** 31 + 5):
        Fs, Ds = [], []
        for k, n in enumerate([12, 37, 50]):
            F, D = instances.uniform_instance(n, 4300 + k, symmetric=(k % 2 == 0))
            if k == 1:
                F = F * 1000
            if k == 2:
                D[0, 1] = D[1, 0] = top
            Fs.append(F)
            Ds.append(D)
        with q.Batch(Fs, Ds) as b:
            assert b.info["delta_bytes"] == 8
            g = b.search(q.make_params(3, seed=14, iters=120, tenure=(4, 10, 0), descend=True))
        for i, (F, D) in enumerate(zip(Fs, Ds)):
            o = oracle.run_walks(F, D, 3, seed=14, iters=120, tenure=(4, 10, 0), descend=True)
            for f in FIELDS[1:]:
                assert np.array_equal(g[f][3 * i:3 * i + 3].astype(np.int64),
                                      o[f].astype(np.int64)), (top, i, f)
