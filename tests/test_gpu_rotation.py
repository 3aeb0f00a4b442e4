"""GPU parity of the rotation layout (int8 flows, phase X from the maintained
products): sizes at the edges of its circle, its warps and its arrays, tenures
at the edges of its ring, and pairs applied while tabu whose new end equals
an old one.  Every walk equals the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu

FIELDS = ["best_p", "best_cost", "final_cost", "best_iter", "iters_done", "status",
          "descent_moves", "hash", "descent_hash"]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    oracle.build()
    q.lib()
    return torch


def check(F, D, W, threads=0, flow_bytes=1, **kw):
    with q.Instance(F, D) as inst:
        assert inst.info["flow_bytes"] == flow_bytes
        g = inst.search(q.make_params(W, threads_per_walk=threads, **kw))
    o = oracle.run_walks(F, D, W, **kw)
    for k in FIELDS:
        assert np.array_equal(g[k].astype(np.int64), o[k].astype(np.int64)), k


# the smallest circles, even and odd n, a block count that C divides and not,
# the last n of a warp of phase X, of the fixed arrays, and of a plan; n = 40:
# the triangle of marks ends on a 16-byte boundary
@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("n", [3, 4, 5, 6, 7, 9, 16, 31, 32, 33, 40, 49, 57, 63, 64, 65, 85, 99,
                               104, 105, 127, 128, 129, 138, 145, 149, 151, 157, 160])
def test_sizes(n, sym):
    F, D = instances.uniform_instance(n, 2000 + n, symmetric=sym)
    np.fill_diagonal(F, np.arange(n) % 7)  # diagonal terms count too
    np.fill_diagonal(D, np.arange(n) % 5)
    check(F, D, 3, seed=5, iters=150, tenure=instances.periodic_tenure(n), descend=True)


# int16 flows: skewed values (costs in 64 bits from n of about 50 on), and
# flows a few times a byte's range on a dense instance with a diagonal
@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("n", [5, 16, 31, 33, 40, 64, 65, 90, 99, 100, 104, 127, 129, 140, 150,
                               151])
def test_int16_flows(n, sym):
    F, D = instances.lognormal_instance(n, 2600 + n, sym)
    F[0, n - 1] = F[n - 1, 0] = 700  # beyond a byte whatever the draw
    check(F, D, 3, flow_bytes=2, seed=5, iters=150, tenure=instances.periodic_tenure(n),
          descend=True)
    if n <= 65:
        F, D = instances.uniform_instance(n, 2700 + n, symmetric=sym, lo=-150, hi=150)
        _, D = instances.uniform_instance(n, 2800 + n, symmetric=sym, lo=-20, hi=60)
        np.fill_diagonal(F, np.arange(n) - 7)
        np.fill_diagonal(D, np.arange(n) % 9)
        check(F, D, 3, flow_bytes=2, seed=6, iters=200, tenure=instances.paper_tenure(n))


def test_int16_flows_at_the_key_bound():
    """Flows scaled up to the largest values that the scan's candidates hold
    and past them: the walks do not change their kind of answer."""
    F, D = instances.uniform_instance(26, 2900, symmetric=False, lo=1)
    for scale in (2, 9, 14, 15, 16, 17, 20, 40):
        check(F * scale, D, 3, flow_bytes=2, seed=7, iters=200, tenure=(3, 9, 0), descend=True)


@pytest.mark.parametrize("threads", [128, 256, 512, 1024])
@pytest.mark.parametrize("n", [12, 37, 60])
def test_thread_counts(n, threads):
    F, D = instances.uniform_instance(n, 2100 + n, symmetric=n % 2 == 0)
    if threads == 128 and n > 52:
        pytest.skip("128 threads hold n up to 52")
    check(F, D, 3, threads=threads, seed=6, iters=200, tenure=instances.paper_tenure(n))


# M in the workspace: the sizes at the edges of its plans, of its warps and of
# its marks, with the frequency memory, both tenure rules, 2opt first
@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("n", [182, 183, 191, 192, 193, 200, 205, 217, 229, 252, 253, 255, 256])
def test_large_n(n, sym):
    F, D = instances.uniform_instance(n, 3000 + n, symmetric=sym)
    np.fill_diagonal(F, np.arange(n) % 7)
    np.fill_diagonal(D, np.arange(n) % 5)
    kw = dict(seed=5, iters=120, tenure=instances.periodic_tenure(n), descend=n % 2 == 0,
              max_descent=40)
    check(F, D, 3, **kw)
    check(F, D, 2, seed=6, iters=300, tenure=(1, 9, 0))
    with q.Instance(F, D) as inst:
        prm = q.make_params(2, **kw)
        assert inst.plan(prm)["workspace"] == 1
        g = inst.search(prm, freq=True)
        assert (g["freq"].sum(axis=(1, 2)) == g["iters_done"]).all()


@pytest.mark.parametrize("tmax", [300, 510, 511])
def test_large_n_long_tenures(tmax):
    F, D = instances.grid_instance(190, 3300)
    check(F, D, 2, seed=14, iters=800, tenure=(tmax - 3, tmax, 0))


def test_large_n_in_batches_and_from_several_walks(gpu):
    """Batches take M's workspace from n = 152 on; more walks than CTAs."""
    ns = [30, 152, 163, 181, 182, 220]
    pairs = [instances.uniform_instance(n, 3400 + n, symmetric=n % 2 == 0) for n in ns]
    with q.Batch([F for F, _ in pairs], [D for _, D in pairs]) as b:
        for tn in ((5, 30, 0), (500, 600, 0), (90, 110, 200)):
            per_n = tn[0] == 90
            g = b.search(q.make_params(3, seed=15, iters=100, tenure=tn, tenure_per_n=per_n))
            for i, (F, D) in enumerate(pairs):
                t = instances.periodic_tenure(ns[i]) if per_n else tn
                o = oracle.run_walks(F, D, 3, seed=15, iters=100, tenure=t)
                for k in FIELDS[1:]:
                    assert np.array_equal(g[k][3 * i:3 * i + 3].astype(np.int64),
                                          o[k].astype(np.int64)), (i, k)
    F, D = pairs[-1]
    W = 2 * gpu.cuda.get_device_properties(0).multi_processor_count + 5
    with q.Instance(F, D) as inst:
        g = inst.search(q.make_params(W, seed=16, iters=60, tenure=(5, 30, 0)))
    o = oracle.run_walks(F, D, 3, seed=16, iters=60, tenure=(5, 30, 0),
                         walk_ids=np.array([0, W // 2, W - 1]))
    for k in FIELDS:
        assert np.array_equal(g[k][[0, W // 2, W - 1]].astype(np.int64), o[k].astype(np.int64)), k


# tabu times of one and two iterations: slots that are on the ring for none, or
# read right after they were hung
@pytest.mark.parametrize("n", [8, 23, 50, 70, 100, 139, 190])
@pytest.mark.parametrize("tmax", [1, 2, 3])
def test_shortest_tenures(n, tmax):
    F, D = instances.uniform_instance(n, 2300 + n, symmetric=n % 2 == 0)
    check(F, D, 3, seed=17, iters=200, tenure=(1, tmax, 0))


# many ties (small values), short random tenures with aspiration: pairs are
# applied again while tabu, ends coincide
@pytest.mark.parametrize("n,hi", [(14, 3), (30, 99), (50, 9), (100, 99), (100, 2), (130, 99)])
def test_short_random_tenures(n, hi):
    F, D = instances.uniform_instance(n, 2200 + n, symmetric=hi < 10, hi=hi)
    check(F, D, 4, seed=13, iters=600, tenure=(1, 9, 0))


# the longest tenure of the ring (254 and 510 iterations) and one more, which
# the row layout takes; a walk whose every pair turns tabu
@pytest.mark.parametrize("n,tmax,iters", [(30, 254, 700), (30, 255, 700), (110, 510, 1100),
                                          (110, 511, 1100), (12, 200, 400)])
def test_long_tenures(n, tmax, iters):
    F, D = instances.uniform_instance(n, 2300 + n, symmetric=True)
    check(F, D, 2, seed=14, iters=iters, tenure=(tmax - 3, tmax, 0))


def test_batch_changes_layout_with_the_tenure(gpu):
    """One batch, searched with tenures the ring holds and then longer ones."""
    ns = [20, 33, 50, 77, 104]
    pairs = [instances.uniform_instance(n, 2400 + n, symmetric=n % 2 == 0) for n in ns]
    with q.Batch([F for F, _ in pairs], [D for _, D in pairs]) as b:
        for tn in ((5, 30, 0), (250, 300, 0), (500, 600, 0), (5, 30, 0)):
            g = b.search(q.make_params(3, seed=15, iters=120, tenure=tn, descend=True))
            for i, (F, D) in enumerate(pairs):
                o = oracle.run_walks(F, D, 3, seed=15, iters=120, tenure=tn, descend=True)
                for k in FIELDS[1:]:
                    assert np.array_equal(g[k][3 * i:3 * i + 3].astype(np.int64),
                                          o[k].astype(np.int64)), (i, k)
