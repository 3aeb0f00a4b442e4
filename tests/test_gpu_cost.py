"""GPU costs of given permutations (Eq. 1) at the edges of the kernel's columns
and warps, for every element width, and rows that are no permutation."""
import numpy as np
import pytest

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    q.lib()
    return torch


def instance(n, width):
    rng = np.random.default_rng(100 * n + width)
    if width == 1:
        lim_f, lim_d = (-27, 101), (-128, 0)  # their differences fit a byte
    elif width == 2:  # up to the largest values that the narrow elements hold
        lim_f, lim_d = (-32768, 32768), (-128, 128)
        if 2 * n * 32768 * 128 >= 2 ** 31:
            m = (2 ** 31 - 1) // (2 * n * 128)
            lim_f = (-m, m + 1)
    else:
        lim_f, lim_d = (0, 1_000_000), (0, 10_000)
    F, D = rng.integers(*lim_f, (n, n)), rng.integers(*lim_d, (n, n))
    F[0, n - 1], D[n - 1, 0] = lim_f[1] - 1, lim_d[1] - 1
    return F.astype(np.int64), D.astype(np.int64)


def perms(n, count, seed=1):
    rng = np.random.default_rng(seed)
    return rng.permuted(np.tile(np.arange(n, dtype=np.int32), (count, 1)), axis=1)


@pytest.mark.parametrize("width", [1, 2, 8])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 31, 32, 33, 63, 99, 100, 127, 128, 129, 130, 255, 256])
def test_costs(n, width):
    F, D = instance(n, width)
    P = perms(n, 67)
    with q.Instance(F, D) as inst:
        assert inst.info["flow_bytes"] == width
        got = [inst.cost(P[:k]) for k in (1, 16, 17, 67)]
    want = np.array([(F * D[np.ix_(p, p)]).sum() for p in P])
    for g in got:
        assert np.array_equal(g, want[:len(g)])


def test_more_permutations_than_the_grid_holds_at_once():
    F, D = instances.uniform_instance(40, 5, symmetric=False)
    P = perms(40, 30000)
    with q.Instance(F, D) as inst:
        got = inst.cost(P)
    pick = np.r_[0:20, 15000:15020, 29980:30000]
    assert np.array_equal(got[pick], [(F * D[np.ix_(p, p)]).sum() for p in P[pick]])


@pytest.mark.parametrize("width", [1, 2, 8])
@pytest.mark.parametrize("n", [2, 33, 128, 256])
def test_rows_that_are_no_permutation(n, width):
    """A repeated, a negative and a too large entry, wherever they stand: an
    error, and the outputs stay as they were."""
    F, D = instance(n, width)
    with q.Instance(F, D) as inst:
        for row in (0, 17, 39):
            for at in (0, n // 2, n - 1):
                for value in (None, -1, n, 2 ** 31 - 1, -2 ** 31):
                    P = perms(n, 40)
                    P[row, at] = P[row, at - 1] if value is None else value
                    out = np.full(40, -7, np.int64)
                    st = q.lib().qap_cost(inst.h, 40, P.ctypes.data, out.ctypes.data)
                    assert st == 1, (row, at, value, st)
                    assert (out == -7).all()
        P = perms(n, 40)
        assert np.array_equal(inst.cost(P), [(F * D[np.ix_(p, p)]).sum() for p in P])
