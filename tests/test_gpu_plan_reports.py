"""What a batch reports of a search is what it launches: where the tenures send
a class to the row layout, the row layout's threads, phase X and workspace."""
import pytest

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu

KEYS = ["threads_per_walk", "pairs_per_thread", "products", "workspace"]


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    q.lib()
    return torch


# n = 100 with two walks per SM: no room for the copies beside the rotation
# layout's arrays, room for them in the rows; n = 160: M in the workspace, in
# batches, and rows without one
@pytest.mark.parametrize("n,walks,short", [(50, 4, dict(products=1, workspace=0)),
                                           (100, 400, dict(products=2, workspace=0)),
                                           (160, 4, dict(products=0, workspace=1)),
                                           (200, 4, dict(products=0, workspace=1))])
def test_reports_follow_the_layout(n, walks, short):
    F, D = instances.uniform_instance(n, 4300 + n, symmetric=False)
    with q.Batch([F], [D]) as b, q.Instance(F, D) as one:
        for tenure in ((5, 30, 0), (600, 700, 0), (5, 30, 0)):
            prm = q.make_params(walks, seed=1, iters=20, tenure=tenure)
            plan = b.plan(prm)
            cls, _ = b.classes(prm)
            for k in KEYS:
                assert cls[0][k] == plan[k], k
            if tenure[0] == 600:  # the rows, as a search of the instance alone reports
                alone = one.plan(prm)
                for k in KEYS + ["smem_bytes"]:
                    assert plan[k] == alone[k], k
            else:
                for k, v in short.items():
                    assert plan[k] == v, (k, plan)


@pytest.mark.parametrize("n", [50, 160, 200])
@pytest.mark.parametrize("tenure", [(5, 30, 0), (600, 700, 0)])
def test_the_autotuner_reports_what_a_search_like_its_trial_runs(n, tenure):
    F, D = instances.uniform_instance(n, 4400 + n, symmetric=False)
    prm = q.make_params(4, seed=1, iters=20, tenure=tenure)
    with q.Batch([F], [D]) as b:
        r = b.autotune(prm, trial_iters=20)[0]
        plan = b.plan(prm)
        for k in KEYS:
            assert r[k] == plan[k], k
