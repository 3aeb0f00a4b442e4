"""The autotuner times the rule's own plan of every class, so that it never keeps
a plan that its trial found slower than the rule's."""
import pytest

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("force_int64", [False, True])
@pytest.mark.parametrize("kind", ["asym", "sym", "lognormal"])
def test_the_rules_plan_is_timed(kind, force_int64):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    ns = [30, 66, 96, 100, 145, 160, 190]
    if kind == "lognormal":
        pairs = [instances.lognormal_instance(n, 4500 + n, False) for n in ns]
    else:
        pairs = [instances.uniform_instance(n, 4500 + n, symmetric=kind == "sym") for n in ns]
    with q.Batch([F for F, _ in pairs], [D for _, D in pairs], force_int64=force_int64) as b:
        # walks enough for two CTAs on every SM: the rule's own preference there
        report = b.autotune(q.make_params(60, seed=2, iters=30, tenure=(5, 20, 0)), trial_iters=10)
    assert sum(r["instances"] for r in report) == len(ns)
    for r in report:
        assert 0 < r["trial_ms"] <= r["rule_ms"], r
