"""One batch searched with the form of phase X changing from call to call: each
call plans and reports its own form, captured calls keep the tables there are,
and the walks are the same."""
import numpy as np
import pytest

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu

FIELDS = ["best_cost", "final_cost", "best_iter", "iters_done", "status", "descent_moves",
          "hash", "descent_hash"]
AUTO, DOTS = 0, 1


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    q.lib()
    return torch


def _batch(ns):
    pairs = [instances.uniform_instance(n, 4100 + n, symmetric=False) for n in ns]
    return q.Batch([F for F, _ in pairs], [D for _, D in pairs])


def _params(form, iters=60):
    return q.make_params(3, seed=8, iters=iters, tenure=(4, 12, 0), phase_x=form)


def test_each_call_has_its_own_form():
    with _batch([20, 50, 145, 200]) as b:
        ref = None
        for form in (AUTO, DOTS, AUTO, DOTS):
            classes, _ = b.classes(_params(form))
            products = [c["products"] for c in classes if c["nmax"] < 150]
            assert all((x > 0) == (form == AUTO) for x in products), (form, classes)
            assert b.plan(_params(form))["threads_per_walk"] == (512 if form == AUTO else 1024)
            g = b.search(_params(form))
            ref = ref or g
            for k in FIELDS:
                assert np.array_equal(g[k], ref[k]), (form, k)


def test_dots_on_tuned_plans():
    """Plans without transposed copies are kept by the autotuner where they win;
    dot products, which need the copies, still run after it."""
    with _batch([145, 146]) as b:
        before = b.search(_params(DOTS))
        b.autotune(_params(AUTO), trial_iters=40)
        tuned = b.search(_params(AUTO))
        assert b.plan(_params(DOTS))["products"] == 0
        after = b.search(_params(DOTS))
        for k in FIELDS:
            assert np.array_equal(before[k], after[k]) and np.array_equal(before[k], tuned[k]), k


@pytest.mark.parametrize("first,captured", [(AUTO, DOTS), (DOTS, AUTO)])
def test_a_captured_call_may_ask_for_the_other_form(gpu, first, captured):
    with _batch([20, 50, 145]) as b:
        outs = b.device_outputs(3)
        stream = gpu.cuda.Stream()
        with gpu.cuda.stream(stream):
            b.search_async(_params(first), outs, stream=stream)
        stream.synchronize()
        ref = {k: outs[k].clone() for k in FIELDS}
        for k in FIELDS:
            outs[k].zero_()
        gpu.cuda.synchronize()
        g = gpu.cuda.CUDAGraph()
        with gpu.cuda.graph(g, stream=stream):
            b.search_async(_params(captured), outs, stream=stream)
        g.replay()
        gpu.cuda.synchronize()
        for k in FIELDS:
            assert gpu.equal(outs[k], ref[k]), k


@pytest.mark.parametrize("captured", [AUTO, DOTS])
def test_a_graph_outlives_searches_of_the_other_form(gpu, captured):
    """A captured search's tables and workspace stay while searches of the other
    form run (n = 160 needs a workspace in one form only)."""
    with _batch([20, 50, 145, 160, 200]) as b:
        outs = b.device_outputs(3)
        stream = gpu.cuda.Stream()
        with gpu.cuda.stream(stream):
            b.search_async(_params(captured), outs, stream=stream)
        stream.synchronize()
        ref = {k: outs[k].clone() for k in FIELDS}
        g = gpu.cuda.CUDAGraph()
        with gpu.cuda.graph(g, stream=stream):
            b.search_async(_params(captured), outs, stream=stream)
        other = b.search(_params(1 - captured))  # its own tables
        fill = gpu.full((1 << 20,), 7, dtype=gpu.int32, device="cuda")  # memory freed would be in use
        for form in (captured, 1 - captured):
            b.search(_params(form))
        for k in FIELDS:
            outs[k].zero_()
        gpu.cuda.synchronize()
        g.replay()
        gpu.cuda.synchronize()
        for k in FIELDS:
            assert gpu.equal(outs[k], ref[k]), k
            assert np.array_equal(other[k].astype(np.int64), ref[k].cpu().numpy().astype(np.int64)), k
        assert int(fill.sum()) == 7 << 20
