"""Large n: once a search has run, one of its size can be captured whatever
layout its tenures or its form of phase X take (the workspace holds either)."""
import numpy as np
import pytest

import paper_2307_11248_gb300 as q
from paper_2307_11248_gb300 import instances

pytestmark = pytest.mark.gpu

FIELDS = ["best_cost", "final_cost", "best_iter", "iters_done", "status", "hash"]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU test selected but no CUDA device is available")
    q.lib()
    return torch


# the second search before the capture has its size, but fits the workspace that
# the first one took for its rows
@pytest.mark.parametrize("walks", [(3,), (50, 60)])
@pytest.mark.parametrize("captured", [dict(tenure=(600, 700, 0)), dict(tenure=(5, 20, 0), phase_x=1)])
def test_capture_after_a_search_of_the_other_layout(gpu, captured, walks):
    F, D = instances.grid_instance(190, 4600)
    kw = dict(seed=3, iters=25)
    with q.Instance(F, D) as inst:
        stream = gpu.cuda.Stream()
        for W in walks:
            outs = inst.device_outputs(W)
            with gpu.cuda.stream(stream):
                inst.search_async(q.make_params(W, tenure=(5, 20, 0), **kw), outs, stream=stream)
            stream.synchronize()
        prm = q.make_params(walks[-1], **captured, **kw)
        g = gpu.cuda.CUDAGraph()
        with gpu.cuda.graph(g, stream=stream):
            inst.search_async(prm, outs, stream=stream)
        for v in outs.values():
            v.zero_()
        gpu.cuda.synchronize()
        g.replay()
        gpu.cuda.synchronize()
        with q.Instance(F, D) as other:
            want = other.search(prm)
        for k in FIELDS:
            got = outs[k].cpu().numpy().astype(np.int64)
            assert np.array_equal(got, want[k].astype(np.int64)), k
