"""GPU: the calls that can be recorded into a CUDA graph.  A replay repeats the recorded step (the random key is a launch
parameter) on whatever the buffers hold by then, so two replays equal two direct calls."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan

pytestmark = pytest.mark.gpu

HP = (0.1, 0.9, 5e-4, 0.0, 10.0)


@pytest.mark.parametrize("what", ["step_passes", "separate"])
@pytest.mark.parametrize("sizes,M", [([1, 33, 5000, 4096, 20001], 3), ([9, 600 * 4096 - 3, 4095], 2)])
def test_captured_calls_equal_direct_ones(what, sizes, M):
    from paper_2206_06257_b200 import api
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d = int(offs[-1])
    g = torch.Generator(device="cuda").manual_seed(M)
    rnd = lambda s: torch.randn(d, generator=g, device="cuda") * s  # noqa: E731
    theta, mom, grads = rnd(0.05), rnd(1e-3), [rnd(1e-2) for _ in range(M)]
    with GpuPlan(api, offs, M, 8) as P:
        lv, sg, sc = P.alloc_message()
        lv1, sg1, sc1 = lv[:P.level_bytes].clone(), sg[:P.sign_bytes].clone(), torch.zeros(P.h, device="cuda")
        gh = torch.zeros(d, device="cuda")

        def step(th, mo, stream=None):
            if what == "step_passes":
                api.dat_step_passes(P.plan, th, mo, grads, 7, 3, HP, stream=stream)
            else:
                api.dat_quantize(P.plan, grads, 7, 3, lv, sg, sc, stream=stream)
                api.dat_aggregate(P.plan, lv, sg, sc, None, gh, stream=stream)
                api.dat_requantize(P.plan, gh, 7, 3, lv1, sg1, sc1, stream=stream)
                api.dat_lalr_step(P.plan, th, mo, gh, HP, stream=stream)
        th1, mo1 = theta.clone(), mom.clone()
        step(th1, mo1)
        th2, mo2 = theta.clone(), mom.clone()
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            graph.capture_begin()
            try:
                step(th2, mo2, stream=s)
            finally:
                graph.capture_end()
        torch.cuda.synchronize()
        assert torch.equal(th2, theta) and torch.equal(mo2, mom)          # recorded, not run
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(th1, th2) and torch.equal(mo1, mo2)
        step(th1, mo1)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(th1, th2) and torch.equal(mo1, mo2)
        assert P.status() == 0
        del graph
