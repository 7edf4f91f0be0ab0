"""GPU: the separate calls one after the other on a stream, whose kernels are set up under the ends of those before: the same
bits as with a wait for the GPU between any two calls, at one tile, a ragged few, and several waves of CTAs; and the same with
copies, memsets and waits for another stream's events between the calls."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, np_of
from test_gpu_parity import HP, LAMB_HP, api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[31], [5, 4096, 33, 9001], [3_000_001, 7, 500_000]])
@pytest.mark.parametrize("per_worker", [False, True])
def test_back_to_back_calls(api, sizes, per_worker):  # noqa: F811
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, M = int(offs[-1]), 3
    out = []
    for wait in (torch.cuda.synchronize, lambda: None):
        gen = torch.Generator(device="cuda").manual_seed(d)
        rnd = lambda s: torch.randn(d, generator=gen, device="cuda") * s  # noqa: E731
        th, mo, va, grads = rnd(0.05), rnd(1e-3), rnd(1e-3).square(), [rnd(1e-2) for _ in range(M)]
        with GpuPlan(api, offs, M, 8, scale_mode=api.DAT_SCALE_PER_WORKER if per_worker else 0) as P:
            lv, sg, sc = P.alloc_message()
            lv2, sg2, sc2 = torch.empty_like(lv[:P.level_bytes]), torch.empty_like(sg[:P.sign_bytes]), torch.empty(P.h, device="cuda")
            gh = torch.zeros(d, device="cuda")
            for step in range(6):                            # every call's inputs are the outputs of the call before
                api.dat_quantize(P.plan, grads, 7, step, lv, sg, sc)
                wait()
                api.dat_aggregate(P.plan, lv, sg, sc, None, gh)
                wait()
                if step & 1:
                    api.dat_requantize(P.plan, gh, 7, step, lv2, sg2, sc2)
                    wait()
                    api.dat_lamb_step(P.plan, th, mo, va, gh, LAMB_HP, step + 1)
                else:
                    api.dat_lalr_step(P.plan, th, mo, gh, HP)
                wait()
                grads[step % M].add_(gh)                     # (a kernel of another library in between)
                wait()
            assert P.status() == 0
            out.append([np_of(x) for x in (lv, sg, sc, lv2, sg2, sc2, gh, th, mo, va)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("sizes", [[31], [5, 4096, 33, 9001], [3_000_001, 7, 500_000]])
@pytest.mark.parametrize("per_worker", [False, True])
def test_copies_memsets_and_events_between_calls(api, sizes, per_worker):  # noqa: F811
    """A message that another stream copies before it is decoded, buffers that are cleared and copied right before and after the
    calls that read and write them."""
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, M, side = int(offs[-1]), 3, torch.cuda.Stream()
    out = []
    for wait in (torch.cuda.synchronize, lambda: None):
        gen = torch.Generator(device="cuda").manual_seed(d)
        rnd = lambda s: torch.randn(d, generator=gen, device="cuda") * s  # noqa: E731
        th, mo, grads = rnd(0.05), rnd(1e-3), [rnd(1e-2) for _ in range(M)]
        with GpuPlan(api, offs, M, 4, scale_mode=api.DAT_SCALE_PER_WORKER if per_worker else 0) as P:
            msg = P.alloc_message()
            arrived = [torch.zeros_like(x) for x in msg]
            gh, gh2, kept = (torch.empty(d, device="cuda") for _ in range(3))
            main = torch.cuda.current_stream()
            torch.cuda.synchronize()
            for step in range(6):
                grads[step % M].copy_(kept) if step else None              # a copy, then the call that reads it
                api.dat_quantize(P.plan, grads, 7, step, *msg)
                wait()
                side.wait_stream(main)
                with torch.cuda.stream(side):
                    for x, y in zip(arrived, msg):
                        x.copy_(y)
                main.wait_stream(side)                                     # an event, then the call behind it
                wait()
                api.dat_aggregate(P.plan, *arrived, None, gh)
                wait()
                for x in arrived + list(msg):
                    x.zero_()                                              # memsets behind the call that reads
                gh2.copy_(gh)
                gh.zero_()
                wait()
                api.dat_lalr_step(P.plan, th, mo, gh2, HP)
                wait()
                kept.copy_(mo)
                gh2.zero_()
                wait()
            assert P.status() == 0
            out.append([np_of(x) for x in (th, mo, kept, gh, gh2)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
