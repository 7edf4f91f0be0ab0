"""GPU: groups of eight at a layer's ends, which a warp draws together with a worker per lane, at the worker counts around one
and two rounds of lanes (with one and two workers by the group's own lane), against the oracle's integers (given the GPU's norm bits: code sums and m' bit for bit)."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, np_of
from test_gpu_parity import HP, _random_problem, api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SIZES = [3, 8, 13, 2049, 5, 4095, 1, 8191]       # ends in one group, in two, on piece and tile boundaries


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("mode", ["shared", "per_worker"])
@pytest.mark.parametrize("M", [1, 2, 3, 31, 32, 33, 64])
def test_ragged_groups(api, oracle, M, mode, form, rng_bits):  # noqa: F811
    sm = oracle.SCALE_PER_WORKER if mode == "per_worker" else oracle.SCALE_SHARED_MAX
    offs, grads, theta, mom = _random_problem(300 + M, SIZES, M)
    d = int(offs[-1])
    with GpuPlan(api, offs, M, 8, rng_bits, scale_mode=api.DAT_SCALE_PER_WORKER if mode == "per_worker" else 0) as P:
        api.dat_plan_test_form(P.plan, form)
        th, mo = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda()
        cs = None if mode == "per_worker" else torch.full((d,), -7, dtype=torch.int32, device="cuda")
        sc = torch.zeros(P.num_scales, device="cuda")
        api.dat_step(P.plan, th, mo, [torch.from_numpy(g).cuda() for g in grads], 3, 5, HP, cs, None, sc)
        torch.cuda.synchronize()
        assert P.status() == 0
        level, neg = oracle.quantize(offs, grads, 8, 3, 5, np_of(sc), sm, rng_bits=rng_bits)
        code_sum, gh = oracle.aggregate(offs, level, neg, np_of(sc), 8, sm)
        if cs is not None:
            assert np.array_equal(np_of(cs), code_sum)
        _, mo_ref, _ = oracle.lalr(offs, theta, mom, gh, *HP)
        assert np.array_equal(np_of(mo).view(np.uint32), mo_ref.view(np.uint32))
