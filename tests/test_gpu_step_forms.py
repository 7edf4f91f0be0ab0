"""GPU: the three forms of a step -- one launch, one launch per phase, and one whose CTAs keep their pieces -- as the rule
chooses them by size, workers and the largest layer, against the separate calls (dat_quantize, dat_aggregate / dat_average, dat_requantize, dat_lalr_step,
dat_lamb_step) on the same inputs.  The quantizer norms and the layers' norms are sums of the same numbers in other orders
(at most one unit in the last place apart); where the bits of the quantizer norms agree, codes and moments have to be the
same, and theta within 1e-5 relative of rounding through the layers' norms.
"""
import numpy as np
import pytest
import torch

from helpers import assert_close_per_layer, np_of, ulp_diff

pytestmark = pytest.mark.gpu

HP = (0.1, 0.9, 5e-4, 0.0, 10.0)
LAMB_HP = (0.1, 0.9, 0.999, 1e-6, 1e-4, 0.0, 10.0)
TILE = 4096
# tiles on a 148-SM GPU: a few pieces (kept by their CTAs; many workers and b = 32 by phases); above one wave (phases, M >= 8 by
# half tiles; b = 32 in one launch); above nine tiles per SM in one layer (phases; b = 32 in one launch), and in eight equal ones
# (one launch; one worker by phases)
SIZES = {"small": [1, 7, 2047, 2049, 4097], "below": [9, 600 * TILE - 3, 4095], "above": [9, 1340 * TILE + 5, 33],
         "spread": [9, 33] + [170 * TILE + k for k in (-3, 0, 5, 1, 8, -7, 2, 11)]}


@pytest.mark.parametrize("kind", ["step", "lamb", "two_sided"])
@pytest.mark.parametrize("where,M,bits,rng_bits,per_worker", [("small", 5, 8, 16, False), ("below", 3, 4, 23, False), ("below", 9, 8, 16, False), ("below", 2, 32, 16, False), ("above", 3, 8, 16, False),
                                                              ("above", 2, 4, 16, True), ("below", 2, 2, 23, True), ("above", 1, 8, 16, False),
                                                              ("spread", 3, 8, 16, False), ("spread", 2, 4, 16, True), ("spread", 9, 1, 23, False),
                                                              ("spread", 2, 16, 23, True), ("spread", 1, 8, 16, False), ("spread", 2, 32, 16, False),
                                                              ("small", 64, 1, 16, True), ("above", 2, 32, 16, False), ("small", 3, 32, 16, False)])
def test_step_forms_equal_separate_calls(kind, where, M, bits, rng_bits, per_worker):
    from paper_2206_06257_b200 import api
    if kind == "two_sided" and bits == 32:
        pytest.skip("nothing to quantize with")
    offs = np.concatenate([[0], np.cumsum(SIZES[where])]).astype(np.int64)
    d, h = int(offs[-1]), len(offs) - 1
    g = torch.Generator(device="cuda").manual_seed(M)
    rnd = lambda s: torch.randn(d, generator=g, device="cuda") * s  # noqa: E731
    theta, mom, var, grads = rnd(0.05), rnd(1e-3), rnd(1e-3).square(), [rnd(1e-2) for _ in range(M)]
    plan = api.dat_plan_create(offs, M, bits, rng_bits=rng_bits, scale_mode=api.DAT_SCALE_PER_WORKER if per_worker else api.DAT_SCALE_SHARED_MAX)
    try:
        th, mo, va, gh = theta.clone(), mom.clone(), var.clone(), torch.empty(d, device="cuda")
        sc = torch.zeros(M * h, device="cuda")
        if kind == "step":
            api.dat_step(plan, th, mo, grads, 7, 3, HP, None, None, sc)
        elif kind == "lamb":
            api.dat_step_lamb(plan, th, mo, va, grads, 7, 3, LAMB_HP, 4, None, None, sc)
        else:
            api.dat_step_two_sided(plan, th, mo, grads, 7, 3, HP, gh, None, None, sc)
        th2, mo2, va2, gh2 = theta.clone(), mom.clone(), var.clone(), torch.empty(d, device="cuda")
        if bits == 32:
            api.dat_average(plan, grads, gh2)
        else:
            lb, sb, ns, _ = api.dat_plan_sizes(plan)
            lv, sg, sc2 = [torch.empty(M * n, dtype=torch.uint8, device="cuda") for n in (lb, sb)] + [torch.empty(ns, device="cuda")]
            api.dat_quantize(plan, grads, 7, 3, lv, sg, sc2)
            assert ulp_diff(np_of(sc)[:ns], np_of(sc2)).max() <= 1
            api.dat_quantize(plan, grads, 7, 3, lv, sg, sc2, scales_in=sc[:ns].clone())      # the step's own bits
            api.dat_aggregate(plan, lv, sg, sc2, None, gh2)
            if kind == "two_sided":
                s_sc = torch.empty(h, device="cuda")
                api.dat_requantize(plan, gh2, 7, 3, lv[:lb].clone(), sg[:sb].clone(), s_sc)
        if kind == "lamb":
            api.dat_lamb_step(plan, th2, mo2, va2, gh2, LAMB_HP, 4)
            assert torch.equal(va, va2)
        else:
            api.dat_lalr_step(plan, th2, mo2, gh2, HP)
        torch.cuda.synchronize()
        assert api.dat_get_status(plan) == 0
        if kind == "two_sided":          # the server's norm is a sum in another order too: at most a last place of every value
            assert_close_per_layer(np_of(gh), np_of(gh2), offs, "receiver's value")
            assert_close_per_layer(np_of(mo), np_of(mo2), offs, "momentum")
        else:
            assert torch.equal(mo, mo2)
        assert_close_per_layer(np_of(th), np_of(th2), offs, "theta")
    finally:
        api.dat_plan_destroy(plan)
