"""GPU: gradients with a NaN or an infinity against the oracle.  The levels are those of the plain form of Eq. xi,
min(floor(fma(|g|, S/nu, u1)) - 1, S) with the minimum of IEEE 754 (a NaN has level S, no sign), and no element changes
another one's code.
"""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, np_of, oracle_planes

pytestmark = pytest.mark.gpu

HP = (0.1, 0.9, 5e-4, 0.0, 10.0)
SIZES = [4700, 5001, 8200, 37, 9003]
OFFS = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
M = 3


def _grads():
    rng = np.random.RandomState(11)
    g = [(rng.randn(int(OFFS[-1])) * 1e-2).astype(np.float32) for _ in range(M)]
    nan, inf = np.float32("nan"), np.float32("inf")
    for e in (0, 1, 9, 2051, 4699):             # layer 0: NaN in worker 1 alone, the shared norm stays finite
        g[1][e] = nan if e % 2 else -nan
    for k, e in enumerate((0, 13, 4097, 5000)):  # layer 1: infinities, the norm is infinite
        g[2][OFFS[1] + e] = inf if k % 2 else -inf
    g[0][OFFS[2] + 77] = nan                    # layer 2: NaN in the first worker, the norm is NaN
    g[1][OFFS[3] + 36] = nan                    # layer 3: small, ragged
    return g                                    # layer 4: finite


@pytest.mark.parametrize("bits", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("per_worker", [False, True])
def test_codes_and_sums(oracle, bits, per_worker, rng_bits):
    from paper_2206_06257_b200 import api
    sm = oracle.SCALE_PER_WORKER if per_worker else oracle.SCALE_SHARED_MAX
    g, d, h = _grads(), int(OFFS[-1]), len(SIZES)
    gd = [torch.from_numpy(x).cuda() for x in g]
    rng = np.random.RandomState(bits)
    theta, mom = (rng.randn(d) * 0.05).astype(np.float32), (rng.randn(d) * 1e-3).astype(np.float32)
    with GpuPlan(api, OFFS, M, bits, rng_bits, scale_mode=api.DAT_SCALE_PER_WORKER if per_worker else 0) as P:
        lv, sg, sc = P.alloc_message()
        own = None
        finite = torch.from_numpy(rng.uniform(0.5, 2.0, P.num_scales).astype(np.float32)).cuda()
        for scales_in in (None, finite):
            api.dat_quantize(P.plan, gd, 3, 5, lv, sg, sc, scales_in)
            level, neg = oracle.quantize(OFFS, g, bits, 3, 5, np_of(sc).reshape((M, h) if per_worker else (h,)), sm, rng_bits=rng_bits)
            lp, sp = oracle_planes(oracle, level, neg, bits)
            assert np.array_equal(np_of(lv).reshape(M, -1), lp) and np.array_equal(np_of(sg).reshape(M, -1), sp)
            if scales_in is None:
                own = np_of(sc).copy()
                assert P.status() & api.DAT_STATUS_NONFINITE
        # the steps: integer sums, or m' where each worker has its own grid
        for entry in [api.dat_step, api.dat_step_pipelined] + ([] if per_worker else [api.dat_step_passes]):
            th, mo, sc2 = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda(), torch.zeros(P.num_scales, device="cuda")
            cs = None if per_worker else torch.zeros(d, dtype=torch.int32, device="cuda")
            entry(P.plan, th, mo, gd, 3, 5, HP, cs, None, sc2)
            assert P.status() & api.DAT_STATUS_NONFINITE
            assert np.array_equal(np_of(sc2), own, equal_nan=True)
            scales = own.reshape((M, h) if per_worker else (h,))
            level, neg = oracle.quantize(OFFS, g, bits, 3, 5, scales, sm, rng_bits=rng_bits)
            with np.errstate(invalid="ignore", over="ignore"):
                cs_ref, gh = oracle.aggregate(OFFS, level, neg, scales, bits, sm)
                _, mo_ref, _ = oracle.lalr(OFFS, theta, mom, gh, *HP)
            if not per_worker:
                assert np.array_equal(np_of(cs), cs_ref)
            assert np.array_equal(np_of(mo), mo_ref, equal_nan=True)


@pytest.mark.parametrize("bits", [1, 2, 4, 8, 16])
def test_requantize_and_ranges(oracle, bits, rng_bits):
    from paper_2206_06257_b200 import api
    from paper_2206_06257_b200.sharded import CudaOps, RangeLayout, partition_layers
    g, h = _grads(), len(SIZES)
    nu = torch.from_numpy(np.random.RandomState(bits).uniform(0.5, 2.0, h).astype(np.float32)).cuda()
    with GpuPlan(api, OFFS, M, bits, rng_bits) as P:
        for k in range(M):
            gh = torch.from_numpy(g[k].copy()).cuda()
            lv, sg, sc = (torch.zeros(P.level_bytes, dtype=torch.uint8, device="cuda"), torch.zeros(P.sign_bytes, dtype=torch.uint8, device="cuda"),
                          torch.zeros(h, device="cuda"))
            api.dat_requantize(P.plan, gh, 5, 2, lv, sg, sc, scales_in=nu)
            out, _, level, neg = oracle.requantize(OFFS, g[k], bits, 5, 2, stream=M, rng_bits=rng_bits, scales_in=np_of(nu))
            lp, sp = oracle.pack(level, neg, bits)
            assert np.array_equal(np_of(lv), lp) and np.array_equal(np_of(sg), sp)
            assert np.array_equal(np_of(gh).view(np.uint32), out.view(np.uint32))
        # a rank's messages to several owners: the codes of the whole vectors, range by range
        level, neg = oracle.quantize(OFFS, g, bits, 7, 1, np_of(nu), rng_bits=rng_bits)
        ops = CudaOps(api, OFFS, M, M, 0, 1, bits, rng_bits)
        try:
            ranges = [RangeLayout(OFFS, a, b) for a, b in partition_layers(OFFS, 3)]
            got = ops.quantize_ranges(ranges, [torch.from_numpy(x).cuda() for x in g], nu, 7, 1)
            for rg, (lv, sg) in zip(ranges, got):
                for i in range(M):
                    lb, sb = lv.numel() // M, sg.numel() // M
                    lev, ng = oracle.unpack(np_of(lv)[i * lb:(i + 1) * lb], np_of(sg)[i * sb:(i + 1) * sb], rg.n, bits)
                    assert np.array_equal(lev[rg.pad:], level[i, rg.a:rg.b]) and np.array_equal(ng[rg.pad:] != 0, neg[i, rg.a:rg.b] != 0)
        finally:
            ops.close()
