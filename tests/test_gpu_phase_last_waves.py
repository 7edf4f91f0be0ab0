"""GPU: the phases of a step whose last wave goes by half tiles, at exact numbers of tiles around one wave, a half and two, against
the one launch."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, assert_close_per_layer, np_of, ulp_diff
from test_gpu_parity import HP, LAMB_HP, api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
ONE_LAUNCH, PHASES = 1, 2
TILE = 4096


def _wave():
    return 4 * torch.cuda.get_device_properties(0).multi_processor_count


def _tiles(offs):
    """Tiles of a layer start at multiples of 8."""
    return sum(-(-(int(hi) - (int(lo) & ~7)) // TILE) for lo, hi in zip(offs[:-1], offs[1:]))


def _offs(tiles):
    """Layers of `tiles` tiles in all: many in one tile, odd ones, one of most of the elements."""
    offs = np.concatenate([[0], np.cumsum([1, 7, 33, 4095, 4097, 9001, 2, 8, 64])]).astype(np.int64)
    lo = int(offs[-1])
    offs = np.append(offs, (lo & ~7) + TILE * (tiles - _tiles(offs)) - 5)
    assert _tiles(offs) == tiles
    return offs


# tiles beyond one wave of CTAs (at one wave all go by halves)
@pytest.mark.parametrize("rest", ["1", "0.4", "0.4 + 1", "half", "half + 1", "wave - 1", "wave", "wave + 1"])
@pytest.mark.parametrize("kind", ["step", "lamb", "two_sided"])
@pytest.mark.parametrize("M,rng_bits,per_worker", [(2, 16, False), (3, 23, True)])
def test_last_wave_by_half_tiles(api, kind, rest, M, rng_bits, per_worker):  # noqa: F811
    wave = _wave()
    offs = _offs(wave + {"1": 1, "0.4": 2 * wave // 5, "0.4 + 1": 2 * wave // 5 + 1, "half": wave // 2, "half + 1": wave // 2 + 1, "wave - 1": wave - 1, "wave": wave, "wave + 1": wave + 1}[rest])
    d = int(offs[-1])
    gen = torch.Generator(device="cuda").manual_seed(d)
    rnd = lambda s: torch.randn(d, generator=gen, device="cuda") * s  # noqa: E731
    theta, mom, var, grads = rnd(0.05), rnd(1e-3), rnd(1e-3).square(), [rnd(1e-2) for _ in range(M)]
    out = {}
    for form in (ONE_LAUNCH, PHASES):
        with GpuPlan(api, offs, M, 8, rng_bits, scale_mode=api.DAT_SCALE_PER_WORKER if per_worker else 0) as P:
            api.dat_plan_test_form(P.plan, form)
            th, mo, va, gh, sc = theta.clone(), mom.clone(), var.clone(), torch.zeros_like(theta), torch.zeros(P.num_scales, device="cuda")
            if kind == "step":
                api.dat_step(P.plan, th, mo, grads, 7, 3, HP, None, None, sc)
            elif kind == "lamb":
                api.dat_step_lamb(P.plan, th, mo, va, grads, 7, 3, LAMB_HP, 4, None, None, sc)
            else:
                api.dat_step_two_sided(P.plan, th, mo, grads, 7, 3, HP, gh, None, None, sc)
            assert P.status() == 0
            out[form] = [np_of(x) for x in (th, mo, va, gh, sc)]
    a, b = out[ONE_LAUNCH], out[PHASES]
    assert ulp_diff(a[4], b[4]).max() <= 1           # codes depend on the norms' bits
    for l in range(len(offs) - 1):
        s = slice(int(offs[l]), int(offs[l + 1]))
        if np.array_equal(a[4].reshape(-1, len(offs) - 1)[:, l], b[4].reshape(-1, len(offs) - 1)[:, l]):
            if kind != "two_sided":                  # (the server's norm is a sum in another order too)
                assert np.array_equal(a[1][s], b[1][s]) and np.array_equal(a[2][s], b[2][s])
            for k, name in enumerate(("theta", "momentum", "var", "g_hat")):
                assert_close_per_layer(b[k][s], a[k][s], [0, s.stop - s.start], name)
