"""GPU: the phases of a step whose last wave goes by half tiles, on both sides of that line, against the one launch."""
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


def _sizes(tiles):
    """Layers of `tiles` tiles in all (or a few more): many in one tile, odd ones, one of most of the elements."""
    small = [1, 7, 33, 4095, 4097, 9001, 2, 8, 64]
    return small + [TILE * (tiles - sum(-(-(s + 7) // TILE) for s in small)) - 5]


@pytest.mark.parametrize("rest", [0, 1, 0.5, 0.51])
@pytest.mark.parametrize("kind", ["step", "lamb", "two_sided"])
def test_last_wave_by_half_tiles(api, kind, rest):  # noqa: F811
    tiles = _wave() + (rest if rest in (0, 1) else int(rest * _wave()))
    offs = np.concatenate([[0], np.cumsum(_sizes(tiles))]).astype(np.int64)
    d, M = int(offs[-1]), 2
    gen = torch.Generator(device="cuda").manual_seed(tiles)
    rnd = lambda s: torch.randn(d, generator=gen, device="cuda") * s  # noqa: E731
    theta, mom, var, grads = rnd(0.05), rnd(1e-3), rnd(1e-3).square(), [rnd(1e-2) for _ in range(M)]
    out = {}
    for form in (ONE_LAUNCH, PHASES):
        with GpuPlan(api, offs, M, 8) as P:
            api.dat_plan_test_form(P.plan, form)
            th, mo, va, gh, sc = theta.clone(), mom.clone(), var.clone(), torch.zeros_like(theta), torch.zeros(P.h, device="cuda")
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
        if a[4][l] == b[4][l]:
            if kind != "two_sided":                  # (the server's norm is a sum in another order too)
                assert np.array_equal(a[1][s], b[1][s]) and np.array_equal(a[2][s], b[2][s])
            for k, name in enumerate(("theta", "momentum", "var", "g_hat")):
                assert_close_per_layer(b[k][s], a[k][s], [0, s.stop - s.start], name)
