"""GPU: the LAMB direction (Algorithm A2) where the bias corrections leave the ordinary range -- second moments that
overflow to infinity for a finite gradient, and moments that have decayed towards the denormal numbers -- against the
oracle.  Layers of one element make the direction itself visible: ||u_l|| = |u_l| without rounding.
"""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, assert_close_per_layer, np_of

pytestmark = pytest.mark.gpu

T = [1, 2, 10, 1000, 20000]                # 1 - beta2^t: below, above and equal to a power of two's quotient (lo < 0, > 0, = 0)


def _bits(x):
    return np.asarray(x, dtype=np.float32).view(np.uint32)


@pytest.mark.parametrize("t", T)
def test_directions_of_small_moments_are_correctly_rounded(oracle, t):
    """m and v over every binade from the smallest denormal number to 2^-90 (and zeros): |u_l| bit for bit."""
    from paper_2206_06257_b200 import api
    rng = np.random.RandomState(t)
    n = 30000
    mag = lambda: np.ldexp(rng.uniform(1.0, 2.0, n), rng.randint(-149, -89, n)).astype(np.float32)  # noqa: E731
    mom, var = mag() * np.where(rng.rand(n) < 0.5, -1, 1).astype(np.float32), mag()
    mom[:n // 2] = np.abs(mom[:n // 2])
    var[:n // 2] = 0.0                      # u = m^ (zeta = 1): the first quotient by itself
    mom[n // 2:n // 2 + 50] = 0.0
    theta, g_hat = np.zeros(n, dtype=np.float32), np.zeros(n, dtype=np.float32)
    for zeta in (1.0, 1e-20):
        hp = (0.1, 0.9, 0.999, zeta, 0.0, 1.0, 10.0)
        with GpuPlan(api, np.arange(n + 1), 1, 8) as P:
            th, mo, va = (torch.from_numpy(x.copy()).cuda() for x in (theta, mom, var))
            norms = torch.zeros(2 * n, device="cuda")
            api.dat_lamb_step(P.plan, th, mo, va, torch.from_numpy(g_hat).cuda(), hp, t, norms)
            torch.cuda.synchronize()
        th_ref, mo_ref, va_ref, n_ref = oracle.lamb(np.arange(n + 1), theta, mom, var, g_hat, t, *hp)
        assert np.array_equal(_bits(np_of(mo)), _bits(mo_ref)) and np.array_equal(_bits(np_of(va)), _bits(va_ref))
        assert np.array_equal(_bits(np_of(norms).reshape(-1, 2)), _bits(n_ref))
        assert np.array_equal(_bits(np_of(th)), _bits(th_ref))       # (the step length is formed from the same bits)


@pytest.mark.parametrize("call", ["lamb_step", "step_lamb", "step_lamb_two_sided"])
@pytest.mark.parametrize("t", T)
def test_second_moment_that_overflows(oracle, call, t):
    """|g_hat| = 1e20 is finite, its square is not: v^ is infinite, u = wd * theta, and nothing else of the layer moves."""
    from paper_2206_06257_b200 import api
    hp = (0.1, 0.9, 0.999, 1e-6, 1e-2, 0.0, 10.0)
    rng = np.random.RandomState(3)
    offs = np.concatenate([[0], np.cumsum([5000, 33, 9001])]).astype(np.int64)
    d = int(offs[-1])
    theta, mom, var = (rng.randn(d) * 0.05).astype(np.float32), np.zeros(d, dtype=np.float32), np.zeros(d, dtype=np.float32)
    g = (rng.randn(d) * 1e-2).astype(np.float32)
    at = [0, 17, 4097, 5005, 5033 + 8999]
    g[at] = np.float32(1e20) * np.array([1, -1, 1, 1, -1], dtype=np.float32)
    with GpuPlan(api, offs, 1, 32 if call == "step_lamb" else 8) as P:
        th, mo, va, gd = (torch.from_numpy(x.copy()).cuda() for x in (theta, mom, var, g))
        if call == "lamb_step":
            api.dat_lamb_step(P.plan, th, mo, va, gd, hp, t)
            gh = g
        elif call == "step_lamb":           # b = 32, one worker: g_hat is the gradient
            api.dat_step_lamb(P.plan, th, mo, va, [gd], 0, 0, hp, t)
            gh = g
        else:                               # the receiver's value is an output
            gh_d = torch.zeros(d, device="cuda")
            api.dat_step_lamb_two_sided(P.plan, th, mo, va, [gd], 0, 0, hp, t, gh_d)
            gh = np_of(gh_d)
        assert P.status() == 0
    with np.errstate(over="ignore"):
        assert np.isinf(gh * gh)[at].all()
    th_ref, mo_ref, va_ref, _ = oracle.lamb(offs, theta, mom, var, gh, t, *hp)
    assert np.array_equal(_bits(np_of(mo)), _bits(mo_ref)) and np.array_equal(_bits(np_of(va)), _bits(va_ref))
    assert_close_per_layer(np_of(th), th_ref, offs, "theta")
