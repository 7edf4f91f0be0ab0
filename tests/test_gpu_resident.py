"""GPU: the oracle's parity cases of the step calls in the resident form (one launch whose CTAs keep their pieces), and its
largest problems against the form of a launch per phase."""
import numpy as np
import pytest
import torch

import test_gpu_parity as parity
from helpers import GpuPlan, assert_close_per_layer, np_of, ulp_diff
from test_gpu_parity import api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
RESIDENT, PHASES = 3, 2


@pytest.fixture
def resident(api, monkeypatch):  # noqa: F811
    create = api.dat_plan_create

    def create_with_form(*args, **kw):
        plan = create(*args, **kw)
        api.dat_plan_test_form(plan, RESIDENT)
        return plan
    monkeypatch.setattr(api, "dat_plan_create", create_with_form)


@pytest.mark.parametrize("bits", [1, 8, 16, 32])
def test_ragged(api, oracle, resident, bits, rng_bits):  # noqa: F811
    parity.test_fused_parity_ragged(api, oracle, bits, rng_bits)


@pytest.mark.parametrize("M", [1, 3, 8, 33, 64])
def test_worker_counts(api, oracle, resident, M, rng_bits):  # noqa: F811
    parity.test_fused_parity_worker_counts(api, oracle, M, rng_bits)


@pytest.mark.parametrize("bits", [2, 16])
def test_extreme_scales(api, oracle, resident, bits, rng_bits):  # noqa: F811
    parity.test_fused_parity_extreme_scales(api, oracle, bits, rng_bits)


@pytest.mark.parametrize("mode", ["shared", "per_worker", "b32"])
def test_lamb(api, oracle, resident, mode):  # noqa: F811
    parity.test_step_lamb_parity_three_steps(api, oracle, mode)


@pytest.mark.parametrize("mode", ["shared", "per_worker"])
def test_two_sided(api, oracle, resident, mode, rng_bits):  # noqa: F811
    parity.test_step_two_sided_parity(api, oracle, 8, mode, rng_bits)
    parity.test_step_lamb_two_sided_parity(api, oracle)


def test_zero_layers_nonfinite_inputs_margins_and_capture(api, oracle, resident):  # noqa: F811
    parity.test_zero_norm_conventions(api, oracle)
    parity.test_all_zero_everything(api, oracle)
    parity.test_nonfinite_input_sets_status_bit(api)
    parity.test_nothing_is_written_outside_the_callers_buffers(api, 8, 16)
    parity.test_step_refuses_stream_capture(api)


def test_a_wait_that_runs_out_is_reported_and_the_plan_recovers(api, oracle):  # noqa: F811
    """A layer whose norm never completes: the status says so, and the next step is the oracle's again."""
    offs, grads, theta, mom = parity._random_problem(5, [4096, 9000, 70], 3)
    with GpuPlan(api, offs, 3, 8) as P:
        th, mo, g = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda(), [torch.from_numpy(x).cuda() for x in grads]
        api.dat_plan_test_stall(P.plan, 2_000_000, 1)
        api.dat_plan_test_form(P.plan, RESIDENT)
        api.dat_step(P.plan, th, mo, g, 3, 5, parity.HP)
        assert api.dat_get_status(P.plan) & api.DAT_STATUS_TIMEOUT
        th, mo, sc = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda(), torch.zeros(P.h, device="cuda")
        api.dat_step(P.plan, th, mo, g, 3, 5, parity.HP, None, None, sc)
        assert P.status() == 0
        ref = oracle.step(offs, theta, mom, grads, 8, 3, 5, *parity.HP, scales_in=np_of(sc))
        assert np.array_equal(np_of(mo), ref["mom"])
        assert_close_per_layer(np_of(th), ref["theta"], offs, "theta")


@pytest.mark.parametrize("pieces", [2, 149, 443, 444])
@pytest.mark.parametrize("kind", ["step", "lamb", "two_sided"])
def test_up_to_the_most_pieces_equals_the_phases(api, pieces, kind):  # noqa: F811
    """Up to three pieces per SM.  Codes depend on the norms' bits, which are sums in another order; with the norms' bits
    equal, moments are equal, and theta within the rounding of the layers' norms."""
    pieces = pieces if pieces < 443 else pieces - 444 + 3 * torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [2048 * (pieces // 3) + 5, 2048 * (pieces - 2 - pieces // 3) - 11, 7] if pieces > 2 else [2043, 9]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, M = int(offs[-1]), 3
    gen = torch.Generator(device="cuda").manual_seed(pieces)
    rnd = lambda s: torch.randn(d, generator=gen, device="cuda") * s  # noqa: E731
    theta, mom, var, grads = rnd(0.05), rnd(1e-3), rnd(1e-3).square(), [rnd(1e-2) for _ in range(M)]
    out = {}
    for form in (PHASES, RESIDENT):
        with GpuPlan(api, offs, M, 8) as P:
            api.dat_plan_test_form(P.plan, form)
            th, mo, va, gh, sc = theta.clone(), mom.clone(), var.clone(), torch.zeros_like(theta), torch.zeros(P.h, device="cuda")
            if kind == "step":
                api.dat_step(P.plan, th, mo, grads, 7, 3, parity.HP, None, None, sc)
            elif kind == "lamb":
                api.dat_step_lamb(P.plan, th, mo, va, grads, 7, 3, parity.LAMB_HP, 4, None, None, sc)
            else:
                api.dat_step_two_sided(P.plan, th, mo, grads, 7, 3, parity.HP, gh, None, None, sc)
            assert P.status() == 0
            out[form] = [np_of(x) for x in (th, mo, va, gh, sc)]
    a, b = out[PHASES], out[RESIDENT]
    assert ulp_diff(a[4], b[4]).max() <= 1
    same = np.array_equal(a[4], b[4])
    if same and kind != "two_sided":
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
    for k, name in enumerate(("theta", "momentum", "var", "g_hat")):
        if same:
            assert_close_per_layer(b[k], a[k], offs, name)


def test_a_larger_problem_has_no_resident_form(api):  # noqa: F811
    n = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    with GpuPlan(api, np.array([0, 2048 * n + 1], dtype=np.int64), 2, 8) as P:
        with pytest.raises(api.DatError) as e:
            api.dat_plan_test_form(P.plan, RESIDENT)
        assert e.value.code == api.DAT_ERR_ARG
