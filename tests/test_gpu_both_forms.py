"""GPU: the oracle's parity cases of the step calls in each of their two forms -- the one launch, and a launch per phase --
whatever form the rule takes at these small sizes.  Every plan of a case gets the form by the test hook; what is compared,
and how closely, stands at the cases themselves."""
import pytest
import torch

import test_gpu_parity as parity
from helpers import GpuPlan, assert_close_per_layer, np_of
from test_gpu_parity import api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[1, 2], ids=["one_launch", "phases"])
def form(request, api, monkeypatch):  # noqa: F811
    create = api.dat_plan_create

    def create_with_form(*args, **kw):
        plan = create(*args, **kw)
        api.dat_plan_test_form(plan, request.param)
        return plan
    monkeypatch.setattr(api, "dat_plan_create", create_with_form)
    return request.param


@pytest.mark.parametrize("bits", [1, 2, 4, 8, 16, 32])
def test_ragged(api, oracle, form, bits, rng_bits):  # noqa: F811
    parity.test_fused_parity_ragged(api, oracle, bits, rng_bits)


@pytest.mark.parametrize("M", [1, 2, 5, 8, 13, 32, 64])
def test_worker_counts(api, oracle, form, M, rng_bits):  # noqa: F811
    parity.test_fused_parity_worker_counts(api, oracle, M, rng_bits)


@pytest.mark.parametrize("M", [9, 13, 64])
def test_b32_more_than_eight_workers(api, oracle, form, M):  # noqa: F811
    parity.test_fused_b32_more_than_eight_workers(api, oracle, M)


@pytest.mark.parametrize("bits", [2, 8, 16])
def test_extreme_scales(api, oracle, form, bits, rng_bits):  # noqa: F811
    parity.test_fused_parity_extreme_scales(api, oracle, bits, rng_bits)


@pytest.mark.parametrize("bits", [1, 4, 8, 16])
def test_per_worker_norms(api, oracle, form, bits, rng_bits):  # noqa: F811
    parity.test_unfused_parity_per_worker_scales(api, oracle, bits, rng_bits)


@pytest.mark.parametrize("mode", ["shared", "per_worker", "b32"])
def test_lamb(api, oracle, form, mode):  # noqa: F811
    parity.test_step_lamb_parity_three_steps(api, oracle, mode)


@pytest.mark.parametrize("mode", ["shared", "per_worker"])
@pytest.mark.parametrize("bits", [1, 8, 16])
def test_two_sided(api, oracle, form, bits, mode, rng_bits):  # noqa: F811
    parity.test_step_two_sided_parity(api, oracle, bits, mode, rng_bits)


def test_lamb_two_sided(api, oracle, form):  # noqa: F811
    parity.test_step_lamb_two_sided_parity(api, oracle)


def test_zero_layers_and_nonfinite_inputs(api, oracle, form):  # noqa: F811
    parity.test_zero_norm_conventions(api, oracle)
    parity.test_all_zero_everything(api, oracle)
    parity.test_nonfinite_input_sets_status_bit(api)


@pytest.mark.parametrize("bits", [1, 4, 8])
def test_nothing_outside_the_buffers(api, form, bits):  # noqa: F811
    parity.test_nothing_is_written_outside_the_callers_buffers(api, bits, 16)


@pytest.mark.parametrize("wait_cycles", [2_000_000, 0])
def test_one_launch_recovers_from_a_wait_that_ran_out(api, oracle, wait_cycles):  # noqa: F811
    """The ticket, the counters and the ready words of the one launch after a call that gave up (0: after the default two
    seconds), on a plan whose steps would go by phases."""
    offs, grads, theta, mom = parity._random_problem(77, [5000, 300, 9000, 40], 3)
    g_dev = [torch.from_numpy(g).cuda() for g in grads]
    with GpuPlan(api, offs, 3, 8) as P, GpuPlan(api, offs, 3, 8) as P2:
        api.dat_plan_test_stall(P.plan, wait_cycles, 2)
        th, mo = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda()
        api.dat_step(P.plan, th, mo, g_dev, 5, 9, parity.HP)
        assert P.status() & api.DAT_STATUS_TIMEOUT
        assert P.status() == 0
        api.dat_plan_test_stall(P.plan, 0, -1)
        for step in (9, 10):
            th1, mo1 = torch.from_numpy(theta).cuda(), torch.from_numpy(mom).cuda()
            th2, mo2 = th1.clone(), mo1.clone()
            api.dat_step_pipelined(P.plan, th1, mo1, g_dev, 5, step, parity.HP)
            api.dat_step_pipelined(P2.plan, th2, mo2, g_dev, 5, step, parity.HP)
            assert P.status() == 0 and P2.status() == 0
            assert torch.equal(th1, th2) and torch.equal(mo1, mo2)
            ref = oracle.step(offs, theta, mom, grads, 8, 5, step, *parity.HP)
            assert_close_per_layer(np_of(th1), ref["theta"], offs, "theta after recovery")
