"""GPU: dat_step_host on vectors large enough to go in several groups of layers equals dat_step on device buffers (bits)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MB = 1 << 18                                            # elements of a megabyte of fp32
HP = (0.1, 0.9, 5e-4, 0.0, 10.0)


@pytest.mark.parametrize("sizes,bits", [([5 * MB + 3], 8), ([3, MB + 1, 2 * MB - 5, 7, MB, MB // 2, 9 * MB + 5, 31], 8),
                                        ([MB // 3 + k for k in range(60)], 4), ([2 * MB + 1, 2 * MB - 1], 32), ([1000, 77], 2)])
def test_host_groups_equal_device_call(sizes, bits):
    """One layer only; layers larger and smaller than a group; as many groups as there can be; b = 32; one group."""
    from paper_2206_06257_b200 import api
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, M = int(offs[-1]), 3
    g = torch.Generator().manual_seed(5)
    theta, mom = torch.randn(d, generator=g) * 0.05, torch.randn(d, generator=g) * 1e-3
    grads = [torch.randn(d, generator=g) * 1e-2 for _ in range(M)]
    plan = api.dat_plan_create(offs, M, bits)
    try:
        th_d, mo_d, g_d = theta.cuda(), mom.cuda(), [x.cuda() for x in grads]
        th_h, mo_h, g_h = theta.clone().pin_memory(), mom.clone().pin_memory(), [x.pin_memory() for x in grads]
        for step in (4, 5):
            api.dat_step(plan, th_d, mo_d, g_d, 9, step, HP)
            api.dat_step_host(plan, th_h, mo_h, g_h, 9, step, HP)
            assert torch.equal(th_h, th_d.cpu()) and torch.equal(mo_h, mo_d.cpu())
        assert api.dat_get_status(plan) == 0
    finally:
        api.dat_plan_destroy(plan)
