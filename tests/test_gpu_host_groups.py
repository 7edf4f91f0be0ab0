"""GPU: dat_step_host on vectors large enough to go in several groups of layers (each in the one launch) equals
dat_step_pipelined on device buffers, and dat_step where it goes in one: small vectors, pageable memory (bits)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MB4 = 1 << 20                                           # elements of four megabytes of fp32: the smallest group
HP = (0.1, 0.9, 5e-4, 0.0, 10.0)


@pytest.mark.parametrize("sizes,bits", [([5 * MB4 + 3], 8), ([3, MB4 + 1, 2 * MB4 - 5, 7, MB4, MB4 // 2, 9 * MB4 + 5, 31], 8),
                                        ([MB4 // 3 + k for k in range(60)], 4), ([2 * MB4 + 1, 2 * MB4 - 1], 32), ([1000, 77], 2)])
@pytest.mark.parametrize("pinned", ["all", "none", "all but one"])
def test_host_groups_equal_device_call(sizes, bits, pinned):
    """One layer only; layers larger and smaller than a group; as many groups as there can be; b = 32; one group."""
    from paper_2206_06257_b200 import api
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, M = int(offs[-1]), 3
    g = torch.Generator().manual_seed(5)
    theta, mom = torch.randn(d, generator=g) * 0.05, torch.randn(d, generator=g) * 1e-3
    grads = [torch.randn(d, generator=g) * 1e-2 for _ in range(M)]
    plan = api.dat_plan_create(offs, M, bits)
    dat_step = api.dat_step_pipelined if pinned == "all" and d >= 2 * MB4 else api.dat_step
    pin = lambda x: x if pinned == "none" else x.pin_memory()  # noqa: E731
    try:
        th_d, mo_d, g_d = theta.cuda(), mom.cuda(), [x.cuda() for x in grads]
        th_h, mo_h, g_h = pin(theta.clone()), pin(mom.clone()), [pin(x) for x in grads[:-1]] + [grads[-1] if pinned == "all but one" else pin(grads[-1])]
        for step in (4, 5):
            dat_step(plan, th_d, mo_d, g_d, 9, step, HP)
            api.dat_step_host(plan, th_h, mo_h, g_h, 9, step, HP)
            assert torch.equal(th_h, th_d.cpu()) and torch.equal(mo_h, mo_d.cpu())
        assert api.dat_get_status(plan) == 0
    finally:
        api.dat_plan_destroy(plan)
