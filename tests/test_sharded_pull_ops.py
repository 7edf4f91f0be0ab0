"""ShardedStep.step_pull on one rank with operations that quantize range by range (the oracle's): the call drives any
object with the operations' interface, and the step is the unsharded oracle's bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2206_06257_b200.sharded import ShardedStep
from sharded_oracle_ops import OracleOps
from test_sharded import HP, _problem


class _Ops(OracleOps):
    def quantize_range(self, q, rg, grads_local, scales, seed, step, out=None):
        planes = super().quantize_range(q, rg, grads_local, scales, seed, step)
        for dst, src in zip(out, planes):
            dst.copy_(src)
        return out

    def aggregate_update_gather(self, rg, lv_ptrs, sg_ptrs, scales, theta_own, mom_own, hp):
        lb, sb = self.plane_bytes(rg)
        read = lambda ptrs, n: torch.from_numpy(np.concatenate([np.frombuffer((ctypes.c_uint8 * n).from_address(p), dtype=np.uint8) for p in ptrs]))  # noqa: E731
        self.aggregate_update(rg, read(lv_ptrs, lb), read(sg_ptrs, sb), scales, theta_own, mom_own, hp)


def test_step_pull_drives_operations_that_quantize_range_by_range(oracle):
    M, bits = 3, 4
    offs, grads, theta, mom = _problem(8, M)
    s = ShardedStep(_Ops(offs, M, M, 0, 1, bits), offs, M, 0, 1)
    th, mo = torch.from_numpy(theta.copy()), torch.from_numpy(mom.copy())
    for t in range(2):
        s.step_pull(th, mo, [torch.from_numpy(g) for g in grads], 11, t, HP)
        ref = oracle.step(offs, theta, mom, grads, bits, 11, t, *HP)
        theta, mom = ref["theta"], ref["mom"]
        assert np.array_equal(th.numpy().view(np.uint32), theta.view(np.uint32)) and np.array_equal(mo.numpy().view(np.uint32), mom.view(np.uint32))


@pytest.mark.gpu
def test_step_pull_on_one_gpu_equals_the_unsharded_step():
    from paper_2206_06257_b200 import api
    from paper_2206_06257_b200.sharded import CudaOps
    from helpers import GpuPlan
    M, bits = 3, 4
    offs, grads, theta, mom = _problem(8, M)
    g = [torch.from_numpy(x).cuda() for x in grads]
    ops = CudaOps(api, offs, M, M, 0, 1, bits)
    try:
        s = ShardedStep(ops, offs, M, 0, 1)
        th, mo, th2, mo2 = (torch.from_numpy(x.copy()).cuda() for x in (theta, mom, theta, mom))
        with GpuPlan(api, offs, M, bits) as P:
            for t in range(2):
                s.step_pull(th, mo, g, 11, t, HP)
                api.dat_quantize(P.plan, g, 11, t, *(msg := P.alloc_message()))
                gh = torch.empty(int(offs[-1]), device="cuda")
                api.dat_aggregate(P.plan, *msg, None, gh)
                api.dat_lalr_step(P.plan, th2, mo2, gh, HP)
            torch.cuda.synchronize()
        assert torch.equal(th, th2) and torch.equal(mo, mo2)
    finally:
        ops.close()
