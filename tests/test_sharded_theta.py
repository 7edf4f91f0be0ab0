"""The pull form of the sharded step (ShardedStep.update_pull) on parameter vectors that the calls could not take as they lie:
a view that is not 16-byte aligned, a strided one.  The operations are a stand-in on the CPU with the calls' demands."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2206_06257_b200.sharded import ShardedStep

SIZES = [40, 21, 16, 51, 7]             # cut for two ranks: the first range has no pad, the second has one


class _Ops:
    def plane_bytes(self, rg):
        return 16, 16

    def aggregate_update_gather(self, rg, lv_ptrs, sg_ptrs, scales, theta_own, mom_own, hp):
        assert theta_own.data_ptr() % 16 == 0, "a device data pointer has to be 16-byte aligned"
        assert theta_own.numel() == rg.n
        raw = np.frombuffer((ctypes.c_float * rg.n).from_address(theta_own.data_ptr()), dtype=np.float32)      # what a kernel sees
        raw[rg.pad:] += 1.0


def _layouts(d):
    base = torch.arange(d, dtype=torch.float32)
    yield "aligned", base.clone()
    for k in (1, 2, 3):
        buf = torch.empty(d + 8)
        buf[k:k + d] = base
        yield "offset %d" % k, buf[k:k + d]
    buf = torch.empty(2 * d)
    buf[::2] = base
    yield "strided", buf[::2]


@pytest.mark.parametrize("rank", [0, 1])
def test_update_pull_takes_any_theta(rank):
    offs = np.concatenate([[0], np.cumsum(SIZES)])
    d = int(offs[-1])
    for what, theta in _layouts(d):
        s = ShardedStep(_Ops(), offs, 2, rank, 2)
        assert (s.own.pad == 0) == (rank == 0)
        want = torch.arange(d, dtype=torch.float32)
        want[s.own.a:s.own.b] += 1.0
        s.update_pull(torch.ones(len(SIZES)), [(0, 0), (0, 0)], theta, None, None)
        assert torch.equal(theta, want), what
