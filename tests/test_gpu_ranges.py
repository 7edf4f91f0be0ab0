"""GPU: dat_quantize_ranges against dat_quantize on each range (whole bytes, no tolerance)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,rng_bits,M,world", [(8, 16, 1, 8), (4, 23, 3, 3), (1, 16, 2, 5), (16, 16, 5, 40), (2, 23, 64, 33)])
def test_ranges_equal_separate_calls(bits, rng_bits, M, world):
    """Ranges with and without a pad, of one layer and of several, more of them than one launch takes; the last one ragged."""
    from paper_2206_06257_b200 import api
    from paper_2206_06257_b200.sharded import CudaOps, RangeLayout, partition_layers
    rng = np.random.RandomState(world)
    sizes = rng.randint(1, 9000, size=max(world, 11))
    sizes[3] = 70001
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d, h = int(offs[-1]), sizes.size
    grads = [torch.from_numpy((rng.standard_normal(d) * 1e-2).astype(np.float32)).cuda() for _ in range(M)]
    nu = torch.from_numpy(rng.uniform(0.5, 2.0, size=h).astype(np.float32)).cuda()
    nu[2] = 0.0
    ranges = [RangeLayout(offs, l0, l1) for l0, l1 in partition_layers(offs, world)]
    assert any(r.pad for r in ranges) and any(not r.pad for r in ranges)
    ops = CudaOps(api, offs, M, M, 0, 1, bits, rng_bits)
    try:
        got = ops.quantize_ranges(ranges, grads, nu, 77, 3)
        for q, rg in enumerate(ranges):
            lv, sg = ops.quantize_range(q, rg, grads, rg.scales(nu).contiguous(), 77, 3)
            assert torch.equal(lv, got[q][0]) and torch.equal(sg, got[q][1]), q
    finally:
        ops.close()
