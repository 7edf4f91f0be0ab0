"""GPU: quantizer norms where a CTA sums several tiles -- few workers, more tiles than the GPU holds -- against 64-bit sums:
layers that end inside a CTA's tiles, many of them, one that spans several CTAs; every norm within a last place."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan, np_of, ulp_diff

pytestmark = pytest.mark.gpu
TILE = 4096


@pytest.mark.parametrize("M", [1, 2, 3, 5])
@pytest.mark.parametrize("tail", [1, 7 * TILE + 5])
def test_norms_of_several_tiles_per_cta(M, tail):
    from paper_2206_06257_b200 import api
    rng = np.random.RandomState(M)
    # 9472 tiles fill 148 SMs eight times over with eight tiles per CTA and one worker
    sizes = [3, TILE, 2 * TILE - 1, 5] + list(rng.randint(1, 3 * TILE, 300)) + [6000 * TILE // M + 11] + list(rng.randint(1, 40, 50)) + [4000 * TILE // M, tail]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    g = torch.Generator(device="cuda").manual_seed(M)
    grads = [torch.randn(int(offs[-1]), generator=g, device="cuda") * 10.0 ** (i - 2) for i in range(M)]
    want = np.stack([[float(torch.linalg.vector_norm(x[a:b].double())) for a, b in zip(offs[:-1], offs[1:])] for x in grads]).astype(np.float32)
    with GpuPlan(api, offs, M, 8) as P:
        got = torch.zeros(M * len(sizes), device="cuda")
        for _ in range(2):                      # the counters are back at zero after the first
            api.dat_worker_norms(P.plan, grads, got.zero_())
            assert ulp_diff(np_of(got).reshape(M, -1), want).max() <= 1
        assert P.status() == 0
