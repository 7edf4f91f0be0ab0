"""GPU: which form a step takes by the rule, on both sides of its lines: the launches of a call (one launch: 1; by phases: 3, of a
two-sided step 4)."""
import numpy as np
import pytest
import torch

from helpers import GpuPlan
from test_gpu_parity import HP, LAMB_HP, api  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _launches(api, sizes, M, kind):  # noqa: F811
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    d = int(offs[-1])
    th, mo, va, gh = (torch.full((d,), 1e-3, device="cuda") for _ in range(4))
    grads = [torch.full((d,), 1e-3 * (i + 1), device="cuda") for i in range(M)]
    with GpuPlan(api, offs, M, 8) as P:
        n = api.dat_plan_launch_count(P.plan)
        if kind == "step":
            api.dat_step(P.plan, th, mo, grads, 1, 0, HP)
        elif kind == "lamb":
            api.dat_step_lamb(P.plan, th, mo, va, grads, 1, 0, LAMB_HP, 1)
        elif kind == "two":
            api.dat_step_two_sided(P.plan, th, mo, grads, 1, 0, HP, gh)
        else:
            api.dat_step_lamb_two_sided(P.plan, th, mo, va, grads, 1, 0, LAMB_HP, 1, gh)
        assert P.status() == 0
        return api.dat_plan_launch_count(P.plan) - n


@pytest.mark.parametrize("kind,M,tiles,share,launches", [
    ("step", 2, 10, 0.2, 1), ("step", 2, 10, 0.3, 3), ("step", 2, 20, 0.3, 3), ("step", 2, 8, 0.2, 3), ("step", 1, 20, 0.05, 3),
    ("two", 2, 8, 0.2, 4), ("two", 2, 10, 0.2, 1), ("two", 2, 10, 0.3, 4), ("two", 2, 26, 0.3, 1), ("two", 2, 26, 0.4, 4), ("two", 16, 26, 0.3, 4),
    ("two", 1, 10, 0.05, 4), ("two", 1, 20, 0.05, 1), ("two", 1, 20, 0.2, 4), ("lamb_two", 1, 20, 0.05, 4), ("lamb_two", 2, 26, 0.3, 4),
    ("lamb", 2, 20, 0.3, 3), ("lamb", 2, 20, 0.2, 1)])
def test_large_layers_and_few_workers(api, kind, M, tiles, share, launches):  # noqa: F811
    """tiles: of 4096 elements, per SM; share: the largest layer's, the others at most 0.04 each."""
    n = tiles * torch.cuda.get_device_properties(0).multi_processor_count - 40
    big, rest = int(4096 * n * share), 4096 * n - int(4096 * n * share)
    assert _launches(api, [rest // 25 + 8 * (k % 3) for k in range(25)] + [big], M, kind) == launches


@pytest.mark.parametrize("kind,M,layers,pieces,launches", [
    ("step", 16, 1, 48, 3), ("step", 16, 1, 49, 1), ("step", 15, 1, 48, 1), ("lamb", 16, 3, 48, 3), ("two", 16, 1, 48, 1), ("two", 32, 1, 48, 4),
    ("two", 32, 1, 49, 1), ("step", 48, 2, 400, 1), ("step", 48, 2, 401, 3), ("step", 47, 2, 401, 1), ("step", 1, 50, 99, 1), ("step", 1, 50, 100, 3),
    ("step", 1, 50, 101, 1), ("lamb_two", 2, 100, 200, 4), ("lamb_two", 2, 100, 201, 1), ("step", 3, 100, 200, 1), ("step", 2, 3, 48, 1),
    ("step", 2, 3, 49, 3), ("step", 2, 3, 249, 3), ("step", 2, 3, 250, 1), ("lamb", 2, 3, 100, 1), ("two", 2, 3, 100, 1)])
def test_small_steps(api, kind, M, layers, pieces, launches):  # noqa: F811
    """pieces: of 2048 elements, spread over the layers (each of whole pieces)."""
    if pieces > 3 * torch.cuda.get_device_properties(0).multi_processor_count:
        pytest.skip("the device holds fewer")
    sizes = [2048 * (pieces // layers + (k < pieces % layers)) for k in range(layers)]
    assert _launches(api, sizes, M, kind) == launches
