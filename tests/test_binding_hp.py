"""The binding's hyper-parameter structs: every value as the caller gave it, whatever was converted before."""
import ctypes

import numpy as np
import pytest


@pytest.mark.parametrize("first", [0.0, -0.0])
def test_signed_zeros_stay_apart(first):
    from paper_2206_06257_b200 import api
    for lr in (first, -first, first):
        hp = api._hp((lr, 0.9, -lr, 0.0, 10.0))
        assert np.signbit(hp.lr) == np.signbit(lr) and np.signbit(hp.weight_decay) == np.signbit(-lr)


def test_values_as_float32():
    from paper_2206_06257_b200 import api
    for hp in [(0.1, 0.9, 5e-4, 0.0, 10.0), [1, True, np.float32(0.3), np.float64(1e-40), 1e39], (0.1, float("nan"), 0.0, 0.0, float("inf")), (0.5, 0.25)]:
        got = api._hp(hp)
        want = [ctypes.c_float(float(v)).value for v in hp] + [0.0] * (5 - len(hp))
        assert np.array_equal([got.lr, got.momentum, got.weight_decay, got.c_l, got.c_u], want, equal_nan=True)
        assert api._hp(got) is got
    with pytest.raises(TypeError):
        api._hp((1, 2, 3, 4, 5, 6))
