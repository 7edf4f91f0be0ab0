"""Host arrays that the binding hands to the library: of the entry's element type and length, whatever the caller's are."""
import ctypes as C
from types import SimpleNamespace

import pytest

from paper_2206_06257_b200 import api


@pytest.fixture
def ranges(monkeypatch):
    """dat_quantize_ranges up to the library: (plans, first_layer, padded, levels) as the C function would read them."""
    seen = []

    def record(n, plans, first_layer, padded, grads, seed, step, norms, levels, signs, stream):
        size = {api._i64: 8, C.c_int32: 4, C.c_void_p: 8}
        out = []
        for arg, ctype in ((plans, C.c_void_p), (first_layer, api._i64), (padded, C.c_int32), (levels, C.c_void_p)):
            assert C.sizeof(arg) >= n * size[ctype]                       # nothing is read past the array's end
            out.append(list((ctype * n).from_buffer_copy(arg)))
        seen.append(out)
        return api.DAT_OK
    monkeypatch.setattr(api, "_lib", SimpleNamespace(dat_quantize_ranges=record))

    def call(plans, first_layer, padded, levels):
        api.dat_quantize_ranges(plans, first_layer, padded, [16], 0, 0, 16, levels, [16] * len(plans), stream=0)
        return seen.pop()
    return call


@pytest.mark.parametrize("make", [list, tuple, C.c_int64 * 3, C.c_int32 * 3, C.c_uint8 * 3])
def test_layers_and_flags_of_any_element_type(ranges, make):
    xs = [2, 0, 1]
    arr = make(*xs) if isinstance(make, type(C.Array)) else make(xs)
    assert ranges([1, 2, 3], arr, arr, [16, 32, 48]) == [[1, 2, 3], xs, xs, [16, 32, 48]]


@pytest.mark.parametrize("ctype", [C.c_void_p, C.c_uint64, C.c_uint32])
def test_addresses_of_any_element_type(ranges, ctype):
    arr = (ctype * 2)(64, 128)
    assert ranges(arr, [0, 1], [0, 0], arr) == [[64, 128], [0, 1], [0, 0], [64, 128]]


def test_short_arrays_are_filled_up_and_long_ones_refused(ranges):
    assert ranges([1, 2], (C.c_int64 * 1)(5), (C.c_int32 * 1)(1), [16, 32])[1:3] == [[5, 0], [1, 0]]
    for first, pad in (((C.c_int64 * 3)(), [0, 0]), ([0, 0], (C.c_int32 * 3)())):
        with pytest.raises(IndexError):
            ranges([1, 2], first, pad, [16, 32])
