"""Argument conversions of the Python binding: the same C values from every kind
of sequence, element counts enforced (CPU)."""
import ctypes

import numpy as np
import pytest

import paper_2605_04178_gb300 as pm

I32, I16 = ctypes.c_int32, ctypes.c_int16


@pytest.mark.parametrize("values", [[3, 70, 5], (3, 70, 5), np.array([3, 70, 5]), np.array([3, 70, 5], dtype=np.uint8),
                                    [np.int64(3), np.int16(70), 5], np.array([3.9, 70.2, 5.0]), [3.9, 70.2, 5.0],
                                    np.array([3, 70, 5, 9, 9])[:3], np.array([3, 0, 70, 0, 5])[::2]])
@pytest.mark.parametrize("ctype", [I32, I16])
def test_integer_arrays(values, ctype):
    assert list(pm._ints(values, 3, ctype)) == [3, 70, 5]


def test_integer_arrays_sizes_and_overflow():
    assert list(pm._ints([1], 3, I32)) == [1, 0, 0]            # a short list is zero-filled, never read past its end
    with pytest.raises(IndexError):
        pm._ints([1, 2, 3, 4], 3, I32)
    assert list(pm._ints([65536 + 128], 1, I16)) == [128] == list(pm._ints(np.array([65536 + 128]), 1, I16))


@pytest.mark.parametrize("theta", [list, tuple, np.array, lambda v: np.array(v, dtype=np.float32),
                                   lambda v: np.repeat(np.array(v), 2)[::2]])
def test_parameters(theta):
    v = [0.1 * (j + 1) for j in range(pm.N_PARAMS)]
    assert list(pm.params(theta(v)).v) == [np.float32(x) for x in v]
    want = [float(x) for x in theta(v)]
    assert list(pm._params_f64(theta(v))) == want
    with pytest.raises(AssertionError):
        pm.params(theta(v)[:-1])
    with pytest.raises(AssertionError):
        pm._params_f64(theta(v)[:-1])
