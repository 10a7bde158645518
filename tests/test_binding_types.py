"""Types of the ctypes binding's public structures and signatures (CPU)."""
import ctypes

import numpy as np
import pytest

from paper_1612_01501_gb300 import ion


def test_float_pointers_are_float_pointers():
    x = np.arange(6, dtype=np.float32)
    inp = ion.ion_input()
    inp.dense = x.ctypes.data_as(ion.c_f32p)          # as a program that fills the structure itself does
    assert inp.dense[5] == 5.0
    assert ion._SIGS["ion_read_state"][1][2] is ion.c_f32p
    with pytest.raises(TypeError):                     # an array of another type is refused
        inp.dense = x.astype(np.float64).ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def test_dense_input_points_at_the_array():
    x = np.arange(6, dtype=np.float32).reshape(2, 3)
    inp, keep = ion._input_struct(dense=x)
    assert ctypes.addressof(inp.dense.contents) == x.ctypes.data and keep[0] is x
    assert [inp.dense[k] for k in range(6)] == list(range(6))


def test_dense_input_from_a_read_only_array_and_a_tensor():
    x = np.arange(6, dtype=np.float32)
    x.flags.writeable = False
    inp, _ = ion._input_struct(dense=x)
    assert ctypes.addressof(inp.dense.contents) == x.ctypes.data
    torch = pytest.importorskip("torch")
    t = torch.arange(6, dtype=torch.float32)
    assert ctypes.addressof(ion._f32(t)) == t.data_ptr()
    ion._f32(np.zeros((0,), np.float32))               # an empty array has an address too
