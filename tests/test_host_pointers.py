"""Addresses of host arrays as the binding takes them: every layout the level lists can have."""
import numpy as np
import pytest

from paper_2005_12716_gb300 import _swense as S


def _readonly():
    a = np.arange(5, dtype=np.float64)
    a.flags.writeable = False
    return a


@pytest.mark.parametrize("a", [
    np.arange(7, dtype=np.float32),
    np.arange(7, dtype=np.float64)[2:],
    np.arange(8, dtype=np.float32)[::2],
    np.arange(8, dtype=np.float32)[::-1],
    np.zeros(0, np.float32),
    np.array(1.5),
    np.ones((3, 4), np.float32, order="F"),
    np.frombuffer(b"\0" * 16, np.float32),
    _readonly(),
], ids=["plain", "offset", "strided", "reversed", "empty", "scalar", "fortran", "bytes", "readonly"])
def test_address_of_host_arrays(a):
    before = a.copy()
    assert S._ptr(a) == a.ctypes.data
    assert np.array_equal(a, before)


def test_struct_addresses():
    z, t = np.linspace(-1, 0.2, 9).astype(np.float32), np.array([0.0, 0.1])
    g = S.make_grid(16, 32, 8, 8, 9, 2, 1.0, 1.0, z, t)
    assert (g.z_levels, g.t_levels) == (z.ctypes.data, t.ctypes.data)
    d = S.make_grid_desc(1, [float(v) for v in z])          # converted: kept by the struct
    assert d.z_levels == d._keep.ctypes.data and d.nz == 9
