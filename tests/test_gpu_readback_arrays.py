"""Fields and populations read back into host arrays of every kind a copy takes: a pinned array at an
address that is no multiple of eight bytes, one that ends with its allocation, arrays
that share memory (written one after another, the last one stays)."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1809_07008_gb300 as imb
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[2, 3])
def lattice(request):
    lib = imb.load()
    if request.param == 2:
        lat = imb.Lattice.from_workload(W.c3sub(steps=0, nx=131, ny=97))
        calls = lib.imb_get_macro, lib.imb_get_populations
    else:
        lat = imb.Lattice3.from_workload(W.spheres3(nx=27, ny=19, nz=23, n=2, r_lo=2.5, r_hi=3.5, seed=5))
        calls = lib.imb3_get_macro, lib.imb3_get_populations
    lat.step(5)
    yield lat, *calls
    lat.close()


def _at(address):
    return ctypes.cast(address, ctypes.POINTER(ctypes.c_double))


def _values(buf, offset, a):
    n = a.nbytes
    return np.frombuffer(buf.numpy()[offset:offset + n].tobytes(), np.float64).reshape(a.shape)


@pytest.mark.parametrize("offset", [0, 4, 8, 12])
def test_pinned_at_any_address(lattice, offset):
    lat, macro, pops = lattice
    f, m = lat.populations(), lat.macro()
    buf = torch.zeros(f.nbytes + offset, dtype=torch.uint8).pin_memory()   # the array ends with the buffer
    assert pops(lat.h, _at(buf.data_ptr() + offset)) == 0
    assert np.array_equal(_values(buf, offset, f), f)
    bufs = [torch.zeros(a.nbytes + offset, dtype=torch.uint8).pin_memory() for a in m]
    assert macro(lat.h, *(_at(b.data_ptr() + offset) for b in bufs)) == 0
    for b, a in zip(bufs, m):
        assert np.array_equal(_values(b, offset, a), a)


def test_shared_arrays_hold_the_last_field(lattice):
    lat, macro, _ = lattice
    m = lat.macro()
    n = m[0].nbytes
    buf = torch.zeros(2 * n, dtype=torch.uint8).pin_memory()
    rest = [_at(buf.data_ptr() + n)] * (len(m) - 1)   # the velocities all into one array
    assert macro(lat.h, _at(buf.data_ptr()), *rest) == 0
    assert np.array_equal(_values(buf, 0, m[0]), m[0]) and np.array_equal(_values(buf, n, m[-1]), m[-1])
    half = (n // 2) // 8 * 8   # each array starts in the middle of the one before
    buf = torch.zeros(n + half * (len(m) - 1), dtype=torch.uint8).pin_memory()
    assert macro(lat.h, *(_at(buf.data_ptr() + k * half) for k in range(len(m)))) == 0
    want = np.zeros(len(buf) // 8)
    for k, a in enumerate(m):
        want[k * half // 8:k * half // 8 + a.size] = a.ravel()
    assert np.array_equal(_values(buf, 0, want), want)
