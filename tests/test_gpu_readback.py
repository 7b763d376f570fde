"""Fields and populations read back into pinned arrays (written by the kernel itself), into pageable
ones, and into a mix of both: the same values to the bit."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1809_07008_gb300 as imb
import workloads as W

pytestmark = pytest.mark.gpu


def _ptr(a):
    addr = a.data_ptr() if isinstance(a, torch.Tensor) else a.ctypes.data
    return ctypes.cast(addr, ctypes.POINTER(ctypes.c_double))


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("dim", [2, 3])
def test_pinned_equals_pageable(dim, storage):
    lib = imb.load()
    if dim == 2:
        lat = imb.Lattice.from_workload(W.c3sub(steps=0, nx=131, ny=97), storage=storage)
        macro, pops = lib.imb_get_macro, lib.imb_get_populations
    else:
        lat = imb.Lattice3.from_workload(W.spheres3(nx=27, ny=19, nz=23, n=2, r_lo=2.5, r_hi=3.5, seed=5), storage=storage)
        macro, pops = lib.imb3_get_macro, lib.imb3_get_populations
    lat.step(5)
    f, m = lat.populations(), lat.macro()
    pf = torch.full(f.shape, np.nan, dtype=torch.float64).pin_memory()
    assert pops(lat.h, _ptr(pf)) == 0 and np.array_equal(pf.numpy(), f)
    for pageable in ((), (1,)):   # all pinned; one array pageable
        out = [np.full(a.shape, np.nan) if k in pageable else torch.full(a.shape, np.nan, dtype=torch.float64).pin_memory()
               for k, a in enumerate(m)]
        assert macro(lat.h, *(_ptr(a) for a in out)) == 0
        for a, b in zip(out, m):
            assert np.array_equal(np.asarray(a), b)
    lat.close()
