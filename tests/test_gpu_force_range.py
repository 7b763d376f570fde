"""The force on a disk is summed to FP64 beyond a warp's partial sums: it stays a number where the
disk's total lies beyond the range of FP32 while every partial sum is within it (a fluid of density
3e36 at rest around a disk that moves at one cell a step, the first step), against the FP64 oracle."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("units", [1, 2])
def test_total_beyond_fp32(orc, units):
    # per row 20 cells of 3e36 at most, 1.2e38 a warp, 4.8e38 in eight rows and 9.4e38 in all
    w = W.Workload(name="heavy", nx=96, ny=96, tau=0.8, bc_x=W.BC_WALL, bc_y=W.BC_WALL, rho0=3.0e36, dem_on=0,
                   x=np.array([[48.0, 47.5]]), v=np.array([[1.0, 0.0]]), omega=np.zeros(1), r=np.array([10.0]))
    o, g = orc.Sim(w), imb.Lattice.from_workload(w, work_units=units)
    o.step(1)
    g.step(1)
    Fo, Fg = o.forces()[0], g.forces()[0]
    assert abs(Fo[0, 0]) > 3.5e38
    assert abs(Fg[0, 0] - Fo[0, 0]) <= 1e-5 * abs(Fo[0, 0])
    g.close()
