"""The force on a disk (a sphere) is summed to FP64 beyond a warp's partial sums: it stays a number where
the total lies beyond the range of FP32 while every partial sum is within it (a fluid of density
3e36 or 8e36 at rest around a body that moves at one cell a step, the first step), against the FP64
oracle."""
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


@pytest.mark.parametrize("n", [1, 2])   # the plain kernel, and the general one (a second sphere shares cells)
@pytest.mark.parametrize("rho0", [8.0e36, 3.0e37])
def test_sphere_total_beyond_fp32(orc, rho0, n):
    # 1.6e38 (6e38) along a row of 20 cells, 6.4e37 (2.4e38) along a column of eight, eight times the row
    # in a warp's columns
    x, v, R = np.array([[32.0, 16.2, 15.7], [44.6, 16.2, 15.7]]), np.array([[1.0, 0.0, 0.0], [0.5, 0.0, 0.0]]), np.array([10.0, 3.0])
    w = W.Workload3(name="heavy3", nx=64, ny=32, nz=32, tau=0.8, wall_y=True, rho0=rho0, x=x[:n], v=v[:n], omega=np.zeros((n, 3)),
                    R=R[:n])
    o, g = orc.Sim3(w), imb.Lattice3.from_workload(w)
    o.step(1)
    g.step(1)
    Fo, Fg = o.forces()[0], g.forces()[0]
    assert np.abs(Fo[:, 0]).min() > (1e40 if n == 1 else 3.5e38)
    assert np.abs(Fg[:, 0] / Fo[:, 0] - 1).max() <= 1e-5
    g.close()
