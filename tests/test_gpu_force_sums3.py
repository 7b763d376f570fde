"""Force sums of the D3Q19 kernel along its columns of eight cells: columns that meet one, two and
more spheres (a third one in a column takes another way), cells shared by two spheres, a lattice
whose last column is short and whose last warp is not full, against the FP64 oracle."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def stack(nx, ny, nz, R, pitch, n, C_smag, per_row=3):
    """Rows of n spheres of radius R, `pitch` apart along z, the rows spread along x."""
    x = np.array([[(k + 0.53) * nx / per_row, ny / 2 + 0.21, 1.7 + j * pitch] for k in range(per_row) for j in range(n)])
    v = 0.002 * np.stack([np.cos(np.arange(len(x))), np.sin(np.arange(len(x))), np.cos(2 + np.arange(len(x)))], 1)
    return W.Workload3(name="stack", nx=nx, ny=ny, nz=nz, tau=0.6, wall_y=True, force=(2e-5, 0.0, 1e-5), C_smag=C_smag,
                       x=x, v=v, omega=0.1 * v, R=np.full(len(x), R))


@pytest.mark.parametrize("C_smag", [0.0, 0.1])
@pytest.mark.parametrize("nx,ny,nz,R,pitch,n", [(45, 13, 21, 1.3, 3.0, 7),    # three and four spheres to a column of eight
                                                (64, 16, 24, 1.4, 2.7, 8),    # neighbours share cells (2.7 < 2 R)
                                                (33, 17, 19, 4.6, 9.5, 2)])   # one or two to a column
def test_column_force_sums(nx, ny, nz, R, pitch, n, C_smag):
    w = stack(nx, ny, nz, R, pitch, n, C_smag)
    g, o = imb.Lattice3.from_workload(w), O.Sim3(w)
    g.step(3)
    o.step(3)
    (Fg, Tg), (Fo, To) = g.forces(), o.forces()
    # FP32 terms: the bar of the other D3Q19 force tests, relative to the largest force (torque)
    assert np.abs(Fg - Fo).max() <= 1e-4 * np.abs(Fo).max()
    assert np.abs(Tg - To).max() <= 1e-4 * max(np.abs(To).max(), np.abs(Fo).max())
    g.close()
