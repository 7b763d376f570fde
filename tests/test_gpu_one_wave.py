"""Lattices whose tiles are resident at once, around the number of tiles where the launch of the step's
tail changes (152 SMs: 380, 400 and 560 cells a side have 144, 169 and 324 tiles): populations after 60
steps against the FP64 oracle (the bar of the other parity tests), and the same bits from eight-row
units, whose tail is launched as the smaller lattices' is."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc_x", [W.BC_PERIODIC, W.BC_INLET_OUTLET])
@pytest.mark.parametrize("n", [380, 400, 560])
def test_step_tail_launch(orc, n, bc_x):
    w = W.Workload(name="wave", nx=n, ny=n, tau=0.6, bc_x=bc_x, bc_y=W.BC_WALL, u_in=(0.02, 0.0), u0=(0.02, 0.01), dem_on=0,
                   x=np.array([[n / 2 + 0.3, n / 2 - 4.2]]), v=np.zeros((1, 2)), omega=np.zeros(1), r=np.array([10.0]))
    o = orc.Sim(w)
    o.step(60)
    f = []
    for units in (1, 2):
        g = imb.Lattice.from_workload(w, work_units=units)
        g.step(60)
        f.append(g.populations())
        g.close()
    assert np.abs(f[0] - o.f()).max() < 1e-6
    assert np.array_equal(f[0], f[1])
