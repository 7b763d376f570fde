"""d J / d u_in of the drag gradient, which the transposed inlet column of the reverse step gives,
against the oracle's reverse mode, with the other components beside it: lattices where one thread takes
both the column behind the inlet and the one before the outlet (nx = 3) or two neighbours do
(nx = 4), widths around a block of columns, and one where every multiple of 32 up to 256 leaves
one column (nx = 26881).

The bars are the gradient's own (1e-5 on J, 2e-3 of the largest component on the gradients): the
adjoint is FP32, 60 steps of some ten roundings each leave 4e-5 of its scale at most, and the sums
over the inlet rows cancel by less than a factor of ten with the disks this close to the inlet."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def channel(nx, ny, x, r):
    n = len(r)
    return W.Workload(name="adj_inlet", nx=nx, ny=ny, tau=0.6, bc_x=W.BC_INLET_OUTLET, bc_y=W.BC_WALL, u_in=(0.02, 0.0),
                      x=np.array(x), v=np.zeros((n, 2)), omega=np.zeros(n), r=np.array(r), dem_on=0)


def two_disks(nx):
    return channel(nx, 32, [[9.3, 15.7], [nx - 9.4, 17.2]], [5.23, 4.37])


CASES = {
    "3": channel(3, 24, [[1.6, 11.3]], [0.9]),
    "4": channel(4, 24, [[1.9, 11.3]], [1.1]),
    "52": two_disks(52),
    "255": two_disks(255),
    "256": two_disks(256),
    "257": two_disks(257),
    "258": two_disks(258),
    "513": two_disks(513),
    "26881": channel(26881, 16, [[9.3, 7.7], [26871.6, 8.2]], [4.23, 3.37]),
}


@pytest.mark.parametrize("width", list(CASES))
def test_inlet_gradient_matches_oracle(orc, width):
    import paper_1809_07008_gb300 as imb
    w = CASES[width]
    o = orc.Sim(w)
    o.step(20)
    Jo, guo, gto, gxo = o.drag_adjoint(60)
    for scheme in (dict(checkpoint_every=16), dict(snapshots=5)):
        g = imb.Lattice.from_workload(w)
        g.step(20)
        Jg, gug, gtg, gxg = g.drag_gradient(60, **scheme)
        g.close()
        assert abs(Jg - Jo) <= 1e-5 * abs(Jo)
        assert abs(gug - guo) <= 2e-3 * abs(guo)
        assert abs(gtg - gto) <= 2e-3 * abs(gto)
        assert np.abs(gxg - gxo).max() <= 2e-3 * np.abs(gxo).max()
