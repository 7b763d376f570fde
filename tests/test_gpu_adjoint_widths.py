"""Drag gradient on widths where the last column would start a block of its own (nx = 1 modulo the
block), with disks close to the inlet and the outlet so that the transposed columns carry the
gradient: J, d J / d tau and d J / d (disk centres) against the oracle's reverse mode, with the bars of
the gradient's own tests (1e-5 on J, 2e-3 of the largest component on the gradients)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [255, 257, 289, 513])
def test_gradient_matches_oracle_at_block_edges(orc, nx):
    import paper_1809_07008_gb300 as imb
    w = W.Workload(name="adj_width", nx=nx, ny=32, tau=0.6, bc_x=W.BC_INLET_OUTLET, bc_y=W.BC_WALL, u_in=(0.02, 0.0),
                   x=np.array([[9.3, 15.7], [nx - 9.4, 17.2]]), v=np.zeros((2, 2)), omega=np.zeros(2), r=np.array([5.23, 4.37]),
                   dem_on=0)
    o, g = orc.Sim(w), imb.Lattice.from_workload(w)
    o.step(20)
    g.step(20)
    Jo, _, gto, gxo = o.drag_adjoint(60)
    Jg, _, gtg, gxg = g.drag_gradient(60, checkpoint_every=16)
    assert abs(Jg - Jo) <= 1e-5 * abs(Jo)
    assert abs(gtg - gto) <= 2e-3 * abs(gto)
    assert np.abs(gxg - gxo).max() <= 2e-3 * np.abs(gxo).max()
