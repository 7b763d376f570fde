"""Large islands in cycles of few sub-cycles, below and above the number of particles that the cluster
takes then (the others are stepped by the whole grid): bit for bit against the sequential FP64
evaluation."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def slab(cols, rows, N_sub):
    g = np.random.default_rng(cols + N_sub)
    R, s, i = 4.2, 8.41, np.arange(cols * rows)
    x = np.stack([(i % cols + 0.5) * s, (i // cols + 0.5) * s], 1) + g.uniform(-0.006, 0.006, (len(i), 2)) + 0.02
    return W.Workload(name="slab", nx=max(92, int(cols * s + R + 4)), ny=max(92, int(rows * s + 8)), tau=0.6, bc_x=W.BC_WALL,
                      bc_y=W.BC_WALL, dem_on=1, N_sub=N_sub, kn=5.0, kt=2.5, gravity=(0.0, -1e-4), e_rest=0.7, mu=0.3, x=x,
                      v=0.02 * g.standard_normal(x.shape).clip(-2, 2), omega=0.01 * g.standard_normal(len(i)),
                      r=R * (1 + 0.0005 * g.uniform(-1, 1, len(i))))


@pytest.mark.parametrize("N_sub", [1, 2, 11, 12])
@pytest.mark.parametrize("cols,rows", [(40, 24), (40, 26), (64, 62)])   # 960, 1040 and 3968 disks
def test_few_subcycles(cols, rows, N_sub):
    w = slab(cols, rows, N_sub)
    g, o = imb.Lattice.from_workload(w), O.Sim(w)
    for _ in range(4):
        o.dem_substeps(w.N_sub)
        g.dem_step(1)
        for a, b in zip(o.particles(), g.particles()):
            assert np.array_equal(a, b)
    assert len(o.contacts()) > 0 and np.array_equal(o.contacts(), g.contacts())
    g.close()
