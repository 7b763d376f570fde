"""The cluster's contact table: a set of large islands whose contacts fill most of it, and one that
overflows a block's (16 candidates a disk and both walls of a narrow box, 2596 contacts in a block of
256 disks), which the cluster then steps particle by particle: bit for bit against the sequential
FP64 evaluation."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def chain(n, skin, seed):
    """n disks in a row along a box 40 cells high, eight candidates on each side, close to contact."""
    g = np.random.default_rng(seed)
    R, s = 1.5, 3.1
    x = np.stack([40.0 + np.arange(n) * s, np.full(n, 20.0)], 1) + g.uniform(-0.047, 0.047, (n, 2))
    w = W.Workload(name="chain", nx=int(80 + n * s), ny=40, tau=0.6, bc_x=W.BC_WALL, bc_y=W.BC_WALL, dem_on=1, N_sub=60,
                   gravity=(0.0, -1e-4), e_rest=0.7, mu=0.3, x=x, v=0.03 * g.standard_normal(x.shape).clip(-2, 2),
                   omega=0.01 * g.standard_normal(n), r=R * (1 + 0.001 * g.uniform(-1, 1, n)))
    return w, skin


CASES = {"overflows a block": chain(4096, 23.4, 1), "fits": chain(3000, 23.4, 2)}


@pytest.mark.parametrize("name", list(CASES))
def test_table(name):
    w, skin = CASES[name]
    d = np.abs(w.x[1:200, None, 0] - w.x[None, 1:200, 0])
    near = ((d > 0) & (np.hypot(d, w.x[1:200, None, 1] - w.x[None, 1:200, 1]) < 3.0 + skin)).sum(1)[20:-20]
    assert near.min() == near.max() == 16 and w.x[:, 1].max() < 40 - w.x[:, 1].min() + 2 < 2 * (1.5 + skin)
    g, o = imb.Lattice.from_workload(w, skin=skin), O.Sim(w)
    rng = np.random.default_rng(9)
    F, T = 1e-2 * rng.standard_normal((w.n_particles, 2)), 1e-2 * rng.standard_normal(w.n_particles)
    g.set_forces(F, T)
    o.set_forces(F, T)
    for _ in range(3):
        o.dem_substeps(w.N_sub)
        g.dem_step(1)
        for a, b in zip(o.particles(), g.particles()):
            assert np.array_equal(a, b)
    assert np.array_equal(o.contacts(), g.contacts())
    g.close()
