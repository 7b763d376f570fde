"""Islands of more than 32 particles, bit for bit against the sequential FP64 evaluation: one above
a warp, sets that fill the cluster's blocks unevenly, both contact laws, walls and a periodic edge
inside the island, two large islands at once, a set whose contacts overflow a block of the cluster
and one larger than the cluster (stepped by the whole grid)."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def slab(cols, rows, R, seed, periodic, gapcol=None, n=None, **kw):
    """cols x rows disks on a grid a hundredth of a cell apart, jittered into contact, moving."""
    g = np.random.default_rng(seed)
    s = 2 * R + 0.01
    i = np.arange(cols * rows)
    x = np.stack([(i % cols + 0.5) * s, (i // cols + 0.5) * s], 1)
    x += g.uniform(-0.006, 0.006, x.shape) + 0.02
    if gapcol is not None:   # a gap that splits the slab in two islands
        x[i % cols >= gapcol, 0] += 3.0
    x = x[:n] if n else x
    nx = cols * s if periodic else cols * s + R + 4
    v = 0.03 * g.standard_normal(x.shape).clip(-2, 2)
    m = len(x)
    return W.Workload(name="slab", nx=max(92, int(round(nx))), ny=max(92, int(rows * s + 8)), tau=0.6,
                      bc_x=W.BC_PERIODIC if periodic else W.BC_WALL, bc_y=W.BC_WALL, dem_on=1, N_sub=60,
                      gravity=(0.0, -1e-4), e_rest=0.7, mu=0.3, x=x, v=v, omega=0.01 * g.standard_normal(m),
                      r=R * (1 + 0.0005 * g.uniform(-1, 1, m)), **kw)


CASES = {
    "one more than a warp": (slab(11, 3, 5.0, 1, False), 1.0),
    "uneven blocks": (slab(17, 13, 5.0, 2, False, n=219), 1.0),
    "hertz-mindlin": (slab(17, 9, 5.0, 3, False, contact_model=1, E_young=2.0e4, nu_poisson=0.3), 1.0),
    "periodic": (slab(25, 8, 4.995, 4, True), 1.0),
    "two islands": (slab(20, 12, 5.0, 5, False, gapcol=8), 1.0),
    "many": (slab(50, 40, 4.2, 6, False), 1.0),
    "contacts overflow a block": (slab(60, 60, 4.2, 7, False), 8.5),   # twelve candidates a disk
    "beyond the cluster": (slab(66, 66, 4.2, 8, False), 1.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_large_islands_bit_exact(name):
    w, skin = CASES[name]
    g, o = imb.Lattice.from_workload(w, skin=skin), O.Sim(w)
    rng = np.random.default_rng(9)
    F, T = 1e-2 * rng.standard_normal((w.n_particles, 2)), 1e-2 * rng.standard_normal(w.n_particles)
    g.set_forces(F, T)
    o.set_forces(F, T)
    for _ in range(3):   # the springs carry over from cycle to cycle
        o.dem_substeps(w.N_sub)
        g.dem_step(1)
        for a, b in zip(o.particles(), g.particles()):
            assert np.array_equal(a, b)
    assert np.array_equal(o.contacts(), g.contacts())
    g.close()
