"""Islands of 2 to 32 particles, whose lanes hand their particles' state to each other in every
sub-cycle, bit for bit against the sequential FP64 evaluation: two lanes, the largest island that
shares a warp, one more, a whole warp, walls beside the island, several islands to a warp, and an
island of more pairs than are evaluated a lane each (stepped particle by particle).  Two islands above
a warp, whose contacts two lanes share, stand beside them."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def block(n, cols, R, gap, seed, repeat=1, at=(40.0, 40.0), **kw):
    """`repeat` islands of n disks, rows of `cols`, a gap of `gap` jittered into contact, moving."""
    g = np.random.default_rng(seed)
    s = 2 * R + gap
    i = np.arange(n)
    one = np.stack([(i % cols) * s, (i // cols) * s], 1) + at
    x = np.concatenate([one + (k * (cols * s + 2 * R + 6), 0.0) for k in range(repeat)])
    x = x + g.uniform(-0.7, 0.7, x.shape) * gap
    m = len(x)
    size = x.max(0) + R + 40
    return W.Workload(name="block", nx=max(160, int(size[0])), ny=max(160, int(size[1])), tau=0.6, bc_x=W.BC_WALL,
                      bc_y=W.BC_WALL, dem_on=1, N_sub=75, gravity=(0.0, -1e-4), e_rest=0.8, mu=0.3, x=x,
                      v=0.04 * g.standard_normal(x.shape).clip(-2, 2), omega=0.01 * g.standard_normal(m),
                      r=R * (1 + 0.0005 * g.uniform(-1, 1, m)), **kw)


CASES = {
    "two": (block(2, 2, 5.0, 0.02, 1), 1.0),
    "four": (block(4, 2, 5.0, 0.02, 2), 1.0),
    "nine of four": (block(4, 2, 5.0, 0.02, 3, repeat=9), 1.0),
    "five": (block(5, 3, 5.0, 0.02, 4), 1.0),
    "chain of 31": (block(31, 31, 5.0, 0.02, 5), 1.0),
    "warp": (block(32, 8, 5.0, 0.02, 6), 1.0),
    "warp at a wall": (block(32, 8, 5.0, 0.02, 7, at=(5.01, 5.01)), 1.0),
    "hertz-mindlin": (block(32, 8, 5.0, 0.02, 8, contact_model=1, E_young=2.0e4, nu_poisson=0.3), 1.0),
    "particle by particle": (block(32, 8, 3.0, 0.05, 9), 6.5),   # twelve candidates a disk inside, over 96 pairs
    # above a warp, two lanes a contact that share its spring (the last lanes of the list idle)
    "cluster at a wall": (block(45, 9, 5.0, 0.02, 10, at=(5.01, 5.01)), 1.0),
    "cluster, hertz-mindlin at a wall": (block(45, 9, 5.0, 0.02, 11, at=(5.01, 5.01), contact_model=1, E_young=2.0e4,
                                               nu_poisson=0.3), 1.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_islands_bit_exact(name):
    w, skin = CASES[name]
    g, o = imb.Lattice.from_workload(w, skin=skin), O.Sim(w)
    rng = np.random.default_rng(9)
    F, T = 1e-2 * rng.standard_normal((w.n_particles, 2)), 1e-2 * rng.standard_normal(w.n_particles)
    g.set_forces(F, T)
    o.set_forces(F, T)
    for _ in range(6):   # contacts open and close, the springs carry over from cycle to cycle
        o.dem_substeps(w.N_sub)
        g.dem_step(1)
        for a, b in zip(o.particles(), g.particles()):
            assert np.array_equal(a, b)
    assert np.array_equal(o.contacts(), g.contacts())
    g.close()
