"""A particle that meets a wall it was further than the skin from at the start of the cycle, and is
back near its place at the end of it, in a small island, a warp's island and one of the cluster, at each
of the four walls: bit for bit against the sequential FP64 evaluation (which tests every wall in
every sub-cycle)."""
import numpy as np
import pytest

import paper_1809_07008_gb300 as imb
import workloads as W
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def row(n, wall, gap=1.2, speed=3.0, R=5.0):
    """n disks in a row along a wall, 0.4 apart (one island), `gap` from it; one flies at it."""
    axis, high = wall // 2, wall % 2
    x = np.full((n, 2), 90.0)
    x[:, 1 - axis] = 60 + np.arange(n) * (2 * R + 0.4)
    size = [130, 130]
    size[1 - axis] = int(x[:, 1 - axis].max() + 60)
    x[:, axis] = size[axis] - R - gap if high else R + gap
    v = np.zeros((n, 2))
    v[n // 2, axis] = speed if high else -speed
    return W.Workload(name="bounce", nx=size[0], ny=size[1], tau=0.6, bc_x=W.BC_WALL, bc_y=W.BC_WALL, dem_on=1, N_sub=400,
                      gravity=(0.0, 0.0), e_rest=1.0, mu=0.3, x=x, v=v, omega=1e-3 * np.arange(n), r=np.full(n, R))


@pytest.mark.parametrize("wall", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [2, 5, 20, 45])
def test_bounce_within_a_cycle(n, wall):
    w = row(n, wall)
    g, o = imb.Lattice.from_workload(w), O.Sim(w)
    o.dem_substeps(w.N_sub)
    x, v, _ = o.particles()
    assert abs(x - w.x).max() < 0.5 and (v * w.v).sum() < 0   # the cycle that reports no IMB_E_SKIN, turned round
    g.dem_step(1)
    for a, b in zip(o.particles(), g.particles()):
        assert np.array_equal(a, b)
    g.close()
