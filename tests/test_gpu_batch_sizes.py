"""Batched sweep on widths around the edges of its layout and work items: rows of one cell more and
less than a 128-byte block of a plane (32 or 64 cells) and than a warp's 32 or 64 cells, odd rows,
whose last cell is alone in its pair, and rows much shorter than a warp.  Populations against the
FP64 oracle on each domain by itself, with the bars of the sweep's own tests (FP32 1e-6, 16 bits the
rounding of the stored f - w: 2e-4, eight times that for bfloat16's three bits less).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(3, 7), (5, 3), (11, 19), (31, 24), (32, 25), (33, 24), (63, 31), (64, 32), (65, 33), (66, 24), (97, 29), (127, 24),
         (128, 23), (129, 25)]
STEPS = 40


@pytest.fixture(scope="module")
def imb():
    import paper_1809_07008_gb300 as imb
    imb.load()
    return imb


def _domain(k, nx, ny):
    if min(nx, ny) >= 19:   # a disk and its images fit
        return W.c5_domain(k, nx, ny, 8.0, 0.15, 0.6, 3.0, 40 + k)
    w = W.c5_domain(k, 64, 48, 12.0, 0.2, 0.7, 1.0, 31)
    return w.with_(nx=nx, ny=ny, x=np.zeros((0, 2)), v=np.zeros((0, 2)), omega=np.zeros(0), r=np.zeros(0))


@pytest.fixture(scope="module")
def reference(orc):
    ds, fs = [_domain(k, *s) for k, s in enumerate(SIZES)], []
    for w in ds:
        o = orc.Sim(w)
        o.step(STEPS)
        fs.append(o.f())
    return ds, fs


@pytest.mark.parametrize("cells", [1, 2])
@pytest.mark.parametrize("storage,bar", [("fp32", 1e-6), ("fp16", 2e-4), ("bf16", 1.6e-3)])
def test_widths_match_oracle(imb, reference, storage, bar, cells):
    ds, fs = reference
    b = imb.Batch(ds, storage=storage)
    b.set_launch(256, cells)
    b.run(STEPS)
    for k, f in enumerate(fs):
        assert np.abs(b.populations(k) - f).max() < bar, SIZES[k]
    b.close()
