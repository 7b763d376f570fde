"""Batched sweep of narrow domains, whose populations lie in whole planes without padding: populations
and drag against the FP64 oracle on each domain by itself (the bars of the sweep's own tests), and the
memory the batch takes."""
import numpy as np
import pytest
import torch

import paper_1809_07008_gb300 as imb
import workloads as W

pytestmark = pytest.mark.gpu

BARS = {"fp32": 1e-6, "fp16": 2e-4, "bf16": 1.6e-3}   # FP32, and the rounding of the stored f - w


def empty(k, nx, ny):
    w = W.c5_domain(k, 64, 48, 12.0, 0.2, 0.7, 1.0, 31)
    return w.with_(nx=nx, ny=ny, x=np.zeros((0, 2)), v=np.zeros((0, 2)), omega=np.zeros(0), r=np.zeros(0))


# mean width below 8 in a batch of a few cells: rows of three to seven cells, a disk in a narrow domain,
# a wide domain with disks among them
SMALL = [empty(0, 3, 7), empty(1, 4, 201), W.c5_domain(2, 41, 24, 8.0, 0.15, 0.6, 3.0, 42), empty(3, 5, 97), empty(4, 7, 33),
         empty(5, 3, 400), W.c5_domain(6, 19, 21, 8.0, 0.15, 0.6, 3.0, 46), empty(7, 6, 64)]
# below 100 in a large one (86 MB of FP32): the same three domains over and over, the last one odd
LARGE = [W.c5_domain(k % 3, 50 + k % 3, 60, 10.0, 0.2, 0.65, 2.0, 50 + k % 3) for k in range(398)] + [empty(9, 37, 41)]


def run(orc, ds, look, storage, cells, steps):
    b = imb.Batch(ds, storage=storage)
    b.set_launch(256, cells)
    b.run(steps)
    F = np.stack(b.mean_drag(), -1)
    for k in look:
        o = orc.Sim(ds[k])
        drag = np.zeros(2)
        for _ in range(steps):
            o.step(1)
            if ds[k].n_particles:
                drag += o.forces()[0].sum(0) / steps
        assert np.abs(b.populations(k) - o.f()).max() < BARS[storage], k
        if storage == "fp32":
            assert np.abs(F[k] - drag).max() <= 1e-4 * max(np.abs(drag).max(), 1e-12), k
    b.close()


@pytest.mark.parametrize("cells", [1, 2])
@pytest.mark.parametrize("storage", list(BARS))
def test_small_batch_of_narrow_domains(orc, storage, cells):
    run(orc, SMALL, range(len(SMALL)), storage, cells, 40)


def test_large_batch_of_narrow_domains(orc):
    run(orc, LARGE, [0, 1, 200, 395, 397, 398], "fp32", 2, 30)


@pytest.mark.parametrize("storage,elem", [("fp32", 4), ("fp16", 2)])
def test_narrow_domains_take_no_padding(storage, elem):
    ds = [empty(k, 3, 2000) for k in range(1000)]
    need = sum(w.nx * w.ny for w in ds) * (18 * elem + 4)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    b = imb.Batch(ds, storage=storage)
    used = before - torch.cuda.mem_get_info()[0]
    b.run(2)
    b.close()
    assert used <= 1.1 * need + 16e6, (used, need)
