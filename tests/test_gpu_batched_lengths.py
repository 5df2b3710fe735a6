"""The staged batch's FFT stages: every line length with an engine, on every
axis, with few and many lines an item, against the oracle; and a batch with a
longer line, which takes the general stages.

Bars of the other batched tests: forces 1e-5, energies 1e-6 (relative), virial 1e-5.
"""
import numpy as np
import pytest
import torch

from oracle.pppm import OraclePPPM

pytestmark = pytest.mark.gpu

# every length from 8 to 64 on each axis, three a box; then a line above 64; and
# the shortest length, which only order 3 admits
LENGTHS = [8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64]
BOXES = {"small": [(LENGTHS[i], LENGTHS[(i + 1) % 7], LENGTHS[(i + 3) % 7]) for i in range(7)],
         "medium": [(LENGTHS[7 + i], LENGTHS[7 + (i + 1) % 7], LENGTHS[7 + (i + 3) % 7]) for i in range(7)],
         "large": [(LENGTHS[14 + i], 20, 18) for i in range(7)] + [(18, LENGTHS[14 + i], 27) for i in range(7)]
         + [(16, 25, LENGTHS[14 + i]) for i in range(7)],
         "long": [(20, 72, 16), (80, 16, 18), (18, 20, 96)],
         "six": [(6, 8, 9), (8, 6, 10), (9, 8, 6), (6, 6, 6)]}
# order 7 on ragged and whole meshes: with tile edge 4 an index has two to four covers
RAGGED = [(20, 18, 15), (12, 27, 25), (16, 20, 30), (45, 18, 50), (15, 50, 54), (24, 16, 64)]


@pytest.mark.parametrize("tile", [0, 4])
def test_staged_order_7(cuda_device, pppm_lib, tile):
    _check_staged(cuda_device, RAGGED, 7, tile)


@pytest.mark.parametrize("name,order", [(k, p) for k in BOXES for p in (3, 5) if k != "six" or p == 3])
def test_staged_lengths(cuda_device, pppm_lib, name, order):
    _check_staged(cuda_device, BOXES[name], order, 0)


def _check_staged(cuda_device, meshes, order, tile):
    from paper_2504_15508_gb300.pppm import BatchPlan
    boxes = [[0.9 * m for m in mesh] for mesh in meshes]
    rng = np.random.default_rng(len(meshes) + order)
    n = [int(150 + 40 * b) for b in range(len(meshes))]
    pos = [rng.random((k, 3)) * np.asarray(L) for k, L in zip(n, boxes)]
    q = [rng.normal(size=k) for k in n]
    off = np.concatenate([[0], np.cumsum(n)])
    tp = torch.tensor(np.concatenate(pos), dtype=torch.float32, device=cuda_device)
    tq = torch.tensor(np.concatenate(q), dtype=torch.float32, device=cuda_device)
    plan = BatchPlan(boxes, meshes, order, 0.5, tile=tile)
    plan.set_launch("staged")
    e, f, v = plan.compute(tp, tq, torch.tensor(off, dtype=torch.int64, device=cuda_device))
    torch.cuda.synchronize()
    assert plan.status() == 0
    p64, q64 = tp.double().cpu().numpy(), tq.double().cpu().numpy()
    for b, (L, mesh) in enumerate(zip(boxes, meshes)):
        s = slice(off[b], off[b + 1])
        ref = OraclePPPM(L, mesh, order, 0.5).compute(p64[s], q64[s])
        fb = f[s].double().cpu().numpy()
        assert np.linalg.norm(fb - ref["forces"]) <= 1e-5 * np.linalg.norm(ref["forces"]), (b, mesh)
        assert abs(e[b].item() - ref["energy"]) <= 1e-6 * abs(ref["energy"]), (b, mesh)
        assert np.linalg.norm(v[b].cpu().numpy() - ref["virial"]) <= 1e-5 * np.linalg.norm(ref["virial"]), (b, mesh)
