"""Sites sorted by one block (up to 256 sites, 4,096 tiles) and by more, on
both sides of each line, against the oracle's spread; crowded tiles overflow
their regions (128 sites at tile 4, 256 at tile 8), and a captured step is replayed
with other sites.

The FP32 spread is held to the bound of the register-patch test: m + 8
roundings of the terms' magnitudes, and the weights' own rounding.
"""
import numpy as np
import pytest
import torch

from oracle.pppm import spread

pytestmark = pytest.mark.gpu


def _sites(rng, n, box, crowd):
    pos = rng.random((n, 3)) * box * (0.03 if crowd else 3.0) - (0.0 if crowd else 1.0) * box
    return pos, rng.normal(size=n)


def _check_spread(plan, tp, tq, box, mesh, order):
    rho = plan.spread(tp, tq).double().cpu().numpy()
    p, q = tp.double().cpu().numpy(), tq.double().cpu().numpy()
    ref, mag = spread(p, q, box, mesh, order), spread(p, np.abs(q), box, mesh, order)
    eps, h = 2.0 ** -24, box / np.asarray(mesh)
    # the weights' rounding also at points without a term in the reference: an
    # argument that rounds onto a cell edge reaches one point beyond its support
    bound = (len(q) + 8) * eps * mag + 8 * order * eps * np.abs(q).max() / np.prod(h)
    assert np.all(np.abs(rho - ref) <= bound)


@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, 513])
@pytest.mark.parametrize("mesh,tile", [((16, 20, 24), 4), ((32, 30, 27), 8), ((64, 64, 64), 4), ((64, 64, 72), 4)])
@pytest.mark.parametrize("crowd", [False, True])
def test_small_sort(cuda_device, pppm_lib, n, mesh, tile, crowd):
    from paper_2504_15508_gb300.pppm import Plan
    rng = np.random.default_rng(n + mesh[2])
    box = np.array([16.0, 15.0, 18.0])
    plan = Plan(box, mesh, 5, 0.5, tile=tile)
    for _ in range(2):  # the second call finds the first one's tiles
        pos, q = _sites(rng, n, box, crowd)
        tp = torch.tensor(pos, dtype=torch.float32, device=cuda_device)
        tq = torch.tensor(q, dtype=torch.float32, device=cuda_device)
        _check_spread(plan, tp, tq, box, mesh, 5)
        assert plan.status() == 0


@pytest.mark.parametrize("n", [200, 256, 257])
def test_small_sort_replayed(cuda_device, pppm_lib, n):
    from paper_2504_15508_gb300.pppm import Plan
    rng = np.random.default_rng(n)
    box, mesh = np.array([16.0, 15.0, 18.0]), (16, 20, 24)
    plan = Plan(box, mesh, 5, 0.5, tile=4)
    a = [torch.tensor(v, dtype=torch.float32, device=cuda_device) for v in _sites(rng, n, box, False)]
    b = [torch.tensor(v, dtype=torch.float32, device=cuda_device) for v in _sites(rng, n, box, True)]
    graph = plan.graph(*a)
    for pos, q in (a, b, a, b):
        e, f, v = graph.launch(pos, q)
        graph.stream.synchronize()
        e2, f2, v2 = plan.compute(pos, q)
        # each tile's sites are spread in the order of their indices, however they arrived
        assert torch.equal(f, f2) and torch.equal(e, e2) and torch.equal(v, v2)
