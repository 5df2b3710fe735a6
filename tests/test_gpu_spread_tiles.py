"""The FP32 spread of 4-cell tiles (patch in registers) against the oracle, at
the edges of its staging batches and ranking, for every order.

Each mesh value is an FP32 sum of m products q Wx Wy Wz, so it is held to
(m + 8) 2^-24 of the sum of the terms' magnitudes (one rounding a term and
sum, a few for the weights), computed with the oracle's spread of |q|.
"""
import numpy as np
import pytest
import torch

from oracle.pppm import spread

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("mesh", [(16, 20, 24), (18, 15, 25)])  # whole tiles, ragged last tiles
@pytest.mark.parametrize("crowd", [1, 31, 32, 33, 65, 256, 257])  # sites in one tile: batch and ranking edges
def test_register_patch(cuda_device, pppm_lib, order, mesh, crowd):
    from paper_2504_15508_gb300.pppm import Plan
    box = np.array([8.0, 9.0, 10.0])
    rng = np.random.default_rng(100 * order + crowd)
    h = box / np.asarray(mesh)
    # one crowded tile, and sites anywhere (some outside the box, some tiles empty)
    pos = np.concatenate([(4.0 + 4.0 * rng.random((crowd, 3))) * h - 0.5 * h, (3.0 * rng.random((40, 3)) - 1.0) * box])
    q = rng.normal(size=pos.shape[0])
    tp = torch.tensor(pos, dtype=torch.float32, device=cuda_device).double()
    tq = torch.tensor(q, dtype=torch.float32, device=cuda_device).double()
    plan = Plan(box, mesh, order, 0.5, tile=4)
    rho = plan.spread(tp, tq)
    again = plan.spread(tp, tq)
    assert torch.equal(rho, again)
    p, qr = tp.cpu().numpy(), tq.cpu().numpy()
    ref = spread(p, qr, box, mesh, order)
    mag = spread(p, np.abs(qr), box, mesh, order)
    # the B-spline argument itself is rounded to 2^-24: the weights move by up to
    # order 2^-24 of their largest value, felt where a point's own terms are small
    bound = (pos.shape[0] + 8) * 2.0 ** -24 * mag + 8 * order * 2.0 ** -24 * np.abs(qr).max() / np.prod(h) * (mag > 0)
    err = np.abs(rho.double().cpu().numpy() - ref)
    assert np.all(err <= bound + 1e-30), float(np.max(err - bound))
