"""The features from the tiles' boxes in shared memory, and the training gradient
in tiles of 32 rows, at the edges of both, against the oracle.

Features are BF16: a potential sample may differ by one BF16 step, or by the
FP32 error of the mesh potential near zero (1e-5 of the largest sample), as in
the other feature tests; the types and paddings are exact.  Gradients are FP32
sums over the rows: 1e-4 of the gradient's norm, as in the other gradient tests.
"""
import numpy as np
import pytest
import torch

from oracle import mlp
from oracle.pppm import OraclePPPM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [4, 8, 16])  # the two boxes, and reading the mesh in place
@pytest.mark.parametrize("order", [3, 4, 5, 6, 7])
@pytest.mark.parametrize("mesh", [(16, 24, 32), (18, 25, 27)])  # whole and ragged last tiles
def test_features(cuda_device, pppm_lib, tile, order, mesh):
    from paper_2504_15508_gb300.pppm import Corrector, Plan
    from workloads.water import init_mlp_params
    box = np.asarray(mesh) * 1.7
    rng = np.random.default_rng(10 * order + tile)
    # one tile with more sites than threads, the others sparse or empty
    pos = np.concatenate([rng.random((200, 3)) * 3.5 * 1.7, (3 * rng.random((150, 3)) - 1) * box])
    q, types = rng.normal(size=350), rng.integers(0, 3, size=350)
    tp = torch.tensor(pos, dtype=torch.float32, device=cuda_device)
    tq = torch.tensor(q, dtype=torch.float32, device=cuda_device)
    tt = torch.tensor(types, dtype=torch.int8, device=cuda_device)
    plan = Plan(box, mesh, order, 0.4, tile=tile)
    corr = Corrector(plan, init_mlp_params(1, 48), 0.5, 1.0)
    feat, _ = corr.features(tp, tq, tt)
    got = feat.float().cpu().numpy().astype(np.float64)
    p64, q64 = tp.double().cpu().numpy(), tq.double().cpu().numpy()
    phi = OraclePPPM(box, mesh, order, 0.4).compute(p64, q64, want_intermediates=True)["phi"]
    X = mlp.features(phi, p64, types, box, mesh, order, s_in=0.5)
    ref = mlp.bf16_round(X.astype(np.float32))
    step = 2.0 ** (np.floor(np.log2(np.maximum(np.maximum(np.abs(got), np.abs(ref)), 1e-30))) - 7)
    d = np.abs(got - ref)
    assert np.all(d[:, :27] <= step[:, :27] + 1e-5 * np.abs(ref[:, :27]).max())
    assert np.array_equal(got[:, 27:30], X[:, 27:30]) and not got[:, 36:].any()
    assert np.all(d[:, 30:36] <= step[:, 30:36] + 2e-6)


@pytest.mark.parametrize("kind", ["cell", "stated"])
@pytest.mark.parametrize("nb", [1, 31, 32, 33, 9727, 9728, 9729, 20011])  # 304 resident blocks of 32 rows: 9,728
def test_gradient(cuda_device, pppm_lib, kind, nb):
    from paper_2504_15508_gb300.pppm import Corrector, Plan
    from workloads.water import init_mlp_params
    n_in = mlp.FEATURE_WIDTH[kind]
    rng = np.random.default_rng(nb)
    feat = torch.tensor(rng.normal(size=(5000, n_in)), dtype=torch.float32, device=cuda_device).to(torch.bfloat16)
    target = torch.tensor(rng.normal(size=(5000, 3)), dtype=torch.float32, device=cuda_device)
    idx = rng.integers(0, 5000, size=nb)
    idx[0] = 4999
    theta = init_mlp_params(3, n_in)
    corr = Corrector(Plan((16.0,) * 3, (16,) * 3, 5, 0.4), theta, 1.0, 1.0, features=kind)
    t_idx = torch.tensor(idx, dtype=torch.int32, device=cuda_device)
    loss, g = corr.grad(feat, target, t_idx)
    loss2, g2 = corr.grad(feat, target, t_idx)
    assert torch.equal(loss, loss2) and torch.equal(g, g2)
    # a table that starts between two 4-byte words
    odd = torch.empty(feat.numel() + 1, dtype=torch.bfloat16, device=cuda_device)[1:].view_as(feat).copy_(feat)
    loss3, g3 = corr.grad(odd, target, t_idx)
    assert torch.equal(loss, loss3) and torch.equal(g, g3)
    x = feat.float().cpu().numpy().astype(np.float64)[idx]
    ref_l, ref_g = mlp.loss_and_grad(theta, x, target.cpu().numpy().astype(np.float64)[idx])
    assert abs(loss.item() - ref_l) <= 1e-5 * abs(ref_l)
    assert np.linalg.norm(g.cpu().numpy() - ref_g) <= 1e-4 * np.linalg.norm(ref_g)
