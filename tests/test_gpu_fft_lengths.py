"""Every line length with a register engine, on every axis, and lengths beside
them that take the run-time engine, against numpy's FP64 transforms; and the
whole path on meshes that mix them.

The real transform of a mesh of N points is a product of one line transform
per axis, each with a relative error of a few roundings a radix stage: 2e-6
(FP32) and 1e-13 (FP64) of the result's norm, as for the other FFT tests.
"""
import numpy as np
import pytest
import torch

from oracle.pppm import OraclePPPM

pytestmark = pytest.mark.gpu

LENGTHS = [8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96,
           100, 108, 120, 125, 128, 135, 144, 150, 160, 162, 180, 192, 200, 216, 225, 240, 250, 256]
BESIDE = [5, 6, 243, 270]  # no engine: too short, no factors, too long
DT = {"fp32": torch.float32, "fp64": torch.float64}
TOL = {"fp32": 2e-6, "fp64": 1e-13}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("length", LENGTHS + BESIDE)
def test_lengths(cuda_device, pppm_lib, prec, axis, length):
    from paper_2504_15508_gb300.pppm import Plan
    # neighbours of odd and even size; 15 x 17 lines leave partly filled blocks
    mesh = [15, 9, 20]
    mesh[axis] = length
    plan = Plan((10.0, 11.0, 12.0), mesh, 5, 0.4, precision=prec)
    x = np.random.default_rng(length + axis).normal(size=mesh)
    xt = torch.tensor(x, dtype=DT[prec], device=cuda_device)
    X = plan.fft_r2c(xt)
    ref = np.fft.rfftn(xt.double().cpu().numpy())
    assert np.linalg.norm(X.cpu().numpy() - ref) <= TOL[prec] * np.linalg.norm(ref)
    y = plan.fft_c2r(X).double().cpu().numpy() / np.prod(mesh)
    x = xt.double().cpu().numpy()
    assert np.linalg.norm(y - x) <= TOL[prec] * np.linalg.norm(x)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("mesh,order,tile", [
    ((27, 25, 45), 5, 0), ((20, 18, 15), 4, 4), ((36, 50, 54), 7, 4),  # odd and even, two to four fold covers
    ((75, 16, 81), 6, 0), ((12, 60, 27), 3, 0), ((8, 9, 10), 5, 0),    # no room for whole tiles: the fold kernel
    ((270, 16, 20), 5, 0), ((16, 270, 20), 5, 0), ((20, 16, 270), 5, 0),  # one run-time axis beside two engines
    ((16, 18, 243), 5, 8), ((18, 15, 405), 7, 8), ((12, 18, 243), 4, 4),  # run-time z, ragged: three covers
    ((16, 25, 225), 7, 8), ((20, 16, 150), 6, 8), ((16, 16, 162), 4, 8)])  # the same where FP64 has no engine
def test_whole_path(cuda_device, pppm_lib, prec, mesh, order, tile):
    from paper_2504_15508_gb300.pppm import Plan
    box = np.asarray(mesh) * 0.9
    rng = np.random.default_rng(sum(mesh))
    pos, q = rng.random((700, 3)) * box, rng.normal(size=700)
    tp = torch.tensor(pos, dtype=DT[prec], device=cuda_device)
    tq = torch.tensor(q - q.mean(), dtype=DT[prec], device=cuda_device)
    plan = Plan(box, mesh, order, 0.5, precision=prec, tile=tile)
    e, f, v = plan.compute(tp, tq)
    ref = OraclePPPM(box, mesh, order, 0.5).compute(tp.double().cpu().numpy(), tq.double().cpu().numpy())
    # the bars of the other parity tests
    ftol, etol = {"fp32": (1e-5, 1e-6), "fp64": (1e-12, 1e-12)}[prec]
    assert np.linalg.norm(f.double().cpu().numpy() - ref["forces"]) <= ftol * np.linalg.norm(ref["forces"])
    assert abs(e.item() - ref["energy"]) <= etol * abs(ref["energy"])
    assert np.linalg.norm(v.cpu().numpy() - ref["virial"]) <= ftol * np.linalg.norm(ref["virial"])
