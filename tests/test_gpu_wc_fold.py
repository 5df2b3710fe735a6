"""GPU parity of the WC force fold (Eq. DPLR:F_final) against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle.wc_fold import fold
from workloads.water import dw_jacobian, make_workload

pytestmark = pytest.mark.gpu


def _dev(a, dt):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _maps(hp, hw, jp, jw, J, dt):
    return (_dev(hp, torch.int32), _dev(hw, torch.int32), _dev(jp, torch.int64), _dev(jw, torch.int32),
            _dev(J, dt))


@pytest.mark.parametrize("name", ["water64", "water4096"])
@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-14), (torch.float32, 1e-6)])
def test_fold_matches_oracle(cuda_device, name, dt, tol):
    from paper_2504_15508_gb300.pppm import wc_fold
    wb, _ = make_workload(name)
    hp, hw, jp, jw, J = dw_jacobian(wb, seed=7)
    rng = np.random.default_rng(1)
    f_sites = rng.normal(size=(wb.n, 3))
    n_atoms = 3 * wb.n_mol
    fs = _dev(f_sites, dt)
    maps = _maps(hp, hw, jp, jw, J, dt)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = wc_fold(fs, n_atoms, *maps, status=status)
    torch.cuda.synchronize()
    ref = fold(fs.double().cpu().numpy(), n_atoms, hp, hw, jp, jw, maps[4].double().cpu().numpy())
    err = np.linalg.norm(out.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    print(f"wc_fold {name} {dt}: {err:.2e}")
    assert err <= tol and status.item() == 0
    again = wc_fold(fs, n_atoms, *maps)
    assert torch.equal(out, again)  # fixed summation order


def test_fold_of_pppm_forces_matches_oracle_chain(cuda_device):
    """End to end in FP64: GPU PPPM forces folded on the GPU vs oracle PPPM
    forces folded by the oracle."""
    from oracle.pppm import OraclePPPM
    from paper_2504_15508_gb300.pppm import Plan, wc_fold
    wb, w = make_workload("water64")
    plan = Plan(wb.box, w["mesh"], w["order"], w["beta"], precision="fp64")
    pos = _dev(wb.pos, torch.float64)
    q = _dev(wb.q, torch.float64)
    _, f, _ = plan.compute(pos, q)
    hp, hw, jp, jw, J = dw_jacobian(wb, seed=3)
    n_atoms = 3 * wb.n_mol
    out = wc_fold(f, n_atoms, *_maps(hp, hw, jp, jw, J, torch.float64))
    torch.cuda.synchronize()
    r = OraclePPPM(wb.box, w["mesh"], w["order"], w["beta"]).compute(wb.pos, wb.q)
    ref = fold(r["forces"], n_atoms, hp, hw, jp, jw, J)
    err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
    print(f"PPPM + fold vs oracle: {err:.2e}")
    assert err <= 1e-12


def test_fold_edge_cases(cuda_device):
    from paper_2504_15508_gb300.pppm import wc_fold
    rng = np.random.default_rng(2)
    f = _dev(rng.normal(size=(10, 3)), torch.float64)
    # no maps: the atoms' own forces
    assert torch.equal(wc_fold(f, 7), f[:7])
    # no WCs at all
    assert torch.equal(wc_fold(f, 10), f)
    # host map only, with empty rows
    hp = _dev([0, 1, 1, 1, 2, 2, 3, 3], torch.int32)
    hw = _dev([2, 0, 1], torch.int32)
    out = wc_fold(f, 7, hp, hw)
    ref = fold(f.cpu().numpy(), 7, hp.cpu().numpy(), hw.cpu().numpy())
    assert torch.allclose(out, torch.tensor(ref, device="cuda"), rtol=0, atol=1e-15)
    # an out-of-range WC index is skipped and flagged
    jp = _dev([0, 2, 2, 2, 2, 2, 2, 3], torch.int64)
    jw = _dev([1, 5, 0], torch.int32)
    J = _dev(rng.normal(size=(3, 3, 3)), torch.float64)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = wc_fold(f, 7, hp, hw, jp, jw, J, status=status)
    torch.cuda.synchronize()
    assert status.item() == 1
    keep = np.array([True, False, True])
    ref = fold(f.cpu().numpy(), 7, hp.cpu().numpy(), hw.cpu().numpy(), jp.cpu().numpy(),
               np.where(keep, jw.cpu().numpy(), 0), J.cpu().numpy() * keep[:, None, None])
    assert np.allclose(out.cpu().numpy(), ref, rtol=0, atol=1e-14)
    # zero atoms
    assert wc_fold(f[:0], 0).shape == (0, 3)


@pytest.mark.parametrize("dt,tol", [(torch.float64, 1e-14), (torch.float32, 1e-6)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])  # values before the Jacobian: 16-byte aligned and not
@pytest.mark.parametrize("lengths", [(0, 1, 5, 0), (31, 32, 33, 8), (127, 0, 1, 128), (300, 2, 65, 1000), (27,) * 9])
def test_fold_row_lengths(cuda_device, dt, tol, offset, lengths):
    """Rows at the edges of a group's pieces and of a row's rounds, empty groups
    between them, the last WC (whose row ends the array) included."""
    from paper_2504_15508_gb300.pppm import wc_fold
    rng = np.random.default_rng(sum(lengths) + offset)
    rows = list(lengths) + [0] * 9 + list(reversed(lengths)) + [3]
    n_atoms, n_wc = len(rows), 13
    jp = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    jw = rng.integers(0, n_wc, size=jp[-1]).astype(np.int32)
    jw[::7] = n_wc - 1
    J = rng.normal(size=(jp[-1], 3, 3))
    f = rng.normal(size=(n_atoms + n_wc, 3))
    flat = torch.empty(9 * jp[-1] + offset, dtype=dt, device="cuda")[offset:]
    tj = flat.view(-1, 3, 3).copy_(torch.tensor(J, dtype=dt))
    tf = torch.empty(3 * (n_atoms + n_wc) + offset, dtype=dt, device="cuda")[offset:].view(-1, 3)
    tf.copy_(torch.tensor(f, dtype=dt))
    out = wc_fold(tf, n_atoms, None, None, _dev(jp, torch.int64), _dev(jw, torch.int32), tj)
    assert torch.equal(out, wc_fold(tf, n_atoms, None, None, _dev(jp, torch.int64), _dev(jw, torch.int32), tj))
    ref = fold(tf.double().cpu().numpy(), n_atoms, None, None, jp, jw, tj.double().cpu().numpy())
    assert np.linalg.norm(out.double().cpu().numpy() - ref) <= tol * np.linalg.norm(ref)


def _torch_fold(f, n_atoms, hp, hw, jp, jw, J):
    """The fold in FP64 and the sum of its terms' magnitudes, by torch's index_add."""
    f, J, out, mag = f.double(), J.double(), f[:n_atoms].double(), f[:n_atoms].double().abs()
    fw = f[n_atoms:]
    rows = torch.arange(n_atoms, device="cuda")
    ok = (jw >= 0) & (jw < fw.shape[0])
    at = rows.repeat_interleave(jp[1:] - jp[:-1])[ok]
    g = fw[jw[ok].long()]
    out.index_add_(0, at, torch.einsum("kab,ka->kb", J[ok], g))
    mag.index_add_(0, at, torch.einsum("kab,ka->kb", J[ok].abs(), g.abs()))
    if hp is not None:
        at = rows.repeat_interleave((hp[1:] - hp[:-1]).long())
        out.index_add_(0, at, fw[hw.long()])
        mag.index_add_(0, at, fw[hw.long()].abs())
    return out, mag


def _check_fold(dt, rows, n_wc, hosts, bad, whole=False):
    """Rows of the given lengths; the error of a sum of m blocks of three products,
    up to two host terms and the atom's own is at most (m + 6) roundings of the
    terms' magnitudes (in FP64 twice, as the reference rounds as often), and
    (m / 32 + 14) in FP32, whose sums run over 32 lanes and then a butterfly.
    whole: blocks and forces of small whole numbers, whose sums are exact."""
    from paper_2504_15508_gb300.pppm import wc_fold
    g = torch.Generator(device="cuda").manual_seed(len(rows))
    rows = torch.as_tensor(rows, device="cuda")
    n_atoms, zero = len(rows), torch.zeros(1, dtype=torch.int64, device="cuda")
    jp = torch.cat([zero, rows.cumsum(0)])
    nnz = int(jp[-1])
    jw = torch.randint(0, n_wc, (nnz,), generator=g, device="cuda", dtype=torch.int32)
    J = torch.randn((nnz, 3, 3), generator=g, device="cuda", dtype=dt)
    f = torch.randn((n_atoms + n_wc, 3), generator=g, device="cuda", dtype=dt)
    if whole:
        J, f = J.round().clamp(-2, 2), f.round().clamp(-2, 2)
    hp = hw = None
    if hosts:
        per = torch.arange(n_atoms, device="cuda") % 3  # 0, 1 or 2 hosted centroids an atom
        hp = torch.cat([zero, per.cumsum(0)]).int()
        hw = torch.randint(0, n_wc, (int(hp[-1]),), generator=g, device="cuda", dtype=torch.int32)
    if bad:
        jw[nnz // 2], jw[-1] = n_wc, -1
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = wc_fold(f, n_atoms, hp, hw, jp, jw, J, status=status)
    assert status.item() == (1 if bad else 0)
    assert torch.equal(out, wc_fold(f, n_atoms, hp, hw, jp, jw, J))
    ref, mag = _torch_fold(f, n_atoms, hp, hw, jp, jw, J)
    if whole:
        assert torch.equal(out.double(), ref)
        return
    m = rows.double()[:, None]
    bound = ((m / 32).floor() + 14) * 2.0 ** -24 if dt == torch.float32 else (m + 6) * 2.0 ** -53 * 2
    assert bool(((out.double() - ref).abs() <= bound * mag).all())


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("n_atoms,mean", [
    (17_031, 27), (17_023, 60),                                # FP32, 17,024 atoms on 152 SMs: groups of one and two
    (34_045, 20), (34_051, 20), (34_051, 60), (34_051, 110),   # and of four; fewer where rows are long
    (97_301, 3), (50_001, 6), (25_003, 13), (12_007, 27)])     # FP64: one, two, four and eight lanes a row
def test_fold_groups_of_rows(cuda_device, dt, n_atoms, mean):
    """Systems large enough that a warp takes several rows, with empty, single,
    piece-long and long rows among them, on both sides of the lines at which
    fewer rows share a warp; last groups that are not whole."""
    rng = np.random.default_rng(n_atoms + mean)
    rows = rng.integers(0, 2 * mean + 1, size=n_atoms)
    special = rng.choice(n_atoms, size=n_atoms // 50, replace=False)
    rows[special] = rng.choice([0, 1, 31, 32, 33, 128, 129], size=len(special))
    rows[rng.choice(n_atoms, size=12, replace=False)] = 1000
    rows[-3:] = 33, 0, 5
    _check_fold(dt, rows, n_atoms // 3, True, mean % 2 == 0)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_fold_of_more_blocks_than_counted_in_32_bits(cuda_device, dt):
    """Rows whose group of four holds more than 2^20 blocks, which the FP32
    kernel counts in 64 bits beyond that: one long row, alone and among short
    ones, and a group whose second, third and fourth rows start beyond it."""
    _check_fold(dt, [5, 2 ** 20 + 77, 0, 3], 50, True, True, whole=True)
    rows = np.random.default_rng(4).integers(0, 9, size=60_001)
    rows[4_000:4_004] = 3, 2 ** 20 + 77, 5, 40
    rows[8_000:8_004] = 2 ** 20 + 1, 33, 0, 7
    _check_fold(dt, rows, 20_000, False, True, whole=True)
