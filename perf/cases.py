"""The work a user has this library do, as measurable cases.

A case is one pass through a public entry point of the Python API:

* ``call``   ``Plan.compute``: one force evaluation issued kernel by kernel (a
             program whose box or site count changes, or that runs few steps);
* ``step``   ``StepGraph.launch``: one step of a molecular-dynamics loop, the
             captured evaluation replayed on the next resident frame;
* ``host``   ``Plan.compute_host``: the same step for a program whose sites
             live in (pinned) host memory;
* ``batch``  ``BatchPlan.compute``: many boxes of uneven size in one call;
* ``apply``  ``Corrector.apply``: the coarse mesh corrected by the network;
* ``grad``   ``Corrector.grad``: loss and gradient of one training batch;
* ``fold``   ``wc_fold``: Wannier-centroid forces folded onto the atoms.

Sizes are those of the repository's own workloads (64, 4,096 and 72,192 water
molecules; 96 boxes of 64-8,192; training batches of 8,192 sites) or generic.
Sites are seeded synthetic water: oxygens on a jittered lattice, rigid
molecules in random orientations, one Wannier centroid (WC) a molecule.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda"
BETA = 0.4                # 1/Angstrom
MOLECULE_VOLUME = 29.9    # Angstrom^3, liquid water
MAX_MESH_POINTS = 160 ** 3
# scales of the correction network, of the size pppm_corr_calibrate finds for
# these boxes on coarse meshes (potential samples of order 1, corrections a few
# percent of the force)
S_IN, S_OUT = 4.5, 0.004


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest box, issued eagerly: host work and launch latency
        dict(name="call_64", kind="call", n_mol=64, lx=12.42, ly=12.42, lz=12.42, mx=32, my=32, mz=32, order=5,
             prec="fp32"),
        # an odd site count in a rectangular box on a mesh of uncommon lengths
        dict(name="call_ragged", kind="call", n_mol=4999, lx=40.3, ly=52.9, lz=70.1, mx=45, my=60, mz=75, order=5,
             prec="fp32"),
        # a medium box, one MD step
        dict(name="step_4096", kind="step", n_mol=4096, lx=49.7, ly=49.7, lz=49.7, mx=64, my=64, mz=64, order=5,
             prec="fp32"),
        # the same in double precision (reference runs)
        dict(name="step_4096_fp64", kind="step", n_mol=4096, lx=49.7, ly=49.7, lz=49.7, mx=64, my=64, mz=64,
             order=5, prec="fp64"),
        # the 216,576-atom system, one MD step
        dict(name="step_72192", kind="step", n_mol=72192, lx=129.3, ly=129.3, lz=129.3, mx=128, my=128, mz=128,
             order=5, prec="fp32"),
        # the same on the finer mesh
        dict(name="step_72192_m160", kind="step", n_mol=72192, lx=129.3, ly=129.3, lz=129.3, mx=160, my=160, mz=160,
             order=5, prec="fp32"),
        # the same from host memory, transfers included
        dict(name="host_72192", kind="host", n_mol=72192, lx=129.3, ly=129.3, lz=129.3, mx=128, my=128, mz=128,
             order=5, prec="fp32"),
        # many boxes of very uneven size
        dict(name="batch_96", kind="batch", nbox=96, lo=64, hi=8192, sizes=5, order=5),
        # the coarse mesh with the learned correction
        dict(name="apply_72192", kind="apply", n_mol=72192, lx=129.3, ly=129.3, lz=129.3, mx=64, my=64, mz=64,
             order=5, features="cell"),
        # one training batch
        dict(name="grad_8192", kind="grad", rows=288768, nb=8192, features="cell"),
        # forces folded onto 216,576 atoms
        dict(name="fold_72192", kind="fold", n_mol=72192, prec="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth_at_least(x):
    n = max(1, int(math.ceil(x - 1e-12)))
    while True:
        m = n
        for r in (2, 3, 5):
            while m % r == 0:
                m //= r
        if m == 1:
            return n
        n += 1


def _draw_box(rng, n_mol):
    """Edges of a box of n_mol molecules, cubic or rectangular (aspect up to 2)."""
    L = (MOLECULE_VOLUME * n_mol) ** (1.0 / 3.0)
    if rng.random() < 0.5:
        return [round(L, 3)] * 3
    a = [math.exp(rng.uniform(-0.35, 0.35)) for _ in range(3)]
    s = (a[0] * a[1] * a[2]) ** (1.0 / 3.0)
    return [round(L * v / s, 3) for v in a]


def _draw_mesh(rng, box, order, coarse=False):
    h = rng.uniform(1.6, 2.2) if coarse else rng.uniform(0.8, 1.25)
    while True:
        mesh = [_smooth_at_least(max(order + 7, L / h)) for L in box]
        if mesh[0] * mesh[1] * mesh[2] <= MAX_MESH_POINTS:
            return mesh
        h *= 1.03


def draw(rng):
    kind = rng.choice(["call", "call", "step", "step", "step", "host", "batch", "apply", "grad", "fold"])
    if kind == "batch":
        lo = _log_int(rng, 64, 256)
        return dict(kind=kind, nbox=_log_int(rng, 3, 90), lo=lo, hi=_log_int(rng, 2 * lo, 6000),
                    sizes=rng.randrange(1000), order=rng.choice([5, 5, 5, 3, 7]))
    if kind == "grad":
        return dict(kind=kind, rows=_log_int(rng, 20000, 280000), nb=_log_int(rng, 100, 16384),
                    features=rng.choice(["cell", "stated"]))
    if kind == "fold":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind=kind, n_mol=_log_int(rng, 200, 70000 if prec == "fp32" else 35000), prec=prec)
    if kind == "apply":
        n_mol, order = _log_int(rng, 500, 70000), rng.choice([5, 5, 5, 4, 7])
        box = _draw_box(rng, n_mol)
        mesh = _draw_mesh(rng, box, order, coarse=True)
        return dict(kind=kind, n_mol=n_mol, lx=box[0], ly=box[1], lz=box[2], mx=mesh[0], my=mesh[1], mz=mesh[2],
                    order=order, features=rng.choice(["cell", "stated"]))
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    n_mol = _log_int(rng, 30, 70000 if prec == "fp32" else 8000)
    order = rng.choice([5, 5, 5, 5, 3, 4, 6, 7])
    box = _draw_box(rng, n_mol)
    mesh = _draw_mesh(rng, box, order)
    return dict(kind=kind, n_mol=n_mol, lx=box[0], ly=box[1], lz=box[2], mx=mesh[0], my=mesh[1], mz=mesh[2],
                order=order, prec=prec)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _lattice(n_mol, box):
    """Lattice points per axis with at least n_mol points in all."""
    s = (box[0] * box[1] * box[2] / n_mol) ** (1.0 / 3.0)
    return [max(1, int(math.ceil(L / s - 1e-9))) for L in box]


def _water(n_mol, box, seed):
    """pos (n, 3) float64, q (n,) float64, types (n,) int8 and the lattice
    coordinates of the molecules; sites ordered O, H1 H2 per molecule, WC."""
    g = _gen(seed)
    ns = _lattice(n_mol, box)
    pick = torch.randperm(ns[0] * ns[1] * ns[2], generator=g, device=DEV)[:n_mol]
    lat = torch.stack([pick // (ns[1] * ns[2]), (pick // ns[2]) % ns[1], pick % ns[2]], 1)
    pitch = torch.tensor([L / k for L, k in zip(box, ns)], dtype=torch.float64, device=DEV)
    jitter = ((pitch - 2.3) / 2).clamp(0.0, 0.2)
    o = (lat.double() + 0.5) * pitch + _uniform(g, (n_mol, 3), -1.0, 1.0) * jitter
    # random orthonormal pairs: the molecule's bisector and its in-plane normal
    b = torch.randn((n_mol, 3), generator=g, device=DEV, dtype=torch.float64)
    b = b / b.norm(dim=1, keepdim=True)
    c = torch.linalg.cross(b, torch.randn((n_mol, 3), generator=g, device=DEV, dtype=torch.float64))
    c = c / c.norm(dim=1, keepdim=True)
    half = math.radians(104.52) / 2
    h1 = o + 0.9572 * (math.cos(half) * b + math.sin(half) * c)
    h2 = o + 0.9572 * (math.cos(half) * b - math.sin(half) * c)
    wc = o + _uniform(g, (n_mol, 1), 0.1, 0.4) * b
    pos = torch.cat([o, torch.stack([h1, h2], 1).reshape(-1, 3), wc])
    q = torch.cat([torch.full((n_mol,), 6.0, device=DEV, dtype=torch.float64),
                   torch.full((2 * n_mol,), 1.0, device=DEV, dtype=torch.float64),
                   torch.full((n_mol,), -8.0, device=DEV, dtype=torch.float64)])
    types = torch.cat([torch.full((n_mol,), t, device=DEV, dtype=torch.int8).repeat_interleave(k)
                       for t, k in ((0, 1), (1, 2), (2, 1))])
    return pos, q, types, lat, ns


def _box(case):
    return [case["lx"], case["ly"], case["lz"]]


def _mesh(case):
    return [case["mx"], case["my"], case["mz"]]


def _sites(case, seed):
    """The case's sites in the precision the entry point takes."""
    dt = torch.float64 if case.get("prec") == "fp64" else torch.float32
    pos, q, types, _, _ = _water(case["n_mol"], _box(case), seed)
    return pos.to(dt).contiguous(), q.to(dt).contiguous(), types.contiguous()


def _batch_boxes(case):
    """Molecule counts (log-uniform), edges and meshes (spacing at most 1.2) of the batch."""
    rng = np.random.default_rng(case["sizes"])
    n_mol = [int(math.exp(v)) for v in rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["nbox"])]
    edge = [(MOLECULE_VOLUME * n) ** (1.0 / 3.0) for n in n_mol]
    mesh = [_smooth_at_least(max(case["order"] + 7, L / 1.2)) for L in edge]
    return n_mol, edge, mesh


def _batch_sites(case, seed):
    n_mol, edge, _ = _batch_boxes(case)
    parts = [_water(n, [L] * 3, 1000 * seed + b)[:2] for b, (n, L) in enumerate(zip(n_mol, edge))]
    off = np.concatenate([[0], np.cumsum([p.shape[0] for p, _ in parts])]).astype(np.int64)
    return (torch.cat([p for p, _ in parts]).float().contiguous(), torch.cat([q for _, q in parts]).float().contiguous(),
            torch.from_numpy(off).to(DEV))


N_IN = {"cell": 48, "stated": 32}


def _params(n_in, seed):
    """Glorot-uniform weights and small biases of the correction network (float32)."""
    rng = np.random.default_rng(seed)
    parts = []
    for fo, fi in ((64, n_in), (64, 64), (3, 64)):
        lim = math.sqrt(6.0 / (fi + fo))
        parts += [rng.uniform(-lim, lim, size=fo * fi), rng.uniform(-0.1, 0.1, size=fo)]
    return np.concatenate(parts).astype(np.float32)


def _training_rows(case, seed):
    """A table of feature rows (BF16) and targets, and one batch of row indices."""
    g, n, n_in = _gen(seed), case["rows"], N_IN[case["features"]]
    x = torch.zeros((n, n_in), device=DEV)
    common = torch.randn((n, 1), generator=g, device=DEV)
    x[:, :27] = 0.8 * common + 0.6 * torch.randn((n, 27), generator=g, device=DEV)
    x[torch.arange(n, device=DEV), 27 + torch.randint(0, 3, (n,), generator=g, device=DEV)] = 1.0
    if case["features"] == "cell":
        u = 2 * math.pi * torch.rand((n, 3), generator=g, device=DEV)
        x[:, 30:36] = torch.stack([u.sin(), u.cos()], 2).reshape(n, 6)
    target = torch.randn((n, 3), generator=g, device=DEV)
    idx = torch.randint(0, n, (case["nb"],), generator=g, device=DEV, dtype=torch.int32)
    return x.to(torch.bfloat16), target, idx


def _fold_inputs(case, seed):
    """Site forces and the Jacobian of a local displacement model: the WC of a
    molecule depends on the three atoms of the (up to 27) molecules around it."""
    n_mol = case["n_mol"]
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    L = (MOLECULE_VOLUME * n_mol) ** (1.0 / 3.0)
    _, _, _, lat, ns = _water(n_mol, [L] * 3, seed)
    dims = torch.tensor(ns, device=DEV)
    grid = torch.full((ns[0] * ns[1] * ns[2],), -1, dtype=torch.int64, device=DEV)
    flat = lambda p: (p[..., 0] * ns[1] + p[..., 1]) * ns[2] + p[..., 2]  # noqa: E731
    grid[flat(lat)] = torch.arange(n_mol, device=DEV)
    step = torch.tensor([(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], device=DEV)
    nb = grid[flat((lat[:, None, :] + step[None]) % dims)].sort(1).values  # (n_mol, 27), -1 where empty
    cnt = (nb >= 0).sum(1)
    rows = torch.cat([nb, nb.repeat_interleave(2, 0)])  # atoms: O, then H1 H2 of each molecule
    jac_wc = rows[rows >= 0].to(torch.int32)
    zero = torch.zeros(1, dtype=torch.int64, device=DEV)
    jac_ptr = torch.cat([zero, torch.cumsum(torch.cat([cnt, cnt.repeat_interleave(2)]), 0)])
    host_ptr = torch.cat([torch.arange(n_mol + 1, device=DEV),
                          torch.full((2 * n_mol,), n_mol, device=DEV)]).to(torch.int32)
    host_wc = torch.arange(n_mol, dtype=torch.int32, device=DEV)
    g = _gen(seed + 1)
    jac = 0.02 * torch.randn((jac_wc.shape[0], 3, 3), generator=g, device=DEV, dtype=dt)
    f = torch.randn((4 * n_mol, 3), generator=g, device=DEV, dtype=dt)
    return f, host_ptr, host_wc, jac_ptr, jac_wc, jac


_compute = []


def _stream():
    """The program's one compute stream, on which its graph replays follow each other."""
    if not _compute:
        _compute.append(torch.cuda.Stream())
    return _compute[0]


def prepare(case, seed):
    from paper_2504_15508_gb300 import pppm as api

    kind = case["kind"]
    if kind == "fold":
        return dict(kind=kind, fold=api.wc_fold, n_atoms=3 * case["n_mol"], args=_fold_inputs(case, seed))
    if kind == "batch":
        _, edge, mesh = _batch_boxes(case)
        pos, q, off = _batch_sites(case, seed)
        plan = api.BatchPlan([[L] * 3 for L in edge], [[m] * 3 for m in mesh], case["order"], BETA)
        out = (torch.empty(case["nbox"], dtype=torch.float64, device=DEV), torch.empty_like(pos),
               torch.empty((case["nbox"], 6), dtype=torch.float64, device=DEV))
        stream = _stream()
        stream.wait_stream(torch.cuda.current_stream())
        plan.compute(pos, q, off, out=out, stream=stream)  # a running program's plan has tuned itself
        return dict(kind=kind, plan=plan, pos=pos, q=q, off=off, out=out, stream=stream)
    if kind == "grad":
        feat, target, idx = _training_rows(case, seed)
        coarse = api.Plan([16.0] * 3, [16] * 3, 5, BETA)
        corr = api.Corrector(coarse, _params(N_IN[case["features"]], 7), S_IN, S_OUT, features=case["features"])
        return dict(kind=kind, corr=corr, feat=feat, target=target, idx=idx)
    pos, q, types = _sites(case, seed)
    plan = api.Plan(_box(case), _mesh(case), case["order"], BETA, precision=case.get("prec", "fp32"))
    plan.reserve(pos.shape[0])
    st = dict(kind=kind, plan=plan, pos=pos, q=q)
    if kind == "step":
        st["graph"], st["stream"] = plan.graph(pos, q), _stream()
    elif kind == "host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()  # noqa: E731
        st["hpos"], st["hq"] = pin(pos), pin(q)
        st["hout"] = (np.zeros(1), pin(torch.zeros_like(pos)), np.zeros(6))
    elif kind == "apply":
        st["types"] = types
        st["corr"] = api.Corrector(plan, _params(N_IN[case["features"]], 7), S_IN, S_OUT, features=case["features"])
    return st


def run(state):
    kind = state["kind"]
    if kind == "call":
        return state["plan"].compute(state["pos"], state["q"])
    if kind == "step":
        return state["graph"].launch(state["pos"], state["q"], stream=state["stream"])
    if kind == "host":
        e, f, v = state["plan"].compute_host(state["hpos"], state["hq"], out=state["hout"])
        return np.array([e]), f, v
    if kind == "batch":
        return state["plan"].compute(state["pos"], state["q"], state["off"], out=state["out"], stream=state["stream"])
    if kind == "apply":
        return state["corr"].apply(state["pos"], state["q"], state["types"])
    if kind == "grad":
        return state["corr"].grad(state["feat"], state["target"], state["idx"])
    f, host_ptr, host_wc, jac_ptr, jac_wc, jac = state["args"]
    return state["fold"](f, state["n_atoms"], host_ptr, host_wc, jac_ptr, jac_wc, jac)


# ---------------------------------------------------------------- work and tolerance
def _solve_work(n, mesh, order, real, inputs):
    """One PPPM solve: sites in, forces out, and the influence table; the
    stencil sums of spread and gather, four real 3D FFTs, the influence
    multiply with energy and virial."""
    N = mesh[0] * mesh[1] * mesh[2]
    half = mesh[0] * mesh[1] * (mesh[2] // 2 + 1)
    p3 = order ** 3
    flops = n * p3 * (3 + 7) + 4 * 2.5 * N * math.log2(N) + 40 * half
    return n * inputs * 7 + half * real, flops


def work(case):
    kind = case["kind"]
    if kind == "fold":
        n, r = case["n_mol"], 8 if case["prec"] == "fp64" else 4
        L = (MOLECULE_VOLUME * n) ** (1.0 / 3.0)
        ns = _lattice(n, [L] * 3)
        blocks = 3 * n * (1 + 26 * (n - 1) / max(1, ns[0] * ns[1] * ns[2] - 1))
        return {"bytes": blocks * (9 * r + 4) + n * (3 * (8 + 4) + 4) + 7 * n * 3 * r, "flops": blocks * 18}
    if kind == "grad":
        n_in, nb = N_IN[case["features"]], case["nb"]
        par = 64 * n_in + 64 * 64 + 3 * 64
        return {"bytes": nb * (2 * n_in + 12 + 4) + 8 * par, "flops": nb * 6 * par}
    if kind == "batch":
        n_mol, _, mesh = _batch_boxes(case)
        w = [_solve_work(4 * n, [m] * 3, case["order"], 4, 4) for n, m in zip(n_mol, mesh)]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    r = 8 if case.get("prec") == "fp64" else 4
    n = 4 * case["n_mol"]
    b, f = _solve_work(n, _mesh(case), case["order"], r, r)
    if kind == "apply":
        n_in, p = N_IN[case["features"]], case["order"]
        f += n * (2 * 3 * p * ((p + 2) ** 2 + 3 * (p + 2) + 9) + 2 * (64 * n_in + 64 * 64 + 3 * 64))
        b += n
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the error against 64 bits, measured over the ranges."""
    kind = case["kind"]
    if kind == "fold":  # one sum of ~80 blocks an atom: 3.4e-8 (2.4e-16)
        return {"rel": 1e-15 if case["prec"] == "fp64" else 1.5e-7}
    if kind == "grad":  # sums over the batch in 32 bits: 1.5e-7
        return {"rel": 6e-7}
    if kind == "apply":  # features and hidden activations in BF16; the correction is a part of the force
        return {"rel": 1e-3}
    if case.get("prec") == "fp64":  # 7e-15 on the forces, more on small boxes and high orders
        return {"rel": 1e-13}
    # the mesh and its transforms in 32 bits: 1.6e-6 on the forces, 3e-6 on the
    # smallest boxes, 4e-6 over a batch of them
    return {"rel": 1.5e-5 if kind == "batch" else 1e-5}


# ---------------------------------------------------------------- 64-bit results
def _weights(pos, box, mesh, p):
    """Per axis the mesh indices (n, p) and B-spline weights (n, p) of every site."""
    idx, wts = [], []
    kmin = -(p - 1) // 2 if p % 2 else -p // 2 + 1
    for d in range(3):
        u = torch.remainder(pos[:, d], box[d]) * (mesh[d] / box[d])
        g = torch.floor(u + 0.5) if p % 2 else torch.floor(u)
        pts = g[:, None] + torch.arange(kmin, kmin + p, device=DEV)
        t = pts - u[:, None] + 0.5 * p  # argument of the uniform B-spline on [0, p)
        w = [((t - j >= 0) & (t - j < 1)).double() for j in range(p)]
        for m in range(2, p + 1):
            w = [((t - j) * w[j] + (m - t + j) * w[j + 1]) / (m - 1) for j in range(p - m + 1)]
        wts.append(w[0])
        idx.append(torch.remainder(pts.long(), mesh[d]))
    return idx, wts


def _interpolate(fields, pos, box, mesh, p):
    (ix, iy, iz), (wx, wy, wz) = _weights(pos, box, mesh, p)
    flat = torch.stack([f.reshape(-1) for f in fields], 1)
    out = torch.zeros((pos.shape[0], len(fields)), dtype=torch.float64, device=DEV)
    for a in range(p):
        for b in range(p):
            row = (ix[:, a] * mesh[1] + iy[:, b]) * mesh[2]
            wab = wx[:, a] * wy[:, b]
            for c in range(p):
                out += (wab * wz[:, c])[:, None] * flat[row + iz[:, c]]
    return out


def _influence(box, mesh, p):
    """Optimal influence function for ik differentiation on the half spectrum,
    alias range 2 in the numerator, 20 in the separable denominator."""
    k1 = []
    for d in range(3):
        i = torch.arange(mesh[d], device=DEV)
        m = torch.where(i <= mesh[d] // 2, i, i - mesh[d]).double()
        if d == 2:
            m = m[: mesh[2] // 2 + 1]
        k1.append(2 * math.pi * m / box[d])
    h = [box[d] / mesh[d] for d in range(3)]
    u2 = lambda k, d: torch.sinc(k * (h[d] / 2) / math.pi) ** (2 * p)  # noqa: E731
    shape = lambda v, d: v.reshape([-1 if e == d else 1 for e in range(3)])  # noqa: E731
    den = 1.0
    for d in range(3):
        den = den * shape(sum(u2(k1[d] + 2 * math.pi * n / h[d], d) for n in range(-20, 21)), d)
    k = [shape(k1[d], d) for d in range(3)]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    num = torch.zeros_like(k2)
    for nx in range(-2, 3):
        for ny in range(-2, 3):
            for nz in range(-2, 3):
                kn = [k[d] + 2 * math.pi * n / h[d] for d, n in enumerate((nx, ny, nz))]
                kn2 = kn[0] ** 2 + kn[1] ** 2 + kn[2] ** 2
                dot = k[0] * kn[0] + k[1] * kn[1] + k[2] * kn[2]
                w = u2(kn[0], 0) * u2(kn[1], 1) * u2(kn[2], 2)
                num += torch.where(kn2 > 0, dot / kn2 * 4 * math.pi * torch.exp(-kn2 / (4 * BETA ** 2)) * w,
                                   torch.zeros_like(kn2))
    return torch.where(k2 > 0, num / (k2 * den * den), torch.zeros_like(k2)), k, k2


def _solve(pos, q, box, mesh, p, potential=False):
    """Energy (1,), forces (n, 3) and virial (6,) of the PPPM solve in 64 bits."""
    pos, q = pos.double(), q.double()
    N = mesh[0] * mesh[1] * mesh[2]
    V = box[0] * box[1] * box[2]
    (ix, iy, iz), (wx, wy, wz) = _weights(pos, box, mesh, p)
    rho = torch.zeros(N, dtype=torch.float64, device=DEV)
    for a in range(p):
        for b in range(p):
            row = (ix[:, a] * mesh[1] + iy[:, b]) * mesh[2]
            wab = q * wx[:, a] * wy[:, b]
            for c in range(p):
                rho.index_add_(0, row + iz[:, c], wab * wz[:, c])
    rho = rho.reshape(mesh) * (N / V)
    hat = torch.fft.rfftn(rho)
    G, k, k2 = _influence(box, mesh, p)
    # weight 2 for the modes whose mirror image the half spectrum leaves out
    w = torch.full((mesh[2] // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    w[0] = 1.0
    if mesh[2] % 2 == 0:
        w[-1] = 1.0
    e = V / (2.0 * N * N) * G * (hat.real ** 2 + hat.imag ** 2)
    c = torch.where(k2 > 0, 2 * (1 + k2 / (4 * BETA ** 2)) / k2, torch.zeros_like(k2))
    vir = [(w * e * (1 - c * k[d] ** 2)).sum() for d in range(3)]
    # an index N/2 is its own mirror image with its sign kept, so off-diagonal
    # terms of a pair add up only if both or neither of their factors flip
    image = [-v for v in k]
    for d in range(3):
        if mesh[d] % 2 == 0:
            image[d].reshape(-1)[mesh[d] // 2] *= -1.0
    for a, b in ((0, 1), (0, 2), (1, 2)):
        vir.append(-(e * c * (k[a] * k[b] + (w - 1.0) * image[a] * image[b])).sum())
    phi = G * hat
    fields = []
    for d in range(3):
        kd = k[d].clone()
        if mesh[d] % 2 == 0:
            kd.reshape(-1)[mesh[d] // 2] = 0.0
        fields.append(torch.fft.irfftn(-1j * kd * phi, s=mesh))
    f = q[:, None] * _interpolate(fields, pos, box, mesh, p)
    out = ((w * e).sum().reshape(1), f, torch.stack(vir))
    return out + (torch.fft.irfftn(phi, s=mesh),) if potential else out


def _network(theta, n_in):
    t = torch.from_numpy(theta).to(DEV).to(torch.bfloat16).double()
    sizes = [(64, n_in), (64,), (64, 64), (64,), (3, 64), (3,)]
    out, o = [], 0
    for s in sizes:
        k = int(np.prod(s))
        out.append(t[o:o + k].reshape(s))
        o += k
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "fold":
        f, host_ptr, host_wc, jac_ptr, jac_wc, jac = _fold_inputs(case, seed)
        n = 3 * case["n_mol"]
        f, jac = f.double(), jac.double()
        out, fw = f[:n].clone(), f[n:]
        rows = torch.arange(n, device=DEV).repeat_interleave((host_ptr[1:] - host_ptr[:-1]).long())
        out.index_add_(0, rows, fw[host_wc.long()])
        rows = torch.arange(n, device=DEV).repeat_interleave(jac_ptr[1:] - jac_ptr[:-1])
        return out.index_add_(0, rows, torch.einsum("kab,ka->kb", jac, fw[jac_wc.long()]))
    if kind == "grad":
        feat, target, idx = _training_rows(case, seed)
        W1, b1, W2, b2, W3, b3 = _network(_params(N_IN[case["features"]], 7), N_IN[case["features"]])
        x, t = feat[idx.long()].double(), target[idx.long()].double()
        h1 = torch.tanh(x @ W1.T + b1)
        h2 = torch.tanh(h1 @ W2.T + b2)
        r = h2 @ W3.T + b3 - t
        dy = 2 * r / x.shape[0]
        d2 = (dy @ W3) * (1 - h2 * h2)
        d1 = (d2 @ W2) * (1 - h1 * h1)
        parts = [d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0)]
        return (r * r).sum().reshape(1) / x.shape[0], torch.cat([v.reshape(-1) for v in parts])
    if kind == "batch":
        _, edge, mesh = _batch_boxes(case)
        pos, q, off = _batch_sites(case, seed)
        o = off.tolist()
        r = [_solve(pos[a:b], q[a:b], [L] * 3, [m] * 3, case["order"])
             for a, b, L, m in zip(o, o[1:], edge, mesh)]
        return torch.cat([v[0] for v in r]), torch.cat([v[1] for v in r]), torch.stack([v[2] for v in r])
    pos, q, types = _sites(case, seed)
    box, mesh, p = _box(case), _mesh(case), case["order"]
    if kind != "apply":
        return _solve(pos, q, box, mesh, p)
    energy, forces, virial, phi = _solve(pos, q, box, mesh, p, potential=True)
    n, n_in = pos.shape[0], N_IN[case["features"]]
    x = torch.zeros((n, n_in), dtype=torch.float64, device=DEV)
    h = torch.tensor([L / m for L, m in zip(box, mesh)], dtype=torch.float64, device=DEV)
    pos = pos.double()
    for a in range(27):
        step = torch.tensor([a // 9 - 1, a // 3 % 3 - 1, a % 3 - 1], dtype=torch.float64, device=DEV)
        x[:, a] = S_IN * _interpolate([phi], pos + h * step, box, mesh, p)[:, 0]
    x[torch.arange(n, device=DEV), 27 + types.long()] = 1.0
    if case["features"] == "cell":
        u = 2 * math.pi * pos / h
        x[:, 30:36] = torch.stack([u.sin(), u.cos()], 2).reshape(n, 6)
    W1, b1, W2, b2, W3, b3 = _network(_params(n_in, 7), n_in)
    y = torch.tanh(torch.tanh(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    return energy, forces + q.double()[:, None] * S_OUT * y, virial
