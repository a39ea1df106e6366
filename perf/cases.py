"""The measured work of the library: what a plane-wave program asks of it, through the public binding.

Each case is a dict of plain values.  `kind` names the call: H|psi> on whole k-point sets, H and S
on an uneven work list (what an iterative solver applies), H on cells with different projector sets
in one launch, H on host buffers, the batched Davidson, the batched Sternheimer CG, the induced
density and the reduced eigensolver.  Inputs are drawn on the GPU from the seed: atoms displaced
around their sites, a random smooth local potential, random symmetric projector coefficients, and
orthonormal vectors whose coefficients fall off with the kinetic energy, as starting wave-functions
do.  Geometry (k-grids, spheres) depends on the case alone and is kept between preparations.

Units are Rydberg; layouts are those of include/pwk.h.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2412_01695_gb300 import pwk

ALAT = 7.5                                            # bohr, every cell
SITES = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]], float)   # cubic cells
Q_FRAC = (0.25, 0.0, 0.0)                             # phonon wave-vector, 2 pi / a
PRECISION = {"fp64": pwk.PWK_FP64, "fp32": pwk.PWK_FP32, "mixed": pwk.PWK_FP32_C128}


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one H application inside an interactive or testing run: launch latency
        _h("hpsi_fp32_8k_8b_n16", "hpsi", "fp32", "fcc", 1, 1, 20.0, 16, (2, 2, 2), 8),
        # the ordinary block of k-points of a one-atom metal: throughput of the FP32 operator
        _h("hpsi_fp32_512k_20b_n24", "hpsi", "fp32", "fcc", 1, 2, 45.0, 24, (8, 8, 8), 20),
        # a four-atom cell with a wide projector set and many bands: the largest operator call
        _h("hpsi_fp32_343k_40b_n36", "hpsi", "fp32", "sc", 4, 2, 40.0, 36, (7, 7, 7), 40),
        # the reference-precision operator on an ordinary block
        _h("hpsi_fp64_64k_20b_n24", "hpsi", "fp64", "fcc", 1, 2, 45.0, 24, (4, 4, 4), 20),
        # H and S of the vectors a solver still iterates on: uneven list, ultrasoft, odd grid
        _h("hspsi_items_fp64_27k_16b_n27", "items", "fp64", "sc", 2, 1, 25.0, 27, (3, 3, 3), 16),
        # work of three cells with 0, 4 and 9 projectors in one launch (a serving loop)
        _h("hpsi_multi_fp32_64k_12b_n24", "multi", "fp32", "fcc", 1, 2, 45.0, 24, (4, 4, 4), 12),
        # vectors that live in host memory: copies in and out around the operator
        _h("hpsi_host_fp32_216k_20b_n24", "host", "fp32", "fcc", 1, 2, 45.0, 24, (6, 6, 6), 20),
        # a band structure or SCF step: the batched Davidson in its mixed mode
        _h("davidson_mixed_64k_20b_n24", "davidson", "mixed", "fcc", 1, 2, 45.0, 24, (4, 4, 4), 20),
        # a small FP64 solve: few k-points, launches and the reduced problem's latency count
        _h("davidson_fp64_8k_8b_n16", "davidson", "fp64", "fcc", 1, 1, 20.0, 16, (2, 2, 2), 8),
        # the DFPT response of one perturbation
        _h("sternheimer_mixed_64k_12b_n20", "sternheimer", "mixed", "fcc", 1, 2, 35.0, 20, (4, 4, 4), 12),
        # the induced density that follows it
        _h("drho_fp64_64k_12b_n20", "drho", "fp64", "fcc", 1, 2, 35.0, 20, (4, 4, 4), 12),
        # the reduced generalized eigenproblems of a Davidson step on their own
        {"name": "eigh_128x80_20", "kind": "eigh", "problems": 128, "n": 80, "nev": 20},
    ]


def _h(name, kind, precision, lattice, atoms, lmax, ecut, grid, mp, bands):
    c = {"name": name} if name else {}
    c.update(kind=kind, precision=precision, lattice=lattice, atoms=atoms, lmax=lmax, ecut=float(ecut),
             grid=grid, k1=mp[0], k2=mp[1], k3=mp[2], bands=bands)
    return c


def draw(rng):
    """One more case: any call, precision, grid size (odd ones among them), cut-off, projector set,
    k-set and band count of the ranges above; sizes spread over their logarithm."""
    kind = rng.choice(["hpsi", "hpsi", "hpsi", "items", "multi", "host", "davidson", "sternheimer", "drho", "eigh"])
    if kind == "eigh":
        n = int(round(math.exp(rng.uniform(math.log(12), math.log(160)))))
        nev = max(1, int(n * rng.uniform(0.1, 0.5)))
        most = 128 * (80 / n) ** 3
        return {"kind": kind, "problems": int(round(math.exp(rng.uniform(0.0, math.log(max(2.0, min(512.0, most))))))),
                "n": n, "nev": nev}
    grids = [12, 15, 16, 18, 20, 24, 25, 27] + ([30, 32, 36] if kind in ("hpsi", "items", "multi") else [])
    grid = rng.choice(grids)
    lattice = rng.choice(["fcc", "sc"])
    atoms = 1 if lattice == "fcc" else rng.choice([1, 2, 4])
    lmax = rng.choice([0, 1, 2])
    shift = 0.5 + (0.25 if kind in ("sternheimer", "drho") else 0.0)
    ai = ALAT / math.sqrt(2) if lattice == "fcc" else ALAT
    root = (grid // 4 + 0.95 - shift) * 2 * math.pi / ai
    ecut = round(root * root * rng.uniform(0.7, 0.98), 2)
    npw = ecut ** 1.5 * ALAT ** 3 * (0.25 if lattice == "fcc" else 1.0) / (6 * math.pi ** 2)
    if kind in ("hpsi", "items", "multi", "host"):
        precision = rng.choice(["fp32", "fp32", "fp64", "mixed"]) if kind != "host" else rng.choice(["fp32", "fp64"])
        cost = grid ** 3 * (30.0 if precision == "fp64" else 1.0)
        most = min(343 * 40 * 36 ** 3 / cost, 20000)
        if kind == "host":
            most = min(most, 216 * 20 * 538 / npw)
        bands = int(round(math.exp(rng.uniform(0.0, math.log(40)))))
        side = max(1.0, (most / bands) ** (1 / 3))
        mp = [max(1, int(math.exp(rng.uniform(0.0, math.log(min(side, 8.0) + 1e-9))) + 0.5)) for _ in range(3)]
        return _h("", kind, precision, lattice, atoms, lmax, ecut, grid, mp, bands)
    precision = rng.choice(["mixed", "fp64"])
    if kind == "davidson":
        # cells whose smallest sphere holds the largest basis (4 bands' worth)
        bands = max(2, min(int(math.exp(rng.uniform(math.log(2), math.log(20)))), int(npw * 0.8 / 8)))
        most = min(64.0, 64 * 538 / npw) * (0.15 if precision == "fp64" else 1.0)
    else:
        bands = max(1, min(int(math.exp(rng.uniform(0.0, math.log(12)))), int(npw / 10)))
        most = min(64.0, 64 * (370 / npw) ** 2) * (0.3 if precision == "fp64" and kind == "sternheimer" else 1.0)
    side = max(1.0, most ** (1 / 3))
    mp = [max(1, int(rng.uniform(1.0, side + 0.5))) for _ in range(3)]
    return _h("", kind, precision, lattice, atoms, lmax, ecut, grid, mp, bands)


# ------------------------------------------------------------------------------ geometry
def _lattice(case):
    if case["lattice"] == "fcc":
        return 0.5 * ALAT * np.array([[0, 1, 1], [1, 0, 1], [1, 1, 0]], float), SITES[:1] @ (ALAT * np.eye(3))
    return ALAT * np.eye(3), ALAT * SITES[:case["atoms"]]


@functools.lru_cache(maxsize=64)
def _spheres(lattice, atoms, ecut, mp, shifted):
    """k-points [nk][3], sphere sizes [nk] and Miller indices [nk][npw_max][3] (zero padded)."""
    A, _ = _lattice({"lattice": lattice, "atoms": atoms})
    B = 2 * np.pi * np.linalg.inv(A).T
    axes = [(2 * np.arange(1, n + 1) - n - 1) / (2.0 * n) for n in mp]
    k = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3) @ B
    if shifted:
        k = k + 2 * np.pi / ALAT * np.array(Q_FRAC)
    top = int(math.sqrt(ecut) * np.linalg.norm(A[0]) / (2 * np.pi) + 2)
    r = np.arange(-top, top + 1)
    m = np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    g = m @ B
    sets = []
    for kc in k:
        g2 = np.sum((g + kc) ** 2, axis=1)
        s = np.nonzero(g2 < ecut)[0]
        sets.append(m[s[np.argsort(g2[s], kind="stable")]])
    npw = np.array([len(s) for s in sets], np.int32)
    out = np.zeros((len(k), int(npw.max()), 3), np.int32)
    for i, s in enumerate(sets):
        out[i, :len(s)] = s
    return k, npw, out


def _geometry(case, shifted=False):
    return _spheres(case["lattice"], case["atoms"], case["ecut"], (case["k1"], case["k2"], case["k3"]), shifted)


# ------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1 + 7919 * int(seed))
    return g


def _uniform(gen, *shape):
    return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1


def _complex(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128)


def _field(gen, case, real):
    """sum_G c(G) e^{iG.r} with c normal, falling off as exp(-|G|^2/8), |G|^2 < 4 ecut."""
    N = case["grid"]
    A, _ = _lattice(case)
    B = torch.from_numpy(2 * np.pi * np.linalg.inv(A).T).cuda()
    f = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
    m = torch.stack(torch.meshgrid(f, f, f, indexing="ij"), -1)
    g2 = ((m @ B) ** 2).sum(-1)
    c = _complex(gen, N, N, N) * torch.exp(-g2 / 8)
    c[g2 >= 4 * case["ecut"]] = 0
    if N % 2 == 0:
        c[(m.abs() * 2 >= N).any(-1)] = 0
    if not real:
        return torch.fft.ifftn(c, norm="forward").contiguous()
    c[0, 0, 0] = 0
    return (torch.fft.ifftn(c, norm="forward").real * math.sqrt(2)).contiguous()


def _symmetric(gen, atoms, per_atom, positive):
    out = torch.zeros(atoms * per_atom, atoms * per_atom, dtype=torch.float64, device="cuda")
    for i in range(atoms):
        r = _uniform(gen, per_atom, per_atom)
        s = slice(i * per_atom, (i + 1) * per_atom)
        out[s, s] = 20.0 / per_atom * (r @ r.T) if positive else torch.triu(r) + torch.triu(r, 1).T
    return out.cpu().numpy() if not positive else (0.5 * (out + out.T)).cpu().numpy()


def _projectors(case, tau, kc, npw, miller, lmax):
    """beta [nk][nkb][npw_max]: Gaussian projectors of angular momentum 0..lmax on every atom."""
    A, _ = _lattice(case)
    B = torch.from_numpy(2 * np.pi * np.linalg.inv(A).T).cuda()
    q = torch.from_numpy(kc).cuda()[:, None, :] + torch.from_numpy(miller).cuda().double() @ B
    x, y, z = q.unbind(-1)
    r2 = x * x + y * y + z * z
    p4 = 4 * math.pi
    sh = [[torch.full_like(x, 1 / math.sqrt(p4))]]
    if lmax >= 1:
        sh.append([math.sqrt(3 / p4) * v for v in (x, y, z)])
    if lmax >= 2:
        a = math.sqrt(15 / p4)
        sh.append([a * x * y, a * y * z, math.sqrt(5 / (4 * p4)) * (3 * z * z - r2), a * x * z, a / 2 * (x * x - y * y)])
    inside = torch.arange(miller.shape[1], device="cuda")[None, :] < torch.from_numpy(npw).cuda()[:, None]
    radial = torch.exp(-r2 / 4) * inside / math.sqrt(abs(np.linalg.det(A)))
    rows = []
    for t in tau:
        w = radial * torch.exp(-1j * (q @ t))
        rows += [((-1j) ** l) * h * w for l in range(lmax + 1) for h in sh[l]]
    return torch.stack(rows, 1).contiguous()


def _kinetic(case, kc, miller):
    A, _ = _lattice(case)
    q = torch.from_numpy(kc).cuda()[:, None, :] + torch.from_numpy(miller).cuda().double() @ torch.from_numpy(
        2 * np.pi * np.linalg.inv(A).T).cuda()
    return (q * q).sum(-1)


def _orthonormal(x):
    """Orthonormal rows spanning those of x [nk][nb][np] (Cholesky, twice)."""
    for _ in range(2):
        lo = torch.linalg.cholesky(x @ x.mH)
        x = torch.linalg.solve_triangular(lo, x, upper=False)
    return x.contiguous()


def _vectors(gen, case, g2, npw, bands, orthonormal=True):
    inside = torch.arange(g2.shape[1], device="cuda")[None, :] < torch.from_numpy(npw).cuda()[:, None]
    x = _complex(gen, g2.shape[0], bands, g2.shape[1]) * (inside / (1 + 4 * g2 / case["ecut"]))[:, None, :]
    if orthonormal and bands <= int(npw.min()):
        return _orthonormal(x)
    return (x / x.abs().square().sum(-1, keepdim=True).sqrt()).contiguous()


def _cell(gen, case, lmax=None, with_v=None):
    """One cell's tables: spheres, projectors, coefficients and potential, as torch tensors."""
    lmax = case["lmax"] if lmax is None else lmax
    kc, npw, miller = _geometry(case)
    A, tau = _lattice(case)
    tau = torch.from_numpy(tau).cuda() + 0.02 * ALAT * _uniform(gen, len(tau), 3)
    c = {"A": A, "k": kc, "npw": npw, "miller": miller, "tau": tau, "beta": None, "D": None, "q": None}
    if lmax >= 0:
        c["beta"] = _projectors(case, tau, kc, npw, miller, lmax)
        c["D"] = _symmetric(gen, len(tau), (lmax + 1) ** 2, False)
        if case["kind"] == "items":
            c["q"] = _symmetric(gen, len(tau), (lmax + 1) ** 2, True)
    c["V"] = _field(gen, case, True) if with_v is None else with_v
    c["g2"] = _kinetic(case, kc, miller)
    return c


def _shifted(case, cell):
    """The k+q set of the same cell."""
    kc, npw, miller = _geometry(case, True)
    d = dict(cell, k=kc, npw=npw, miller=miller, g2=_kinetic(case, kc, miller))
    d["beta"] = _projectors(case, cell["tau"], kc, npw, miller, case["lmax"])
    return d


def _plan(case, cell):
    p = pwk.plan_create(cell["A"], case["grid"], cell["k"], cell["npw"], cell["miller"], cell["beta"], cell["D"],
                        cell["V"])
    if cell["q"] is not None:
        p.set_overlap(cell["q"])
    return p


def _dense(case, cell, ks):
    """H(k) of the k-points ks, dense, padding decoupled on the diagonal."""
    N = case["grid"]
    vg = torch.fft.fftn(cell["V"], norm="forward").reshape(-1)
    m = torch.from_numpy(cell["miller"][ks]).cuda().long()
    d = (m[:, :, None, :] - m[:, None, :, :]) % N
    H = vg[(d[..., 0] * N + d[..., 1]) * N + d[..., 2]]
    b = cell["beta"][ks]
    H = H + (b.mT @ torch.from_numpy(cell["D"]).cuda().to(b.dtype)) @ b.conj()
    np_ = m.shape[1]
    inside = torch.arange(np_, device="cuda")[None, :] < torch.from_numpy(cell["npw"][ks]).cuda()[:, None]
    H = H * (inside[:, :, None] & inside[:, None, :])
    return H + torch.diag_embed(torch.where(inside, cell["g2"][ks], torch.full_like(cell["g2"][ks], 1e3)).to(H.dtype))


def _lowest(case, cell, bands):
    """The lowest eigenpairs of H(k), as a program has them after its band calculation: inverse
    iteration on the dense matrices and a Rayleigh-Ritz step, in 64 bits."""
    nk, np_ = cell["miller"].shape[:2]
    block = min(bands + 12, int(cell["npw"].min()))
    gen = _generator(12345)
    vecs, vals = [], []
    step = max(1, 6000000 // (np_ * np_))
    for k0 in range(0, nk, step):
        ks = np.arange(k0, min(nk, k0 + step))
        H = _dense(case, cell, ks)
        b = cell["beta"][ks]
        weight = torch.linalg.matrix_norm(b.conj() @ b.mT).max() * float(np.linalg.norm(cell["D"], 2))
        sigma = cell["V"].min() - weight
        inv = torch.linalg.inv(H - sigma * torch.eye(np_, device="cuda", dtype=H.dtype))
        x = _vectors(gen, case, cell["g2"][ks], cell["npw"][ks], block)
        for it in range(60):
            x = x @ inv.mT
            if it % 4 == 3:
                x = _orthonormal(x)
        w, u = torch.linalg.eigh(x.conj() @ H @ x.mT)
        vecs.append((u.mT @ x)[:, :bands])
        vals.append(w[:, :bands + 1])
    return torch.cat(vecs).contiguous(), torch.cat(vals)


def _response(case, seed):
    """Inputs of the Sternheimer solve: valence states at k and k+q, eigenvalues, alpha, dv.  The
    occupied energies are kept 0.05 Ry below the first empty state at k+q (an insulator's gap)."""
    gen = _generator(seed)
    cell = _cell(gen, case)
    cell_q = _shifted(case, cell)
    u, e = _lowest(case, cell, case["bands"])
    uq, eq = _lowest(case, cell_q, case["bands"])
    n = case["bands"]
    eps = torch.minimum(e[:, :n], eq[:, n:n + 1] - 0.05).contiguous()
    both = torch.cat([eps, eq[:, :n]], 1)
    alpha = torch.clamp(2 * (both.amax(1) - both.amin(1)), min=0.01).contiguous()
    return cell, cell_q, u, uq, eps, alpha, _field(gen, case, False)


def _density_inputs(case, seed):
    gen = _generator(seed)
    cell = _cell(gen, case)
    cell_q = _shifted(case, cell)
    u = _vectors(gen, case, cell["g2"], cell["npw"], case["bands"])
    uq = _vectors(gen, case, cell_q["g2"], cell_q["npw"], case["bands"])
    du = _vectors(gen, case, cell_q["g2"], cell_q["npw"], case["bands"], False)
    w = torch.full((u.shape[0],), 1.0 / u.shape[0], dtype=torch.float64, device="cuda")
    return cell, cell_q, u, uq, du, w


def _pencils(case, seed):
    """Reduced matrices as a Davidson step has them: H~ with a spectrum spread over a few Ry, S~ of
    unit-norm basis vectors that are not orthogonal."""
    gen = _generator(seed)
    p, n = case["problems"], case["n"]
    x = _complex(gen, p, n, 3 * n)
    x[:, n // 2:] += 0.5 * x[:, :n - n // 2]
    x = x / x.abs().square().sum(-1, keepdim=True).sqrt()
    d = torch.sort(torch.rand(p, 1, 3 * n, generator=gen, device="cuda", dtype=torch.float64) * 10 - 1, -1)[0]
    H, S = (x.conj() * d) @ x.mT, x.conj() @ x.mT
    return (0.5 * (H + H.mH)).contiguous(), (0.5 * (S + S.mH)).contiguous()


def _worklist(case, seed):
    """(k, in, out) entries: an uneven number of bands per k-point, slots in any order."""
    r = np.random.Generator(np.random.PCG64(int(seed)))
    nk, nb = case["k1"] * case["k2"] * case["k3"], case["bands"]
    rows = []
    for k in range(nk):
        n = int(r.integers(0, nb + 1)) if k else nb
        a, b = r.permutation(nb)[:n], r.permutation(nb)[:n]
        rows += [(k, i, j) for i, j in zip(a, b)]
    return np.array(rows, np.int32)


def _multi_cells(gen, case):
    return [_cell(gen, case, l) for l in (case["lmax"], min(1, case["lmax"]), -1)]


# ------------------------------------------------------------------------------ the calls
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "eigh":
        s["H"], s["S"] = _pencils(case, seed)
        return s
    s["prec"] = PRECISION[case["precision"]]
    dt = torch.complex64 if case["precision"] == "fp32" else torch.complex128
    nb, N = case["bands"], case["grid"]
    if kind == "sternheimer":
        cell, cell_q, u, uq, eps, alpha, dv = _response(case, seed)
        s.update(plan=_plan(case, cell), plan_q=_plan(case, cell_q), u=u, uq=uq, eps=eps, alpha=alpha, dv=dv,
                 out=torch.zeros_like(uq))
    elif kind == "drho":
        cell, cell_q, u, uq, du, w = _density_inputs(case, seed)
        s.update(plan=_plan(case, cell), plan_q=_plan(case, cell_q), u=u, uq=uq, du=du, w=w,
                 out=torch.zeros(N, N, N, dtype=torch.complex128, device="cuda"))
    elif kind == "multi":
        gen = _generator(seed)
        cells = _multi_cells(gen, case)
        s["plans"] = [_plan(case, c) for c in cells]
        s["x"] = [_vectors(gen, case, c["g2"], c["npw"], nb).to(dt) for c in cells]
        s["out"] = [torch.zeros_like(x) for x in s["x"]]
        nk = len(cells[0]["k"])
        i, k, b = np.meshgrid(np.arange(3), np.arange(nk), np.arange(nb), indexing="ij")
        s["items"] = torch.from_numpy(np.stack([i, k, b, b], -1).reshape(-1, 4).astype(np.int32)).cuda()
    else:
        gen = _generator(seed)
        cell = _cell(gen, case)
        s["plan"] = _plan(case, cell)
        x = _vectors(gen, case, cell["g2"], cell["npw"], nb)
        s["x"] = x.to(dt)
        s["out"] = torch.zeros_like(s["x"])
        if kind == "items":
            s["sout"] = torch.zeros_like(s["x"])
            s["items"] = torch.from_numpy(_worklist(case, seed)).cuda()
        elif kind == "host":
            s["hx"] = s["x"].cpu().pin_memory()
            s["hout"] = torch.zeros_like(s["hx"]).pin_memory()
        elif kind == "davidson":
            s["eig"] = torch.zeros(x.shape[0], nb, dtype=torch.float64, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "hpsi":
        pwk.hpsi_batched(s["plan"], s["prec"], s["x"], s["out"], s["case"]["bands"])
        return s["out"]
    if kind == "items":
        pwk.hspsi_items(s["plan"], s["prec"], s["x"], s["out"], s["sout"], s["items"], s["case"]["bands"])
        return [s["out"], s["sout"]]
    if kind == "multi":
        pwk.hpsi_multi(s["plans"], s["prec"], s["x"], s["out"], s["items"])
        return s["out"]
    if kind == "host":
        pwk.hpsi_batched_host(s["plan"], s["prec"], s["hx"], s["hout"], s["x"], s["out"], s["case"]["bands"], 4)
        torch.cuda.current_stream().synchronize()   # the program reads the host result next
        return s["hout"]
    if kind == "davidson":
        psi = s["x"].to(torch.complex128, copy=True)
        pwk.davidson_batched(s["plan"], s["prec"], psi, s["eig"], s["case"]["bands"], 1e-10, 1e-7, 300)
        # the eigenvectors turned to the trial set (as an SCF loop aligns them with the last
        # step's): sum_n |psi_n><psi_n|phi_b>, free of their phases and of mixing in a level
        return [s["eig"], (s["x"] @ psi.mH) @ psi]
    if kind == "sternheimer":
        pwk.sternheimer_cg_batched(s["plan_q"], s["plan"], s["prec"], s["u"], s["eps"], s["uq"], s["case"]["bands"],
                                   s["alpha"], s["dv"], s["out"], 1e-10)
        return s["out"]
    if kind == "drho":
        pwk.drho_batched(s["plan_q"], s["plan"], s["prec"], s["u"], s["uq"], s["du"], s["case"]["bands"], s["w"], s["out"])
        return s["out"]
    eig, vec = pwk.eigh_batched(s["H"], s["S"], s["case"]["nev"])
    return [eig, vec @ vec.mH]   # the eigenvalues and the density matrix of the lowest states


# ------------------------------------------------------------------------------ work
def _operator_work(case, cells, items, io):
    """Bytes and flops of H (and S) on `items` band-k: the pruned transform pair, the kinetic and
    local products, and the two projector products; projector tables read once per k-point."""
    N = case["grid"]
    b = f = 0.0
    wide = 16 if case["precision"] == "fp64" else 8
    for lmax in cells:
        kc, npw, miller = _geometry(case)
        n, nk = float(npw.mean()), len(kc)
        nkb = 0 if lmax < 0 else (1 if case["lattice"] == "fcc" else case["atoms"]) * (lmax + 1) ** 2
        m0 = miller[0, :npw[0]]
        sticks = len({(int(a), int(c)) for a, c, _ in m0})
        planes = len({int(a) for a, _, _ in m0})
        lines = sticks + planes * N + N * N
        f += items * (2 * lines * 5 * N * math.log2(N) + 2 * N ** 3 + 2 * n + 16 * nkb * n)
        outs = 3 if case["kind"] == "items" else 2
        b += items * outs * n * io + nk * n * (nkb * wide + 12) + N ** 3 * wide / 2
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "eigh":
        p, n, m = case["problems"], case["n"], case["nev"]
        return {"bytes": p * (32.0 * n * n + 16.0 * n * n + 8 * m), "flops": p * (12.0 * n ** 3 + 12.0 * n * n * m + 8.0 * n * n * m)}
    io = 8 if case["precision"] == "fp32" else 16
    nk, nb = case["k1"] * case["k2"] * case["k3"], case["bands"]
    _, npw, _ = _geometry(case)
    n = float(npw.mean())
    if kind in ("hpsi", "host"):
        b, f = _operator_work(case, [case["lmax"]], nk * nb, io)
    elif kind == "items":
        b, f = _operator_work(case, [case["lmax"]], nk * nb / 2, io)
    elif kind == "multi":
        b, f = _operator_work(case, [case["lmax"], min(1, case["lmax"]), -1], nk * nb, io)
    elif kind == "davidson":
        # ten corrections of every band, each with H, its residual and its Gram columns over a
        # basis of 3 nb vectors, and the reduced eigenproblem of that size
        _, f1 = _operator_work(case, [case["lmax"]], nk * nb, io)
        m = 3 * nb
        f = 10 * (f1 + nk * nb * 32 * m * n + nk * (12.0 * m ** 3 + 12.0 * m * m * nb))
        b = nk * nb * n * 16 * 4
    elif kind == "sternheimer":
        # twenty conjugate-gradient steps of every pair: H and the valence projection
        _, f1 = _operator_work(case, [case["lmax"]], nk * nb, io)
        f = 20 * (f1 + nk * nb * 16 * nb * n)
        b = nk * nb * n * 16 * 3 + case["grid"] ** 3 * 16
    else:
        _, f1 = _operator_work(case, [-1], nk * nb, io)   # two half transform pairs
        f = f1 + nk * nb * (16 * nb * n + 8 * case["grid"] ** 3)
        b = nk * nb * n * 16 * 3 + case["grid"] ** 3 * 16
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------------------ correctness
def tolerance(case):
    """About four times the largest difference seen against `exact` over sixty draws of each kind:
    64-bit operators 3e-16, 32-bit ones 1.2e-7, densities 8e-16 and 2e-7, reduced eigenproblems
    1.5e-14.  The solvers stop at a residual: a Sternheimer solution at 1e-10 times the condition
    number of its system (2e-9 seen), the span of a Davidson's eigenvectors at 1e-7 over the gap
    above the last band (2e-5 where that gap is smallest)."""
    kind = case["kind"]
    if kind == "eigh":
        return {"rel": 6e-14}
    if kind == "davidson":
        return {"rel": 5e-5}
    if kind == "sternheimer":
        return {"rel": 8e-9}
    if kind == "drho":
        return {"rel": 4e-15 if case["precision"] == "fp64" else 1e-6}
    return {"rel": 1.5e-15 if case["precision"] == "fp64" else 5e-7}


def _to_grid(cell, x, ks, N):
    m = torch.from_numpy(cell["miller"][ks]).cuda().long() % N
    idx = (m[..., 0] * N + m[..., 1]) * N + m[..., 2]
    inside = torch.arange(m.shape[1], device="cuda")[None, :] < torch.from_numpy(cell["npw"][ks]).cuda()[:, None]
    idx = torch.where(inside, idx, torch.full_like(idx, N ** 3))          # padding to a spare point
    grid = torch.zeros(x.shape[0], x.shape[1], N ** 3 + 1, dtype=torch.complex128, device="cuda")
    grid.scatter_(2, idx[:, None, :].expand(-1, x.shape[1], -1), x)
    return idx, inside, torch.fft.ifftn(grid[..., :-1].reshape(*x.shape[:2], N, N, N), dim=(2, 3, 4), norm="forward")


def _apply(case, cell, x, q=False):
    """H x (or S x) in 64 bits, by full transforms, in blocks of k-points."""
    N, out = case["grid"], torch.zeros_like(x)
    step = max(1, 200_000_000 // (x.shape[1] * N ** 3))
    for k0 in range(0, x.shape[0], step):
        ks = np.arange(k0, min(x.shape[0], k0 + step))
        y = x[ks]
        if q:
            r = y.clone()
        else:
            idx, inside, u = _to_grid(cell, y, ks, N)
            v = torch.fft.fftn(u * cell["V"], dim=(2, 3, 4), norm="forward").reshape(*y.shape[:2], -1)
            v = torch.cat([v, torch.zeros_like(v[..., :1])], -1)
            r = v.gather(2, idx[:, None, :].expand(-1, y.shape[1], -1)) + (cell["g2"][ks] * inside)[:, None, :] * y
        if cell["beta"] is not None:
            b = cell["beta"][ks]
            c = torch.from_numpy(cell["q"] if q else cell["D"]).cuda().to(b.dtype)
            r = r + ((y @ b.mH) @ c) @ b
        out[ks] = r
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "eigh":
        H, S = _pencils(case, seed)
        lo = torch.linalg.cholesky(S)
        c = torch.linalg.solve_triangular(lo, torch.linalg.solve_triangular(lo, H, upper=False).mH, upper=False).mH
        w, v = torch.linalg.eigh(0.5 * (c + c.mH))
        v = torch.linalg.solve_triangular(lo.mH, v[..., :case["nev"]].contiguous(), upper=True)
        return [w[:, :case["nev"]], v @ v.mH]
    nb, N = case["bands"], case["grid"]
    wide = lambda x: x.to(torch.complex64).to(torch.complex128) if case["precision"] == "fp32" else x  # noqa: E731
    gen = _generator(seed)
    if kind == "multi":
        cells = _multi_cells(gen, case)
        xs = [wide(_vectors(gen, case, c["g2"], c["npw"], nb)) for c in cells]
        return [_apply(case, c, x) for c, x in zip(cells, xs)]
    if kind in ("hpsi", "host", "items"):
        cell = _cell(gen, case)
        x = wide(_vectors(gen, case, cell["g2"], cell["npw"], nb))
        h = _apply(case, cell, x)
        if kind != "items":
            return h if kind == "hpsi" else h.cpu()
        it = torch.from_numpy(_worklist(case, seed)).cuda().long()
        out = []
        for y in (h, _apply(case, cell, x, True)):
            z = torch.zeros_like(y)
            z[it[:, 0], it[:, 2]] = y[it[:, 0], it[:, 1]]
            out.append(z)
        return out
    if kind == "davidson":
        cell = _cell(gen, case)
        x = _vectors(gen, case, cell["g2"], cell["npw"], nb)
        if x.shape[0] * x.shape[2] ** 3 > 64 * 600 ** 3:
            return None
        vals, turned = [], []
        for k in range(x.shape[0]):
            w, v = np.linalg.eigh(_dense(case, cell, np.array([k]))[0].cpu().numpy())
            v = torch.from_numpy(np.ascontiguousarray(v[:, :nb])).cuda()
            vals.append(torch.from_numpy(w[:nb]).cuda())
            turned.append(((x[k] @ v.conj()) @ v.mT))
        return [torch.stack(vals), torch.stack(turned)]
    if kind == "sternheimer":
        cell, cell_q, u, uq, eps, alpha, dv = _response(case, seed)
        out = torch.zeros_like(uq)
        miller_q = torch.from_numpy(cell_q["miller"]).cuda().long() % N
        for k in range(u.shape[0]):
            ks = np.array([k])
            _, _, f = _to_grid(cell, u[ks], ks, N)
            g = torch.fft.fftn(f[0] * dv, dim=(1, 2, 3), norm="forward")
            m, n = miller_q[k], int(cell_q["npw"][k])
            w = g[:, m[:, 0], m[:, 1], m[:, 2]]
            w[:, n:] = 0
            b = -(w - (w @ uq[k].mH) @ uq[k])
            A = _dense(case, cell_q, ks) + alpha[k] * (uq[k].mT @ uq[k].conj())
            A = A - eps[k][:, None, None] * torch.eye(A.shape[-1], device="cuda", dtype=A.dtype)
            out[k] = torch.linalg.solve(A, b[:, :, None])[..., 0]
        return out
    cell, cell_q, u, uq, du, w = _density_inputs(case, seed)
    du = du - (du @ uq.mH) @ uq
    total = torch.zeros(N, N, N, dtype=torch.complex128, device="cuda")
    for k in range(u.shape[0]):
        ks = np.array([k])
        a, b = _to_grid(cell, u[ks], ks, N)[2], _to_grid(cell_q, du[ks], ks, N)[2]
        total += 4 * w[k] * (a.conj() * b).sum((0, 1))
    return total
