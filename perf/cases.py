"""Workloads of the density-matrix library, measured through its Python entry points.

Every case is one whole call (or the few calls that belong together) as a program makes them:
colouring and probe signs of a geometry, a density-matrix build from geometry and Hamiltonian, a
batch of systems, the non-orthogonal pair of calls.  The systems are water-like boxes at the
density of 64 molecules in a 12.42 A cube, generated on the GPU from the seed: molecules on a
jittered lattice, on-site blocks with the levels of a minimal (b = 6) or polarised double-zeta
(b = 23) basis under a random orthogonal matrix, couplings that decay with distance up to about 6 A.

`exact` restates the method in 64-bit torch: greedy colours, probe blocks, block-Lanczos with
Householder QR, dense diagonalisation of the projected matrices, the chemical-potential rule and
the extraction on the pattern.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_20918_gb300 as css

KT = 0.05
COLOUR_SEED, SIGN_SEED = 1004, 1005
DENSITY = 64.0 / 12.42 ** 3  # molecules per cubic Angstrom
PRECISION = {"fp64": css.CSS_FP64, "mixed": css.CSS_MIXED_FP32, "split": css.CSS_FP64_SPLIT}
_context = None


def listed():
    return [
        # colouring + probe signs of one MD geometry, as each step of a trajectory starts
        {"name": "colour_20000", "kind": "colour", "n": 20000, "b": 6, "r_col": 10.0},
        # the smallest reference build: a 64-molecule box, all FP64; latency and launches
        {"name": "fp64_b6_64", "kind": "build", "n": 64, "b": 6, "r_col": 8.0, "m": 30, "precision": "fp64"},
        # small and middling single systems in the minimal basis, the usual MD snapshot
        {"name": "mixed_b6_512", "kind": "build", "n": 512, "b": 6, "r_col": 10.0, "m": 30, "precision": "mixed"},
        {"name": "mixed_b6_4001", "kind": "build", "n": 4001, "b": 6, "r_col": 10.0, "m": 30, "precision": "mixed"},
        # serving: snapshots of uneven size in one call
        {"name": "batch_b6_8", "kind": "batch", "n": 207, "n_max": 2011, "systems": 8, "b": 6, "r_col": 10.0, "m": 30,
         "precision": "mixed"},
        # reference-quality builds in the polarised basis: FP64, and FP64-accurate H*V in FP32 pairs
        {"name": "fp64_b23_128", "kind": "build", "n": 128, "b": 23, "r_col": 10.0, "m": 40, "precision": "fp64"},
        {"name": "split_b23_256", "kind": "build", "n": 256, "b": 23, "r_col": 10.0, "m": 40, "precision": "split"},
        # production builds in the polarised basis, up to the 10,000-molecule headline system
        {"name": "mixed_b23_1000", "kind": "build", "n": 1000, "b": 23, "r_col": 10.0, "m": 40, "precision": "mixed"},
        {"name": "mixed_b23_10000", "kind": "build", "n": 10000, "b": 23, "r_col": 10.0, "m": 40,
         "precision": "mixed"},
        # large systems whose Krylov rows are regenerated instead of stored (the million-molecule mode)
        {"name": "two_pass_b6_60000", "kind": "build", "n": 60000, "b": 6, "r_col": 10.0, "m": 30,
         "precision": "mixed", "two_pass": True},
        # a non-orthogonal basis: S^(-1/2) and H', then its density matrix
        {"name": "nonorth_b6_700", "kind": "nonorth", "n": 700, "b": 6, "r_col": 10.0, "m": 30, "m_s": 10,
         "precision": "mixed"},
        # the energy-weighted matrix of a force evaluation at a given mu, another block width
        {"name": "weighted_b13_343", "kind": "weighted", "n": 343, "b": 13, "r_col": 9.0, "m": 30,
         "precision": "mixed"},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["colour", "build6", "build6", "build23", "build23", "reference6", "reference23", "split",
                       "two_pass", "batch", "nonorth", "weighted"])
    r_col = rng.choice([8.0, 9.0, 10.0])
    if kind == "colour":
        return {"kind": "colour", "n": size(64, 60000), "b": rng.choice([6, 23]), "r_col": r_col}
    if kind == "build6":
        return {"kind": "build", "n": size(64, 20000), "b": 6, "r_col": r_col, "m": rng.randint(20, 30),
                "precision": "mixed"}
    if kind == "build23":
        return {"kind": "build", "n": size(64, 7000), "b": 23, "r_col": r_col, "m": rng.randint(24, 40),
                "precision": "mixed"}
    if kind == "reference6":
        return {"kind": "build", "n": size(48, 1500), "b": 6, "r_col": r_col, "m": rng.randint(20, 30),
                "precision": "fp64"}
    if kind == "reference23":
        return {"kind": "build", "n": size(48, 200), "b": 23, "r_col": r_col, "m": rng.randint(20, 40),
                "precision": "fp64"}
    if kind == "split":
        b = rng.choice([6, 23])
        return {"kind": "build", "n": size(64, 400 if b == 23 else 2000), "b": b, "r_col": r_col,
                "m": rng.randint(20, 40 if b == 23 else 30), "precision": "split"}
    if kind == "two_pass":
        return {"kind": "build", "n": size(4000, 60000), "b": 6, "r_col": r_col, "m": rng.randint(20, 30),
                "precision": "mixed", "two_pass": True}
    if kind == "batch":
        n = size(100, 400)
        return {"kind": "batch", "n": n, "n_max": size(3 * n, 3000), "systems": rng.randint(3, 10), "b": 6,
                "r_col": r_col, "m": rng.randint(20, 30), "precision": rng.choice(["mixed", "mixed", "fp64"])}
    if kind == "nonorth":
        return {"kind": "nonorth", "n": size(64, 1200), "b": 6, "r_col": r_col, "m": rng.randint(20, 30), "m_s": 10,
                "precision": rng.choice(["mixed", "fp64"])}
    return {"kind": "weighted", "n": size(64, 700), "b": rng.randint(4, 30), "r_col": r_col, "m": rng.randint(20, 30),
            "precision": rng.choice(["mixed", "fp64"])}


# ------------------------------------------------------------------ inputs
def _positions(n, rng):
    """Jittered simple-cubic lattice in a periodic cube (host float64 [n, 3], box side)."""
    box = (n / DENSITY) ** (1.0 / 3.0)
    n_s = 1
    while n_s ** 3 < n:
        n_s += 1
    sites = np.sort(rng.permutation(n_s ** 3)[:n])
    ijk = np.stack([sites // (n_s * n_s), (sites // n_s) % n_s, sites % n_s], axis=1)
    return (ijk + 0.5) * (box / n_s) + rng.uniform(-0.4, 0.4, (n, 3)), box


def _pairs(pos, box):
    """The 13.5 n closest pairs i < j (i, j, distance), by distance: about 6 A at this density.  A fixed
    number of pairs instead of a fixed cut-off gives every geometry of n molecules the same block count."""
    n = pos.shape[0]
    chunk = max(1, 40_000_000 // n)
    out_i, out_j, out_d = [], [], []
    for s in range(0, n, chunk):
        d2 = torch.zeros((min(chunk, n - s), n), dtype=torch.float64, device=pos.device)
        for x in range(3):
            d = pos[s:s + chunk, None, x] - pos[None, :, x]
            d -= box * torch.round(d / box)
            d2 += d * d
        i, j = torch.nonzero(d2 <= 7.2 * 7.2, as_tuple=True)
        out_d.append(d2[i, j])
        out_i.append(i + s)
        out_j.append(j)
    i, j, d2 = torch.cat(out_i), torch.cat(out_j), torch.cat(out_d)
    i, j, d2 = i[i < j], j[i < j], d2[i < j]
    d2, order = torch.sort(d2, stable=True)
    keep = (27 * n) // 2
    return i[order[:keep]], j[order[:keep]], torch.sqrt(d2[:keep])


def _levels(n, b, gen):
    """On-site spectra [n, b] in eV and the number of occupied levels."""
    dev = gen.device
    if b == 6:
        return torch.tensor([-20.0, -15.0, -13.0, -11.0, 2.0, 5.0], dtype=torch.float64, device=dev).expand(n, 6), 4
    occ = 4 if b > 6 else max(1, b // 2)
    u = torch.rand((n, b), generator=gen, dtype=torch.float64, device=dev)
    return torch.cat([-25.0 + 15.0 * u[:, :occ], 2.0 + 28.0 * u[:, occ:]], dim=1), occ


def _matrix(n, b, pairs, onsite, coupling, gen):
    """Symmetric BSR matrix: the given on-site blocks, coupling * exp(-(r - 2.8)/0.5) * N(0,1)/sqrt(b) on the
    pairs (no closer than water molecules come)."""
    i, j, r = pairs
    dev = i.device
    g = torch.randn((i.numel(), b, b), generator=gen, dtype=torch.float64, device=dev)
    g *= (coupling / math.sqrt(b)) * torch.exp(-(r.clamp(min=2.5) - 2.8) / 0.5)[:, None, None]
    k = torch.arange(n, device=dev)
    row, col = torch.cat([i, j, k]), torch.cat([j, i, k])
    order = torch.argsort(row * n + col)
    val = torch.cat([g, g.transpose(1, 2), onsite])[order].contiguous()
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return css.DeviceBSR(n, b, row_ptr.to(torch.int32), col[order].to(torch.int32), val)


def _system(n, b, seed, overlap=False):
    """Geometry, Hamiltonian and (for a non-orthogonal basis) overlap of one box."""
    rng = np.random.RandomState(seed % (1 << 32))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    host, box = _positions(n, rng)
    pos = torch.as_tensor(host, device="cuda")
    lv, occ = _levels(n, b, gen)
    u = torch.eye(b, dtype=torch.float64, device="cuda").expand(n, b, b)
    for _ in range(4):  # a random orthogonal matrix per molecule, as a product of reflections
        v = torch.randn((n, b, 1), generator=gen, dtype=torch.float64, device="cuda")
        v = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
        u = u - 2.0 * (u @ v) @ v.transpose(1, 2)
    onsite = (u * lv[:, None, :]) @ u.transpose(1, 2)
    onsite = 0.5 * (onsite + onsite.transpose(1, 2))
    pairs = _pairs(pos, box)
    s = {"n": n, "b": b, "pos": pos, "box": box, "n_elec": 2.0 * occ * n,
         "H": _matrix(n, b, pairs, onsite, 0.5, gen)}
    if overlap:  # the 6 n closest pairs, about 4.5 A
        unit = torch.eye(b, dtype=torch.float64, device="cuda").expand(n, b, b)
        s["S"] = _matrix(n, b, [x[:6 * n] for x in pairs], unit, 0.05, gen)
    return s


def _sizes(case):
    """Molecule counts of a batch: spread evenly in the logarithm from n to n_max."""
    k = case["systems"]
    f = math.log(case["n_max"] / case["n"])
    return [int(round(case["n"] * math.exp(f * i / (k - 1)))) for i in range(k)]


def _systems(case, seed):
    sizes = _sizes(case) if case["kind"] == "batch" else [case["n"]]
    return [_system(n, case["b"], seed * 16 + i, overlap=case["kind"] == "nonorth") for i, n in enumerate(sizes)]


def _flags(case):
    if case["kind"] == "weighted":  # forces take the matrix as extracted
        return css.CSS_ENERGY_WEIGHTED
    return css.CSS_SYMMETRIZE | (css.CSS_TWO_PASS if case.get("two_pass") else 0)


def _handle():
    """One context for the whole process, as a program keeps it: its workspace is reused."""
    global _context
    if _context is None:
        _context = css.Context(0)
    return _context


def prepare(case, seed):
    if case["kind"] == "colour":
        pos, box = _positions(case["n"], np.random.RandomState(seed % (1 << 32)))
        systems = [{"n": case["n"], "b": case["b"], "pos": torch.as_tensor(pos, device="cuda"), "box": box}]
    else:
        systems = _systems(case, seed)
    for s in systems:
        s["colour"] = torch.empty(s["n"], dtype=torch.int32, device="cuda")
        s["sign"] = torch.empty(s["n"] * s["b"], dtype=torch.int8, device="cuda")
        if "H" in s:
            s["P"] = torch.empty_like(s["H"].val)
        if "S" in s:
            s["Sinv"], s["Hp"] = torch.empty_like(s["S"].val), torch.empty_like(s["H"].val)
    # probe signs follow the seed, so that the colouring path too has other outputs for other inputs
    return {"case": dict(case), "systems": systems, "ctx": _handle(), "sign_seed": SIGN_SEED + seed}


# --------------------------------------------------------------------- run
def _kept(case, *blocks, scalars):
    """The call's results.  The mixed modes carry their matrices to single precision (Krylov vectors
    and block products are FP32), so a program that picks them keeps FP32; FP64 modes keep doubles."""
    dt = torch.float32 if case["precision"] == "mixed" else torch.float64
    return [x.to(dt) for x in blocks] + [torch.tensor(scalars, dtype=dt)]


def run(state):
    case, ctx = state["case"], state["ctx"]
    seed = state["sign_seed"]
    if case["kind"] == "build":
        s = state["systems"][0]
        r = ctx.pbuild(s["pos"], s["box"], s["H"], s["P"], r_col=case["r_col"], colour_seed=COLOUR_SEED,
                       sign_seed=seed, kT=KT, n_elec=s["n_elec"], m=case["m"], precision=PRECISION[case["precision"]],
                       flags=_flags(case), colour_out=s["colour"])
        return {"colour": s["colour"], "result": _kept(case, s["P"], scalars=[r["trP"], r["trPH"], r["mu"]])}
    for s in state["systems"]:
        s["n_colours"] = ctx.color(s["pos"], s["box"], case["r_col"], COLOUR_SEED, s["colour"])
        ctx.probes(s["colour"], s["b"], seed, s["sign"])
    s = state["systems"][0]
    if case["kind"] == "colour":
        return {"colour": s["colour"], "sign": s["sign"], "n_colours": s["n_colours"]}
    if case["kind"] == "batch":
        sy = state["systems"]
        r = ctx.density_batch([s["H"] for s in sy], [s["colour"] for s in sy], [s["sign"] for s in sy],
                              [s["n_colours"] for s in sy], [s["P"] for s in sy],
                              [{"kT": KT, "n_elec": s["n_elec"], "solve_mu": True} for s in sy], m=case["m"],
                              precision=PRECISION[case["precision"]], flags=_flags(case))
        return {"systems": [{"colour": s["colour"],
                             "result": _kept(case, s["P"], scalars=[r["trP"][i], r["trPH"][i], r["mu"][i]])}
                            for i, s in enumerate(sy)]}
    if case["kind"] == "weighted":
        r = ctx.density(s["H"], s["colour"], s["sign"], s["n_colours"], s["P"], mu=-4.0, kT=KT, solve_mu=False,
                        m=case["m"], precision=PRECISION[case["precision"]], flags=_flags(case))
        return {"colour": s["colour"], "result": _kept(case, s["P"], scalars=[r["trP"], r["trPH"]])}
    H = s["H"]
    h = ctx.hprime(s["S"], H, s["colour"], s["sign"], s["n_colours"], s["Sinv"], s["Hp"], m=case["m_s"],
                   precision=PRECISION[case["precision"]])
    Hp = css.DeviceBSR(H.n_brow, H.b, H.row_ptr, H.col_idx, s["Hp"])
    r = ctx.density_nonorth(s["S"], s["Sinv"], Hp, H.val, s["colour"], s["sign"], s["n_colours"], s["P"], kT=KT,
                            n_elec=s["n_elec"], m=case["m"], precision=PRECISION[case["precision"]])
    return {"colour": s["colour"], "result": _kept(case, s["Sinv"], s["Hp"], s["P"],
                                                   scalars=[h["trHp"], r["trPS"], r["trPH"], r["mu"]])}


# -------------------------------------------------------------------- work
def _counts(n, r_col):
    """Blocks of H and expected colours of a box of n molecules."""
    blocks = n + 2 * ((27 * n) // 2)
    colours = min(n, 0.47 * DENSITY * 4.0 / 3.0 * math.pi * r_col ** 3)
    return blocks, colours


def work(case):
    """Bytes: inputs read and outputs written once.  Flops: the products H*V of the recurrence, and per
    step the projections on two blocks, the two updates, the Gram and the triangular solve."""
    if case["kind"] == "colour":
        return {"bytes": case["n"] * (24.0 + 4.0 + case["b"]), "flops": 0.0}
    nbytes = flops = 0.0
    for n in _sizes(case) if case["kind"] == "batch" else [case["n"]]:
        b, m = case["b"], case["m"]
        blocks, colours = _counts(n, case["r_col"])
        width = colours * b
        passes = 2 if case.get("two_pass") else 1
        nbytes += 24.0 * n + 2 * 8.0 * blocks * b * b
        flops += passes * m * 2.0 * width * (blocks * b * b + n * b * b * 5.0)
        if case["kind"] == "nonorth":
            nbytes += 2 * 8.0 * blocks * b * b
            flops += 2 * (m + case["m_s"]) * 2.0 * width * blocks * b * b
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact
def _splitmix(seed, x):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.asarray(x, np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _greedy(pos, box, r_col):
    """Greedy colours by (degree, hash, -id) descending; neighbours strictly inside r_col in 2^-20 A units."""
    n = pos.shape[0]
    q = torch.round(pos * 1048576.0).to(torch.int64)
    side, rad = int(np.rint(box * 1048576.0)), int(np.rint(r_col * 1048576.0))
    chunk = max(1, 20_000_000 // n)
    ni, nj = [], []
    for s in range(0, n, chunk):
        d2 = torch.zeros((min(chunk, n - s), n), dtype=torch.int64, device=pos.device)
        for x in range(3):
            d = torch.remainder(q[s:s + chunk, None, x] - q[None, :, x], side)
            d = torch.where(d > side // 2, d - side, d)
            d2 += d * d
        i, j = torch.nonzero(d2 < rad * rad, as_tuple=True)
        ni.append((i + s)[i + s != j])
        nj.append(j[i + s != j])
    i, j = torch.cat(ni).cpu().numpy(), torch.cat(nj).cpu().numpy()
    degree = np.bincount(i, minlength=n)
    start = np.concatenate([[0], np.cumsum(degree)])
    ids = np.arange(n)
    order = np.lexsort((ids, ~_splitmix(COLOUR_SEED, ids), -degree))
    colour = np.full(n, -1, np.int64)
    for v in order:
        used = set(colour[j[start[v]:start[v + 1]]].tolist())
        c = 0
        while c in used:
            c += 1
        colour[v] = c
    return torch.as_tensor(colour, device=pos.device), int(colour.max()) + 1


def _sparse(M, val=None):
    """A BSR matrix as a 64-bit CSR one."""
    n, b = M.n_brow, M.b
    val = M.val if val is None else val
    ptr = M.row_ptr.to(torch.int64)
    brow = torch.repeat_interleave(torch.arange(n, device=ptr.device), ptr[1:] - ptr[:-1])
    k = torch.arange(b, device=ptr.device)
    rows = (brow[:, None, None] * b + k[None, :, None]).expand(-1, b, b).reshape(-1)
    cols = (M.col_idx.to(torch.int64)[:, None, None] * b + k[None, None, :]).expand(-1, b, b).reshape(-1)
    order = torch.argsort(rows * (n * b) + cols)
    crow = torch.zeros(n * b + 1, dtype=torch.int64, device=ptr.device)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=n * b), 0)
    return torch.sparse_csr_tensor(crow, cols[order], val.reshape(-1)[order], size=(n * b, n * b))


def _blocks(V, nc, b):
    return V.reshape(V.shape[0], nc, b).transpose(0, 1)  # [colour, N, b]


def _lanczos(A, start, nc, b, m):
    """Krylov blocks Q [m, colour, N, b], projected matrices T [colour, mb, mb] and start factors B0."""
    N = start.shape[0]
    Q = torch.empty((m, nc, N, b), dtype=torch.float64, device=start.device)
    T = torch.zeros((nc, m * b, m * b), dtype=torch.float64, device=start.device)
    q, B0 = torch.linalg.qr(_blocks(start, nc, b))
    Q[0] = q
    B = None
    for j in range(m):
        W = _blocks(torch.sparse.mm(A, Q[j].transpose(0, 1).reshape(N, nc * b)), nc, b)
        if j > 0:
            W = W - Q[j - 1] @ B.transpose(1, 2)
        a = Q[j].transpose(1, 2) @ W
        T[:, j * b:(j + 1) * b, j * b:(j + 1) * b] = 0.5 * (a + a.transpose(1, 2))
        if j + 1 == m:
            break
        W = W - Q[j] @ a
        for i in (j, j - 1):
            if i >= 0:
                W = W - Q[i] @ (Q[i].transpose(1, 2) @ W)
        Q[j + 1], B = torch.linalg.qr(W)
        T[:, (j + 1) * b:(j + 2) * b, j * b:(j + 1) * b] = B
        T[:, j * b:(j + 1) * b, (j + 1) * b:(j + 2) * b] = B.transpose(1, 2)
    return Q, T, B0


def _fermi(x, mu):
    return 0.5 * (1.0 - torch.tanh((x - mu) / (2.0 * KT)))


def _chemical_potential(lam, weight, n_elec):
    """Midpoint of {mu : |N(mu) - n_elec/2| <= 1e-4 n_elec/2}, each end by bisection."""
    target, tol, ends = 0.5 * n_elec, 1e-4 * max(1.0, 0.5 * n_elec), []
    for lower in (True, False):
        lo, hi = float(lam.min()) - 1.0, float(lam.max()) + 1.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            g = float((_fermi(lam, mid) * weight).sum()) - target
            if (g >= -tol) if lower else (g > tol):
                hi = mid
            else:
                lo = mid
            if hi - lo <= 1e-13 * max(1.0, abs(mid)):
                break
        ends.append(0.5 * (lo + hi))
    return 0.5 * (ends[0] + ends[1])


def _probe_block(s, colour, nc, sign):
    n, b = s["n"], s["b"]
    row = torch.arange(n * b, device=colour.device)
    R = torch.zeros((n * b, nc * b), dtype=torch.float64, device=colour.device)
    R[row, colour[row // b] * b + row % b] = sign
    return R


def _extract(M, X, colour, sign, symmetric):
    """Blocks X[I, colour(J)] diag(sign_J) on M's pattern, optionally averaged with the transpose."""
    n, b = M.n_brow, M.b
    ptr = M.row_ptr.to(torch.int64)
    i = torch.repeat_interleave(torch.arange(n, device=ptr.device), ptr[1:] - ptr[:-1])
    j = M.col_idx.to(torch.int64)
    X4 = X.reshape(n, b, -1, b)
    out = X4[i, :, colour[j], :] * sign.reshape(n, 1, b)[j]
    if symmetric:
        out = 0.5 * (out + out[torch.searchsorted(i * n + j, j * n + i)].transpose(1, 2))
    diag = torch.nonzero(i == j).flatten()
    return out, float(out[diag].diagonal(dim1=1, dim2=2).sum())


def _combine(Q, Z, nc, b):
    """X = sum_j Q_j Z_j as N x (nc b)."""
    m, _, N, _ = Q.shape
    X = torch.zeros((nc, N, b), dtype=torch.float64, device=Q.device)
    for j in range(m):
        X += Q[j] @ Z[:, j * b:(j + 1) * b]
    return X.transpose(0, 1).reshape(N, nc * b)


def _exact_system(case, s, sign_seed):
    b, n = s["b"], s["n"]
    colour, nc = _greedy(s["pos"], s["box"], case["r_col"])
    bit = (_splitmix(sign_seed, np.arange(n * b)) & np.uint64(1)).astype(np.float64)
    sign = torch.as_tensor(1.0 - 2.0 * bit, device=colour.device)
    R = _probe_block(s, colour, nc, sign)
    H, symmetric = s["H"], bool(_flags(case) & css.CSS_SYMMETRIZE)
    out = {"colour": None}
    if case["kind"] == "nonorth":
        S = s["S"]
        Q, T, B0 = _lanczos(_sparse(S), R, nc, b, case["m_s"])
        lam, U = torch.linalg.eigh(T)
        Z = (U * lam[:, None, :] ** -0.5) @ (U[:, :b].transpose(1, 2) @ B0)
        Y = _combine(Q, Z, nc, b)
        Sinv, _ = _extract(S, Y, colour, sign, True)
        Si = _sparse(S, Sinv)
        Hp, trHp = _extract(H, torch.sparse.mm(Si, torch.sparse.mm(_sparse(H), Y)), colour, sign, True)
        Q, T, B0 = _lanczos(_sparse(H, Hp), torch.sparse.mm(Si, R), nc, b, case["m"])
        u = _blocks(torch.sparse.mm(Si, torch.sparse.mm(_sparse(S), R)), nc, b)  # Si is symmetric
        V = torch.cat([q.transpose(1, 2) @ u for q in Q], dim=1)
        lam, U = torch.linalg.eigh(T)
        Yk = U[:, :b].transpose(1, 2) @ B0
        mu = _chemical_potential(lam, ((U.transpose(1, 2) @ V) * Yk).sum(2), s["n_elec"])
        Z = (U * _fermi(lam, mu)[:, None, :]) @ Yk
        P, _ = _extract(H, torch.sparse.mm(Si, _combine(Q, Z, nc, b)), colour, sign, True)
        trPS = float((torch.sparse.mm(_sparse(S), torch.eye(n * b, dtype=torch.float64, device=P.device))
                      * _sparse(H, P).to_dense()).sum())
        out["result"] = [Sinv, Hp, P, torch.tensor([trHp, trPS, float((P * H.val).sum()), mu], dtype=torch.float64)]
        return out
    Q, T, B0 = _lanczos(_sparse(H), R, nc, b, case["m"])
    lam, U = torch.linalg.eigh(T)
    Yk = U[:, :b].transpose(1, 2) @ B0
    weighted = case["kind"] == "weighted"
    mu = -4.0 if weighted else _chemical_potential(lam, (Yk * Yk).sum(2), s["n_elec"])
    f = _fermi(lam, mu) * (lam if weighted else 1.0)
    P, trP = _extract(H, _combine(Q, (U * f[:, None, :]) @ Yk, nc, b), colour, sign, symmetric)
    scalars = [trP, float((P * H.val).sum())] + ([] if weighted else [mu])
    out["result"] = [P, torch.tensor(scalars, dtype=torch.float64)]
    return out


def exact(case, seed):
    if case["kind"] == "colour":
        return None  # whole numbers only
    if case["kind"] == "nonorth" and case["n"] > 1500:
        return None
    # the 64-bit restatement of the largest systems takes minutes
    if work(case)["flops"] > 5e12:
        return None
    systems = [_exact_system(case, s, SIGN_SEED + seed) for s in _systems(case, seed)]
    return {"systems": systems} if case["kind"] == "batch" else systems[0]
