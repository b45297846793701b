"""Performance cases of the VBARMS library: what a user's program has it do.

Every case is a pass through the public entry points
(``paper_1508_02219_gb300.vbarms``) on a seeded synthetic matrix of the shapes
that ``paper_1508_02219_gb300.synth`` configures: block Jacobians of a 3-D mesh
(a random geometric node graph with about 15 neighbours, or a 7-point grid)
with ``ell`` unknowns per node.  The matrices are drawn here on the GPU, so
that the largest takes about a second to make.

Kinds of pass (``case["kind"]``):

  whole     Step 1, factorization and FGMRES from a CSR matrix in host memory
  compress  Step 1 on a CSR matrix in device memory; the permutation, the block
            sizes, and one step of GMRES without a preconditioner, which takes
            the block matrix's values to the output
  factor    factorization of a compressed matrix and one application of it
  batch     the same for several matrices at once
  ras       restricted additive Schwarz with local factorizations, and FGMRES
  apply     one application of a factorization that the program keeps
  fgmres    FGMRES with a factorization that the program keeps
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1508_02219_gb300 import vbarms as V

_DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
def _case(kind, nodes, ell, **kw):
    c = dict(kind=kind, gen="geo", nodes=int(nodes), ell=int(ell), tau=0.8, dominance=0.0, ill_frac=0.0,
             precision="fp32", nlev=4, droptol=1e-4, lfil=30, group_size=1)
    c.update(kw)
    return c


def listed():
    jac = dict(dominance=1.5, ill_frac=1e-3)  # dominant pivot blocks, 0.1 % of them ill-conditioned
    fp64 = dict(precision="fp64", nlev=3, lfil=-1)
    return [
        # the smallest call: 5 000 unknowns on a 10 x 10 x 10 grid, one linear system of a small model problem;
        # launches, synchronisations and allocations are what it costs
        dict(_case("whole", 1000, 5, gen="grid", tau=1.0, precision="fp64", nlev=2, droptol=1e-3, lfil=20),
             name="whole_grid_5k_fp64"),
        # an ordinary linear system handed over in host memory: 60 000 unknowns, mixed factor
        dict(_case("whole", 10_000, 6), name="whole_geo_60k_fp32"),
        # Step 1 on a Jacobian that is already on the device: 360 000 unknowns, approximate blocks
        dict(_case("compress", 60_000, 6), name="compress_geo_360k"),
        # the FP64 factor at the size of the configured FP64 workload, no bound on the blocks kept per row
        dict(_case("factor", 60_000, 6, **fp64), name="factor_geo_360k_fp64"),
        # the largest: the mixed factor of the configured precision workload, 3.0 million unknowns
        dict(_case("factor", 500_000, 6, **jac), name="factor_geo_3m_fp32"),
        # tau = 0.9 splits the node blocks into small ones: a last level of wide rows, tight dropping
        dict(_case("factor", 8_009, 6, tau=0.9, nlev=5, droptol=1e-5, lfil=40), name="factor_tau09_48k_fp32"),
        # Step 3 with groups of four supernodes: few rows reach the last level
        dict(_case("factor", 60_013, 5, group_size=4, **jac), name="factor_groups_300k_fp32"),
        # many independent systems at once (a batch of Jacobians of uneven sizes and unknowns per node)
        dict(_case("batch", 3_000, 0, count=24, ratio=8.0), name="batch_24_fp32"),
        # Section 5: 16 overlapping subdomains on one GPU, set up and solved
        dict(_case("ras", 60_000, 6, nparts=16, overlap=2, **jac), name="ras_360k_fp32"),
        # one application on a small factorization: a smoother or an inner solver that calls it again and again
        dict(_case("apply", 3_001, 6, **fp64), name="apply_geo_18k_fp64"),
        # one application at the largest size: the cost of one outer iteration of any Krylov method
        dict(_case("apply", 500_000, 6, **jac), name="apply_geo_3m_fp32"),
        # the linear solves of a time step: the factorization kept, a new right-hand side
        dict(_case("fgmres", 120_000, 6, **jac), name="fgmres_geo_720k_fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "compress", "factor", "factor", "tau09", "batch", "ras", "apply", "apply", "fgmres"])
    ell = rng.choice([4, 5, 6])
    prec = rng.choice(["fp64", "fp32", "fp32"])
    jac = dict(dominance=1.5, ill_frac=1e-3) if rng.random() < 0.5 else {}
    par = dict(precision=prec, nlev=rng.choice([2, 3, 4]), droptol=rng.choice([1e-3, 3e-4, 1e-4]),
               lfil=rng.choice([20, 30, -1]), **jac)
    if kind == "whole":
        if rng.random() < 0.3:
            side = rng.randint(6, 16)
            return _case("whole", side ** 3, ell, gen="grid", **{**par, "tau": 1.0, "dominance": 0.0, "ill_frac": 0.0})
        return _case("whole", _log(rng, 500, 20_000), ell, **par)
    if kind == "compress":
        return _case("compress", _log(rng, 2_000, 150_000), ell, tau=rng.choice([0.75, 0.8, 0.9]))
    if kind == "factor":
        return _case("factor", _log(rng, 2_000, 50_000 if prec == "fp64" else 250_000), ell,
                     group_size=rng.choice([1, 1, 2, 4, 8]), **par)
    if kind == "tau09":
        return _case("factor", _log(rng, 800, 8_000), ell, tau=0.9, nlev=5, droptol=1e-5, lfil=40, precision=prec)
    if kind == "batch":
        return _case("batch", _log(rng, 300, 3_000), 0, count=rng.randint(3, 32), ratio=rng.choice([2.0, 8.0]), **par)
    if kind == "ras":
        return _case("ras", _log(rng, 6_000, 80_000), ell, nparts=rng.randint(3, 48), overlap=rng.choice([1, 2]),
                     **{**par, "lfil": 30, "droptol": 1e-4, "dominance": 1.5, "ill_frac": 1e-3})
    if kind == "apply":
        return _case("apply", _log(rng, 500, 40_000 if prec == "fp64" else 250_000), ell, **par)
    return _case("fgmres", _log(rng, 2_000, 30_000 if prec == "fp64" else 120_000), ell, **par)


# ---------------------------------------------------------------------------
# matrices (torch on the GPU; the recipe of synth.geometric / synth.grid_7pt)
def _morton(pts):
    q = (pts * 1024).long().clamp_(max=1023)

    def spread(v):
        v = (v | (v << 16)) & 0x030000FF
        v = (v | (v << 8)) & 0x0300F00F
        v = (v | (v << 4)) & 0x030C30C3
        return (v | (v << 2)) & 0x09249249

    return spread(q[:, 0]) | (spread(q[:, 1]) << 1) | (spread(q[:, 2]) << 2)


def _torus_pairs(pts, r):
    """Index pairs (i, j), i != j included both ways, and i = j, closer than r on the torus."""
    n = pts.shape[0]
    if n <= 4096:
        d = (pts[:, None, :] - pts[None, :, :]).abs_()
        d = torch.minimum(d, 1.0 - d)
        return torch.nonzero((d * d).sum(2) < r * r, as_tuple=True)
    nc = max(3, int(1.0 / r))
    cell = (pts * nc).long().clamp_(max=nc - 1)
    key = (cell[:, 2] * nc + cell[:, 1]) * nc + cell[:, 0]
    skey, srt = torch.sort(key, stable=True)
    start = torch.searchsorted(skey, torch.arange(nc ** 3 + 1, device=pts.device))
    most = int((start[1:] - start[:-1]).max())
    k = torch.arange(most, device=pts.device)
    out_i, out_j = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                o = (cell + torch.tensor([dx, dy, dz], device=pts.device)) % nc
                c = (o[:, 2] * nc + o[:, 1]) * nc + o[:, 0]
                at = start[c][:, None] + k
                j = srt[at.clamp(max=n - 1)]
                d = (pts[:, None, :] - pts[j]).abs_()
                d = torch.minimum(d, 1.0 - d)
                ok = (at < start[c + 1][:, None]) & ((d * d).sum(2) < r * r)
                i, q = torch.nonzero(ok, as_tuple=True)
                out_i.append(i)
                out_j.append(j[i, q])
    return torch.cat(out_i), torch.cat(out_j)


def _grid_pairs(side):
    idx = torch.arange(side ** 3, device=_DEV).reshape(side, side, side)
    lo = [idx[:-1], idx[:, :-1], idx[:, :, :-1]]
    hi = [idx[1:], idx[:, 1:], idx[:, :, 1:]]
    a = torch.cat([x.reshape(-1) for x in lo])
    b = torch.cat([x.reshape(-1) for x in hi])
    d = idx.reshape(-1)
    return torch.cat([a, b, d]), torch.cat([b, a, d])


def _orthogonal(n, m, g):
    """Random orthogonal m x m matrices: products of m random reflections."""
    q = torch.eye(m, dtype=torch.float64, device=_DEV).expand(n, m, m).contiguous()
    for _ in range(m):
        v = torch.randn(n, m, 1, dtype=torch.float64, device=_DEV, generator=g)
        q = q - 2.0 * (q @ v) @ v.transpose(1, 2) / (v * v).sum(1, keepdim=True)
    return q


def _matrix(gen, nodes, ell, dominance, ill_frac, seed):
    """(n, rowptr int64, colind int32, val float64) on the GPU, columns ascending."""
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed))
    f64 = dict(dtype=torch.float64, device=_DEV)
    if gen == "grid":
        i, j = _grid_pairs(round(nodes ** (1.0 / 3.0)))
    else:
        pts = torch.rand(nodes, 3, generator=g, **f64)
        pts = pts[torch.sort(_morton(pts), stable=True)[1]]
        i, j = _torus_pairs(pts, min(0.4999, (45.0 / (4.0 * math.pi * nodes)) ** (1.0 / 3.0)))
    pair = torch.sort(i * nodes + j)[0]
    i, j = pair // nodes, pair % nodes
    nblk = pair.numel()
    deg = torch.bincount(i, minlength=nodes)
    nptr = torch.cat([deg.new_zeros(1), deg.cumsum(0)])
    diag = torch.nonzero(i == j)[:, 0]
    blocks = torch.randn(nblk, ell, ell, generator=g, **f64) * 0.1
    eye = torch.eye(ell, **f64)
    blocks[diag] = torch.randn(nodes, ell, ell, generator=g, **f64) + 8.0 * eye
    keep = torch.ones(nblk, ell, ell, dtype=torch.bool, device=_DEV)
    if gen != "grid":  # approximate blocks: a tenth of the entries missing, noise on the others
        keep = torch.rand(nblk, ell, ell, generator=g, device=_DEV) >= 0.1
        keep[diag] |= eye.bool()
        blocks += torch.randn(nblk, ell, ell, generator=g, **f64) * math.sqrt(1e-3)
    if dominance:
        u, v = _orthogonal(nodes, ell, g), _orthogonal(nodes, ell, g)
        sig = 1.0 + torch.rand(nodes, ell, generator=g, **f64)
        ill = torch.randperm(nodes, generator=g, device=_DEV)[: int(round(ill_frac * nodes))]
        sig[ill] = 1.0
        sig[ill, -1] = 1e-6
        keep[diag] = True
        fro = torch.where(keep, blocks, 0.0).square().sum((1, 2)).sqrt()
        fro[diag] = 0.0
        off = torch.segment_reduce(fro, "sum", lengths=deg)
        low = sig.min(1)[0]
        low[ill] = 1.0
        s = torch.where(off > 0, dominance * off / low, 1.0)
        blocks[diag] = ((u * sig[:, None, :]) @ v.transpose(1, 2)) * s[:, None, None]
    # scalar rows: (block k, a, b) goes to row i ell + a, after the row's earlier blocks
    ar = torch.arange(ell, device=_DEV)
    local = torch.arange(nblk, device=_DEV) - nptr[i]
    pos = ((nptr[i] * (ell * ell))[:, None, None] + ar[:, None] * (deg[i] * ell)[:, None, None]
           + (local * ell)[:, None, None] + ar)
    val = torch.empty(nblk * ell * ell, **f64)
    col = torch.empty(nblk * ell * ell, dtype=torch.int32, device=_DEV)
    kept = torch.empty(nblk * ell * ell, dtype=torch.bool, device=_DEV)
    flat = pos.reshape(-1)
    val[flat] = blocks.reshape(-1)
    col[flat] = (j[:, None, None] * ell + ar + 0 * ar[:, None]).to(torch.int32).reshape(-1)
    kept[flat] = keep.reshape(-1)
    del pos, flat, blocks, keep
    n = nodes * ell
    full = (deg * ell).repeat_interleave(ell)
    ends = kept.cumsum(0)[full.cumsum(0) - 1]
    rowptr = torch.cat([ends.new_zeros(1), ends])
    return n, rowptr, col[kept], val[kept]


def _rhs(rowptr, col, val, x):
    return torch.segment_reduce(val * x[col.long()], "sum", lengths=rowptr[1:] - rowptr[:-1])


def _vector(n, seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed) + 104729)
    return torch.randn(n, dtype=torch.float64, device=_DEV, generator=g)


def _shapes(case):
    """(nodes, unknowns per node) of a batch's matrices: sizes spread evenly over the logarithm."""
    c = int(case["count"])
    return [(int(round(case["nodes"] * case["ratio"] ** (k / max(1, c - 1)))), 4 + (7 * k) % 3) for k in range(c)]


def _csr(case, seed):
    return _matrix(case["gen"], case["nodes"], case["ell"], case["dominance"], case["ill_frac"], seed)


# ---------------------------------------------------------------------------
def _factor(s, A):
    return V.vbarms_factor(A, s["nlev"], s["droptol"], s["lfil"], precision=s["precision"],
                           group_size=s["group_size"])


def prepare(case, seed):
    s = dict(case)
    kind = case["kind"]
    if kind == "batch":
        s["A"], s["x"] = [], []
        for k, (nodes, ell) in enumerate(_shapes(case)):
            n, rp, ci, va = _matrix("geo", nodes, ell, case["dominance"], case["ill_frac"], seed * 64 + k)
            s["A"].append(V.vbarms_compress(n, rp, ci, va, case["tau"]))
            s["x"].append(_vector(n, seed * 64 + k))
        s["y"] = [torch.empty_like(x) for x in s["x"]]
        return s
    n, rp, ci, va = _csr(case, seed)
    s["n"] = n
    if kind == "whole":
        s["b"] = _rhs(rp, ci, va, _vector(n, seed))
        s["csr"] = (rp.cpu().numpy(), ci.cpu().numpy(), va.cpu().numpy())
        return s
    if kind == "compress":
        s["csr"] = (rp, ci, va)
        s["b"] = _vector(n, seed)
        return s
    s["A"] = V.vbarms_compress(n, rp, ci, va, case["tau"])
    if kind in ("ras", "fgmres"):
        s["b"] = _rhs(rp, ci, va, _vector(n, seed))
    else:
        s["x"] = _vector(n, seed)
        s["y"] = torch.empty_like(s["x"])
    if kind in ("apply", "fgmres"):
        s["M"] = _factor(s, s["A"])
    return s


def _solve(s, A, M):
    x = torch.zeros_like(s["b"])
    its, _, status = V.fgmres_solve(A, M, s["b"], x, rtol=1e-8, restart=50, maxit=500)
    return {"x": x, "its": its, "status": status}


def run(s):
    kind = s["kind"]
    if kind == "whole":
        A = V.vbarms_compress(s["n"], *s["csr"], s["tau"])
        return _solve(s, A, _factor(s, A))
    if kind == "compress":
        A = V.vbarms_compress(s["n"], *s["csr"], s["tau"])
        q = A.query()
        perm, bsz = np.empty(q["n"], np.int32), np.zeros(q["n"], np.int32)  # at most n blocks
        V.lib().vbarms_vbsr_export(A.h, perm.ctypes.data, bsz.ctypes.data, None, None, None, None)
        x = torch.zeros_like(s["b"])
        V.fgmres_solve(A, None, s["b"], x, rtol=0.0, restart=1, maxit=1)
        return {"x": x, "perm": perm, "bsz": bsz, "nnzb": q["nnzb"], "nval": q["nval"]}
    if kind == "factor":
        V.vbarms_apply(_factor(s, s["A"]), s["x"], s["y"])
        return s["y"]
    if kind == "batch":
        Ms = V.vbarms_factor_batched(s["A"], s["nlev"], s["droptol"], s["lfil"], precision=s["precision"])
        V.vbarms_apply_batched(Ms, s["x"], s["y"])
        return s["y"]
    if kind == "ras":
        M = V.vbarms_dd_factor(s["A"], s["nparts"], s["overlap"], True, s["nlev"], s["droptol"], s["lfil"],
                               precision=s["precision"])
        return _solve(s, s["A"], M)
    if kind == "apply":
        V.vbarms_apply(s["M"], s["x"], s["y"])
        return s["y"]
    return _solve(s, s["A"], s["M"])


# ---------------------------------------------------------------------------
def _nnz(nodes, ell, gen="geo"):
    if gen == "grid":
        return (7.0 * nodes - 6.0 * round(nodes ** (2.0 / 3.0))) * ell * ell
    return nodes * (15.0 * 0.9 + 1.0) * ell * ell


def work(case):
    """Bytes: the matrix and the vectors read once, the factors and the results
    written once (the factors hold about as many scalars as the matrix; they
    are read once by each application).  Flops: two per scalar of a product
    with the matrix or the factors; the elimination itself is counted as one
    pass over the factors."""
    kind = case["kind"]
    if kind == "batch":
        shapes = _shapes(case)
    else:
        shapes = [(case["nodes"], case["ell"])]
    nnz = sum(_nnz(n, e, case["gen"]) for n, e in shapes)
    rows = float(sum(n * e for n, e in shapes))
    size = 8.0 if case["precision"] == "fp64" else 4.0
    fill = 2.0 if case["tau"] == 0.9 and case["nlev"] == 5 else 1.2
    csr, factors, vecs = 12.0 * nnz + 8.0 * rows, fill * size * nnz, 16.0 * rows
    steps = 10.0  # iterations of FGMRES to 1e-8 on these matrices, about
    if kind == "compress":
        return {"bytes": csr + 8.0 * nnz + 20.0 * rows, "flops": 2.0 * nnz}
    if kind in ("factor", "batch"):
        return {"bytes": 8.0 * nnz + 2.0 * factors + vecs, "flops": 2.0 * fill * nnz}
    if kind == "apply":
        return {"bytes": factors + vecs, "flops": 2.0 * fill * nnz}
    solve = steps * (8.0 * nnz + factors + 4.0 * vecs)
    flops = steps * 2.0 * (1.0 + fill) * nnz
    if kind == "fgmres":
        return {"bytes": solve, "flops": flops}
    if kind == "ras":
        return {"bytes": 8.0 * nnz + factors + solve, "flops": flops}
    return {"bytes": csr + 8.0 * nnz + factors + solve, "flops": flops}


def exact(case, seed):
    """The solution where the pass solves A x = b (b was made from it), one
    step of GMRES(1) for ``compress``; an incomplete factorization's own
    application has no value apart from its factors."""
    kind = case["kind"]
    if kind in ("whole", "ras", "fgmres"):
        return {"x": _vector(case["nodes"] * case["ell"], seed), "its": None, "status": None}
    if kind == "compress":
        n, rp, ci, va = _csr(case, seed)
        b = _vector(n, seed)
        ab = _rhs(rp, ci, va, b)
        return {"x": b * (torch.dot(ab, b) / torch.dot(ab, ab)), "perm": None, "bsz": None, "nnzb": None,
                "nval": None}
    return None
