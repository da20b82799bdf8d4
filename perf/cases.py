"""The work a user of the framework has it do, as cases that can be timed.

Every case goes through the public binding (`paper_2512_01257_gb300.rafeast`):
the building blocks of RA-FEAST one at a time (sparse product,
orthonormalisation, Rayleigh-Ritz, randomized warmstart, quadrature filter),
whole solves and a batched solve. The graphs are the families of
`workloads/configs.py` (grids, kNN graphs of points in the unit cube, random
geometric graphs, stochastic block models) at that file's sizes and between
them, generated here on the GPU from the seed alone.

What a user has from earlier runs or estimates (a block rich in low
eigenvectors, a search interval that ends in a gap) comes from a
Chebyshev-filtered subspace iteration written in torch below.
"""
import math

import numpy as np
import torch

from paper_2512_01257_gb300 import rafeast as R

DEV = "cuda"
F64 = torch.float64


# ---- graphs --------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _laplacian(n, i, j):
    """CSR (int32, int32, float64) of D - W for the unit-weight graph whose edges
    are {i, j}, in either direction and possibly repeated."""
    keep = i != j
    i, j = i[keep].long(), j[keep].long()
    key = torch.unique(torch.cat([i * n + j, j * n + i]))
    row, col = key // n, key % n
    deg = torch.bincount(row, minlength=n)
    diag = torch.arange(n, device=DEV)
    key = torch.cat([key, diag * n + diag])
    val = torch.cat([torch.full_like(row, -1, dtype=F64), deg.double()])
    key, order = torch.sort(key)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(deg + 1, 0)
    return rp.int(), (key % n).int().contiguous(), val[order].contiguous()


def _grid(dims):
    idx = torch.arange(math.prod(dims), device=DEV).reshape(dims)
    a, b = [], []
    for d in range(len(dims)):
        a.append(idx.narrow(d, 0, dims[d] - 1).reshape(-1))
        b.append(idx.narrow(d, 1, dims[d] - 1).reshape(-1))
    return _laplacian(idx.numel(), torch.cat(a), torch.cat(b))


def _knn(n, seed, k=10):
    """k nearest neighbours among n uniform points of the unit cube, union-
    symmetrised (searched in the 27 cells around a point; the order of the
    points is random, as the points come)."""
    g = _generator(seed)
    x = torch.rand(n, 3, device=DEV, dtype=F64, generator=g)
    s = max(1, int((n / 6.0) ** (1.0 / 3.0)))
    c = (x * s).long().clamp_(0, s - 1) + 1
    cell = (c[:, 0] * (s + 2) + c[:, 1]) * (s + 2) + c[:, 2]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=(s + 2) ** 3)
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full(((s + 2) ** 3, cap), -1, dtype=torch.int64, device=DEV)
    sc = cell[order]
    table[sc, torch.arange(n, device=DEV) - start[sc]] = order
    o = torch.tensor([-1, 0, 1], device=DEV)
    near = ((o[:, None, None] * (s + 2) + o[None, :, None]) * (s + 2) + o[None, None, :]).reshape(-1)
    src, dst = [], []
    for p in torch.arange(n, device=DEV).split(16384):
        cand = table[cell[p][:, None] + near[None, :]].reshape(len(p), -1)
        d = ((x[cand.clamp(min=0)] - x[p][:, None, :]) ** 2).sum(-1)
        d[(cand < 0) | (cand == p[:, None])] = math.inf
        d, at = torch.topk(d, min(k, d.shape[1]), dim=1, largest=False)
        ok = torch.isfinite(d)
        src.append(p[:, None].expand_as(at)[ok])
        dst.append(torch.gather(cand, 1, at)[ok])
    return _laplacian(n, torch.cat(src), torch.cat(dst))


def _rgg(n, seed):
    """Random geometric graph in the unit square, r = 1.5 sqrt(log n / n)."""
    x = torch.rand(n, 2, device=DEV, dtype=F64, generator=_generator(seed))
    r2 = 2.25 * math.log(n) / n
    src, dst = [], []
    for p in torch.arange(n, device=DEV).split(2048):
        d = (x[p, None, 0] - x[None, :, 0]) ** 2 + (x[p, None, 1] - x[None, :, 1]) ** 2
        a, b = torch.nonzero(d <= r2, as_tuple=True)
        src.append(p[a])
        dst.append(b)
    return _laplacian(n, torch.cat(src), torch.cat(dst))


def _sbm(n, blocks, seed):
    """Stochastic block model of equal blocks: about 20 neighbours inside a
    vertex's block and one outside."""
    g = _generator(seed)
    m = 10 * n
    block = torch.randint(0, blocks, (m,), device=DEV, generator=g)
    size = n // blocks
    i = block * size + torch.randint(0, size, (m,), device=DEV, generator=g)
    j = block * size + torch.randint(0, size, (m,), device=DEV, generator=g)
    u = torch.randint(0, n, (n // 2,), device=DEV, generator=g)
    v = torch.randint(0, n, (n // 2,), device=DEV, generator=g)
    return _laplacian(n, torch.cat([i, u]), torch.cat([j, v]))


def _dims(n, d):
    """d unequal grid sides with a product near n."""
    a = max(2, round(n ** (1.0 / d)))
    return tuple([a + t for t in range(d - 1)] + [max(2, round(n / math.prod(a + t for t in range(d - 1))))])


def _graph(case, seed):
    """(CSR, diagonal shift, lower end of the search interval, dims or None) of the
    case's family."""
    fam, n = case["family"], case["n"]
    if fam in ("grid2d", "grid3d"):
        dims = _dims(n, 2 if fam == "grid2d" else 3)
        # the shift a user adds to make the grid's Laplacian definite
        shift = 1e-2 * (1.0 + 0.1 * (seed % 7))
        return _grid(dims), shift, 0.5 * shift, dims
    if fam == "knn":
        return _knn(n, seed), 1e-3, 5e-4, None
    if fam == "rgg":
        return _rgg(n, seed), 0.0, 1e-3, None
    return _sbm(n, case["blocks"], seed), 1e-3, 5e-4, None


class Handle:
    """A library handle that is given back with its state."""

    def __init__(self, csr, shift):
        self.h = R.rafeast_create(csr[0], csr[1], csr[2], shift)

    def __del__(self):
        R.rafeast_destroy(self.h)


# ---- 64-bit torch arithmetic for inputs and expected values -----------------------

class Ell:
    """A = D - W + shift I over padded neighbour lists; blocks are (n, m) float64
    or complex128."""

    def __init__(self, csr, shift):
        rp, ci, _ = csr
        rp, ci = rp.long(), ci.long()
        n = rp.numel() - 1
        row = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
        off = ci != row
        row, ci = row[off], ci[off]
        deg = torch.bincount(row, minlength=n)
        first = torch.cumsum(deg, 0) - deg
        self.w = int(deg.max())
        self.nb = torch.full((self.w, n), n, dtype=torch.int64, device=DEV)
        self.nb[torch.arange(row.numel(), device=DEV) - first[row], row] = ci
        self.diag = deg.double()[:, None] + shift
        self.n, self.top = n, 2.0 * float(deg.max()) + shift

    def __matmul__(self, x):
        pad = torch.cat([x, torch.zeros_like(x[:1])])
        y = self.diag * x
        for t in range(self.w):
            y -= pad[self.nb[t]]
        return y


def _orth(x):
    for _ in range(2):
        low = torch.linalg.cholesky(x.T @ x)
        x = torch.linalg.solve_triangular(low, x.T, upper=False).T
    return x


def _ritz(a, x):
    """Orthonormal Ritz vectors and values (host) of span(x)."""
    x = _orth(x)
    g = (x.T @ (a @ x)).cpu().numpy()
    th, v = np.linalg.eigh(0.5 * (g + g.T))
    return x @ torch.from_numpy(v).to(DEV), th


def _low_block(a, m, seed, rounds):
    """m Ritz vectors rich in a's low eigenvectors: `rounds` Chebyshev filters
    that damp the spectrum above the last Ritz value."""
    x = torch.randn(a.n, m, device=DEV, dtype=F64, generator=_generator(seed + 17))
    cut = a.top * min(0.25, (m / a.n) ** (2.0 / 3.0))
    for _ in range(rounds):
        deg = max(8, min(240, int(2.5 * math.sqrt(a.top / cut))))
        c, e = 0.5 * (a.top + cut), 0.5 * (a.top - cut)
        y0, y1 = x, (a @ x - c * x) / e
        for k in range(deg):
            y0, y1 = y1, (2.0 / e) * (a @ y1 - c * y1) - y0
            if k % 16 == 15:
                scale = 1.0 / y1.norm(dim=0)
                y0, y1 = y0 * scale, y1 * scale
        x, th = _ritz(a, y1)
        cut = max(float(th[-1]), 1e-6 * a.top)
    return x, th


def _upper_end(th, count, slack=2):
    """Search interval's upper end: the middle of the widest gap near `count`
    eigenvalues."""
    best = max(range(max(1, count - slack), min(len(th) - 1, count + slack) + 1), key=lambda t: th[t] - th[t - 1])
    return float(0.5 * (th[best - 1] + th[best]))


def _colmajor(x):
    return x.T.contiguous()


# ---- the cases -------------------------------------------------------------------

def listed():
    return [
        # the smallest product: A times a 24-column block of the 40 x 50 grid
        dict(name="spmm_grid2k", op="spmm", family="grid2d", n=2000, m=24),
        # A Q of a Rayleigh-Ritz step at the kNN benchmark's size
        dict(name="spmm_knn200k", op="spmm", family="knn", n=200000, m=80),
        # the QR step of an outer iteration at that size
        dict(name="orth_knn200k", op="orth", family="knn", n=200000, m=80),
        # the Rayleigh-Ritz step of an outer iteration at that size
        dict(name="rr_knn200k", op="rr", family="knn", n=200000, m=80),
        # Phase 1 alone on the small kNN graph (52 columns, five products)
        dict(name="warmstart_knn8k", op="warmstart", family="knn", n=8000, m=42, p=10, q=2),
        # plain FEAST's filter on the small grid: accurate solves, launch bound
        dict(name="filter_grid2k_fp64", op="filter", family="grid2d", n=2000, m=24, nc=8, precision="fp64",
             form="direct", tol=1e-10, cap=20000),
        # the same on the paper's random geometric graph (about 68 neighbours a row)
        dict(name="filter_rgg16k_fp64", op="filter", family="rgg", n=16000, m=69, nc=8, precision="fp64",
             form="direct", tol=1e-10, cap=20000),
        # the first, relaxed filter of a mixed-precision run on the million-vertex
        # grid from a random start (later filters of a float32 run amplify
        # rounding so much that a single one is no reference for another; the
        # whole solves below cover them)
        dict(name="filter_grid1m_mixed", op="filter", family="grid3d", n=1000000, m=96, nc=4, precision="mixed",
             form="direct", tol=1e-2, cap=100),
        # RA-FEAST in FP64 on the small kNN graph
        dict(name="solve_knn8k_fp64", op="solve", family="knn", n=8000, m=42, nc=2, precision="fp64", tol=1e-4,
             outer=1e-10, cap=20000, p=10, q=2, max_outer=40),
        # the paper's experiment: RA-FEAST in FP64, at most four outer iterations
        dict(name="solve_rgg16k_fp64", op="solve", family="rgg", n=16000, m=69, nc=2, precision="fp64", tol=1e-4,
             outer=1e-10, cap=2000, p=10, q=2, max_outer=4),
        # the headline workload: RA-FEAST, mixed precision, 64 of 80 vectors
        dict(name="solve_knn200k_mixed", op="solve", family="knn", n=200000, m=80, nc=4, precision="mixed", tol=1e-2,
             outer=1e-11, cap=60, p=20, q=2, max_outer=40),
        # a serving batch: twelve block-model graphs of uneven sizes at once
        dict(name="batch_sbm_mixed", op="batch", family="sbm", count=12, lo=2000, hi=100000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["spmm", "orth", "rr", "warmstart", "filter", "filter", "solve", "solve", "batch"])
    if op in ("spmm", "orth", "rr"):
        fam = rng.choice(["grid2d", "knn", "grid3d"])
        return dict(op=op, family=fam, n=_log(rng, 2000, 200000), m=rng.randint(12, 96))
    if op == "warmstart":
        return dict(op=op, family=rng.choice(["knn", "grid3d"]), n=_log(rng, 2000, 200000), m=rng.randint(16, 80),
                    p=rng.choice([10, 20]), q=rng.choice([1, 2]))
    if op == "filter":
        if rng.random() < 0.5:
            return dict(op=op, family="grid3d", n=_log(rng, 20000, 1000000), m=rng.randint(16, 96),
                        nc=rng.choice([2, 4, 8]), precision="mixed", form="direct", tol=1e-2,
                        cap=rng.choice([60, 100]))
        return dict(op=op, family=rng.choice(["grid2d", "rgg"]), n=_log(rng, 2000, 16000), m=rng.randint(16, 69),
                    nc=rng.choice([2, 4, 8]), precision="fp64", form="direct", tol=1e-10, cap=20000)
    if op == "solve":
        if rng.random() < 0.5:
            fam = rng.choice(["knn", "grid3d"])
            return dict(op=op, family=fam, n=_log(rng, 10000, 200000 if fam == "knn" else 100000),
                        m=rng.randint(24, 80), nc=4, precision="mixed", tol=1e-2, outer=1e-11, cap=60, p=20, q=2,
                        max_outer=40)
        return dict(op=op, family=rng.choice(["knn", "rgg"]), n=_log(rng, 2000, 8000), m=rng.randint(18, 44), nc=2,
                    precision="fp64", tol=1e-4, outer=1e-10, cap=20000, p=10, q=2, max_outer=40)
    return dict(op=op, family="sbm", count=rng.randint(3, 12), lo=2000, hi=_log(rng, 8000, 100000))


def _params(c, lmin, lmax, m, start):
    return R.make_params(lmin, lmax, m, c["nc"], c.get("e", 1.0), c["tol"], c.get("outer", 1e-10),
                         c.get("max_outer", 40), c["cap"], R.RAFEAST_MIXED if c["precision"] == "mixed" else R.RAFEAST_FP64,
                         R.RAFEAST_FORM_DIRECT if c.get("form") == "direct" else R.RAFEAST_FORM_CORRECTION, start)


def _batch_members(case, seed):
    """n, blocks and seed of the graphs of a batch: the sizes are the case's own,
    spread over its range; the edges come from the seed."""
    k = case["count"]
    for t in range(k):
        n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** ((t + 0.5) / k)))
        blocks = 4 + (5 * t) % 13
        yield dict(family="sbm", n=n // blocks * blocks, blocks=blocks), seed * 100 + t


def _one(case, seed, rounds=6):
    """A matrix, its low Ritz pairs and the search interval."""
    csr, shift, lmin, dims = _graph(case, seed)
    a = Ell(csr, shift)
    m, fam = case["m"], case["family"]
    x, th = _low_block(a, m, seed, rounds)
    count = {"sbm": int(m / 1.5), "rgg": int(m / 1.5)}.get(fam, int(0.8 * m))
    return csr, shift, a, x, th, lmin, _upper_end(th, count), dims


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        s = dict(case=case, hs=[], prms=[], warm=[], evals=[], evecs=[], signals=[])
        for g, gseed in _batch_members(case, seed):
            k = g["blocks"] + 8
            g["m"] = math.ceil(1.5 * k)
            csr, shift, a, _, _, lmin, lmax, _ = _one(g, gseed)
            c = dict(nc=2, e=0.3, tol=1e-2, outer=1e-10, cap=100, max_outer=150, precision="mixed")
            s["hs"].append(Handle(csr, shift))
            s["prms"].append(_params(c, lmin, lmax, g["m"], R.RAFEAST_START_SUBSPACE))
            s["warm"].append((lmin, lmax, g["m"], 10, 2, gseed))
            s["evals"].append(torch.zeros(g["m"], dtype=F64, device=DEV))
            s["evecs"].append(torch.zeros(g["m"], a.n, dtype=F64, device=DEV))
        return s
    if op in ("spmm", "orth"):
        csr, shift, _, _ = _graph(case, seed)
        x = torch.randn(case["m"], case["n"] if case["family"] == "knn" else csr[0].numel() - 1, device=DEV, dtype=F64,
                        generator=_generator(seed))
        if op == "orth":  # a filtered block: columns of uneven size that lean on one another
            mix = torch.randn(case["m"], case["m"], device=DEV, dtype=F64, generator=_generator(seed + 1))
            x = (mix * torch.logspace(0, -2, case["m"], device=DEV, dtype=F64)) @ x
        return dict(case=case, h=Handle(csr, shift), x=x, y=torch.empty_like(x))
    if op == "warmstart":
        csr, shift, lmin, _ = _graph(case, seed)
        n = csr[0].numel() - 1
        return dict(case=case, h=Handle(csr, shift), lmin=lmin, seed=seed,
                    q=torch.empty(case["m"], n, dtype=F64, device=DEV))
    csr, shift, a, x, th, lmin, lmax, _ = _one(case, seed, 2 if op == "rr" else 6)
    s = dict(case=case, h=Handle(csr, shift), lmin=lmin, lmax=lmax)
    if op == "rr":  # the block as it leaves the QR step: orthonormal, not yet Ritz vectors
        mix = torch.randn(case["m"], case["m"], device=DEV, dtype=F64, generator=_generator(seed + 1))
        s["x"] = _colmajor(x @ torch.linalg.qr(mix)[0])
        s["y"] = torch.empty_like(s["x"])
    elif op == "filter":
        # a random start's orthonormal block
        x = _orth(torch.randn(a.n, case["m"], device=DEV, dtype=F64, generator=_generator(seed + 2)))
        s["x"] = _colmajor(x)
        s["y"] = torch.empty_like(s["x"])
        s["prm"] = _params(case, lmin, lmax, case["m"], R.RAFEAST_START_SUBSPACE)
    else:
        s["prm"] = _params(case, lmin, lmax, case["m"], R.RAFEAST_START_SUBSPACE)
        s["seed"] = seed
        s["evals"] = torch.zeros(case["m"], dtype=F64, device=DEV)
        s["evecs"] = torch.zeros(case["m"], a.n, dtype=F64, device=DEV)
        s["signals"] = torch.randn(a.n, 8, device=DEV, generator=_generator(seed + 3))
    return s


def _low_pass(evecs, signals):
    """The graph signals' part in the eigenspace found: what the eigenvectors are
    for, and free of their signs and of rotations inside clusters."""
    v = evecs.float()
    return v.T @ (v @ signals)


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "spmm":
        R.rafeast_spmm(s["h"].h, c["m"], 1.0, 0.0, s["x"], s["y"], R.RAFEAST_FP64)
        return s["y"]
    if op == "orth":
        s["y"].copy_(s["x"])  # in place: the filtered block itself is kept
        r = R.rafeast_orthonormalize(s["h"].h, c["m"], s["y"], want_r=True)
        return s["y"], r
    if op == "rr":
        s["y"].copy_(s["x"])
        theta, resid = R.rafeast_rayleigh_ritz(s["h"].h, c["m"], s["y"])
        return dict(q=s["y"], theta=theta, resid=resid)
    if op == "warmstart":
        R.rafeast_warmstart(s["h"].h, s["lmin"], 40.0 * s["lmin"], c["m"], c["p"], c["q"], s["seed"])
        theta = R.rafeast_get_subspace(s["h"].h, s["q"], c["m"])
        return dict(q=s["q"], theta=theta)
    if op == "filter":
        R.rafeast_filter(s["h"].h, s["prm"], s["x"], None, s["y"])
        # the mixed filter's solves are float32, so its result is handed on as that
        return s["y"].float() if c["precision"] == "mixed" else s["y"]
    if op == "solve":
        p = s["prm"]
        R.rafeast_warmstart(s["h"].h, p.lmin, p.lmax, c["m"], c["p"], c["q"], s["seed"])
        status, found, _ = R.rafeast_solve(s["h"].h, p, s["evals"], s["evecs"])
        # the first `found` pairs are the answer: the others lie outside the interval
        s["evals"][found:] = 0.0
        return dict(found=found, evals=s["evals"], low=_low_pass(s["evecs"][:found], s["signals"]))
    for h, w in zip(s["hs"], s["warm"]):
        R.rafeast_warmstart(h.h, *w)
    status, found, _ = R.rafeast_solve_batched([h.h for h in s["hs"]], s["prms"], s["evals"], s["evecs"])
    for e, k in zip(s["evals"], found):
        e[k:] = 0.0
    return dict(found=list(found), evals=s["evals"])


# ---- what a pass cannot do without ------------------------------------------------

_ROW = {"grid2d": 5.0, "grid3d": 7.0, "knn": 12.5, "rgg": 68.0, "sbm": 22.0}  # nonzeros a row
# Krylov steps of a pass, roughly: an accurate filter runs to 1e-10, a relaxed
# solve repeats its capped or loosely converged filter
_STEPS = {"filter": 400, "solve_fp64": 700, "solve_mixed": 600, "batch": 1500}


def work(case):
    op = case["op"]
    if op == "batch":
        every = [(g["n"], math.ceil(1.5 * (g["blocks"] + 8))) for g, _ in _batch_members(case, 0)]
        cells = sum(n * m for n, m in every)
        step = cells * 2 * 4 + sum(n for n, _ in every) * 4 * _ROW["sbm"]
        return dict(bytes=_STEPS["batch"] / 4 * step, flops=_STEPS["batch"] / 4 * cells * (_ROW["sbm"] + 30))
    n, m, d = case["n"], case["m"], _ROW[case["family"]]
    matrix, block = n * d * 4, n * m * 8
    if op == "spmm":
        return dict(bytes=matrix + 2 * block, flops=2 * n * m * d)
    if op == "orth":
        return dict(bytes=2 * block, flops=4 * n * m * m)
    if op == "rr":  # A Q, Q^T A Q, Q V
        return dict(bytes=matrix + 2 * block, flops=2 * n * m * (d + 2 * m))
    if op == "warmstart":
        k = m + case["p"]
        return dict(bytes=matrix + block, flops=2 * n * k * ((2 * case["q"] + 2) * d + 4 * k))
    # a Krylov step reads the matrix and one block and writes one block
    size = 4 if case["precision"] == "mixed" else 8
    steps = case["cap"] if case["precision"] == "mixed" and op == "filter" else \
        _STEPS[op if op == "filter" else "solve_" + case["precision"]]
    step = matrix + 2 * n * m * size
    return dict(bytes=2 * block + steps * step, flops=steps * n * m * (2 * d + 10 + 8 * case["nc"]))


# ---- the same in 64 bits -----------------------------------------------------------

def _nodes(prm):
    x, om = np.polynomial.legendre.leggauss(prm.nc)
    t = 0.5 * math.pi * (1.0 + x)
    c, r, e = 0.5 * (prm.lmin + prm.lmax), 0.5 * (prm.lmax - prm.lmin), prm.ellipse_ratio
    return c + r * (np.cos(t) + 1j * e * np.sin(t)), 0.5 * r * om * (e * np.cos(t) + 1j * np.sin(t))


def _filtered(a, prm, q):
    """Sum over the nodes of Re(w (z - A)^-1 q) with each system solved as the
    parameters say: conjugate orthogonal CG from zero, a column stopping at
    tol |q| or at the cap (an accurate solve is run on to 1e-14)."""
    tol = prm.solve_tol if prm.solve_tol > 1e-8 else 1e-14
    out = torch.zeros_like(q)
    stop = tol * q.norm(dim=0)
    for zj, wj in zip(*_nodes(prm)):
        r = q.to(torch.complex128)
        x, p, rho = torch.zeros_like(r), torch.zeros_like(r), None
        on = torch.ones(r.shape[1], dtype=torch.bool, device=DEV)
        for _ in range(min(prm.max_inner, 6000)):
            on = on & (torch.linalg.vector_norm(r, dim=0) > stop)
            if not bool(on.any()):
                break
            new = (r * r).sum(0)
            p = r if rho is None else r + (new / rho) * p
            ap = zj * p - a @ p
            alpha = torch.where(on, new / (p * ap).sum(0), 0)
            x, r, rho = x + alpha * p, r - alpha * ap, new
        out += (complex(wj) * x).real
    return out


def exact(case, seed):
    op = case["op"]
    if op in ("warmstart", "batch"):
        return None  # the random block is the library's own; the sweep takes too long
    if op == "solve":
        return _solved(case, seed)
    s = prepare(case, seed)
    csr, shift, _, _ = _graph(case, seed)
    a = Ell(csr, shift)
    x = _colmajor(s["x"])
    if op == "spmm":
        return _colmajor(a @ x)
    if op == "orth":
        q, r = torch.linalg.qr(x)
        sign = torch.sign(torch.diagonal(r))
        return _colmajor(q * sign), (sign[:, None] * r).cpu().numpy()
    if op == "rr":
        q, th = _ritz(a, x)
        resid = (a @ q - q * torch.from_numpy(th).to(DEV)).norm(dim=0) / a.top
        return dict(q=None, theta=th, resid=resid.cpu().numpy())  # the vectors' signs are free
    return _colmajor(_filtered(a, s["prm"], x))


def _solved(case, seed):
    """Closed form on the grids, a dense eigensolver on small graphs."""
    if case["family"] == "rgg" and case["max_outer"] < 10 or case["family"] != "grid3d" and case["n"] > 8000:
        return None
    csr, shift, a, _, _, lmin, lmax, dims = _one(case, seed)
    if dims is None:
        dense = torch.diag(a.diag[:, 0])
        for t in range(a.w):
            i = torch.nonzero(a.nb[t] < a.n)[:, 0]
            dense[i, a.nb[t][i]] = -1.0
        lam, vec = torch.linalg.eigh(dense)
        at = torch.nonzero((lam >= lmin) & (lam <= lmax))[:, 0]
        lam, vec = lam[at], vec[:, at]
    else:
        one, basis = [], []
        for d in dims:
            k = torch.arange(d, device=DEV, dtype=F64)
            one.append(4.0 * torch.sin(0.5 * math.pi * k / d) ** 2)
            v = torch.cos(math.pi * (k[:, None] + 0.5) * k[None, :] / d)
            basis.append(v / v.norm(dim=0))
        total = (one[0][:, None, None] + one[1][None, :, None] + one[2][None, None, :]).reshape(-1) + shift
        lam, order = torch.sort(total)
        order, lam = order[lam <= lmax], lam[lam <= lmax]
        i, j, k = order // (dims[1] * dims[2]), order // dims[2] % dims[1], order % dims[2]
        vec = torch.einsum("am,bm,cm->abcm", basis[0][:, i], basis[1][:, j], basis[2][:, k]).reshape(-1, len(lam))
    signals = torch.randn(a.n, 8, device=DEV, generator=_generator(seed + 3)).double()
    evals = torch.zeros(case["m"], dtype=F64, device=DEV)
    evals[:len(lam)] = lam[:case["m"]]
    return dict(found=len(lam), evals=evals, low=vec @ (vec.T @ signals))
