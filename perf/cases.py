"""The work a user of this package has it do, as timed cases: one-call solves,
the phases of a factorization kept by a program that calls them again and
again, preconditioner applications, Krylov solves on kept factors, batched
systems and a differentiable solve.

Matrices: upwind convection-diffusion on 2D (5-point) and 3D (7-point) grids,
with constant or per-cell log-uniform diffusion; the 27-point Poisson stencil on
3D grids, also with random weights; random band matrices (9 off-diagonals a
row).  Sizes and options are those of the package's own workloads, tests and
benchmark, and the ranges they span.

A case holds: ``kind`` (what is called), ``grid`` (g2, g3, p27 or band), ``N``
(grid side, or rows of a band matrix), ``hw`` (half-width of the band), ``k``
(level of fill), ``m`` (GMRES restart), and options of its kind.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_0803_0048_gb300 as P
from paper_0803_0048_gb300 import workloads as W

RTOL = 1e-8

# Entries of F per row (interior rows of the grids; averages of the band matrices)
ROW_A = {"g2": 5, "g3": 7, "p27": 27, "band": 10}
ROW_F = {"g2": (5, 7, 9, 13), "g3": (7, 13, 23, 43), "p27": (27, 63, 115, 183),
         "band": (10, 30, 118, 545)}


def listed():
    return [
        # One call on a small system, as inside an outer loop: latency and launches.
        dict(name="solve_g2_64_k2", kind="solve", grid="g2", N=64, k=2, m=30, theta=False),
        # One call on a large matrix without grid structure: a deep, narrow dependency graph.
        dict(name="solve_band_160k_k2", kind="solve", grid="band", N=160000, hw=2000, k=2, m=50,
             theta=False),
        # The symbolic phase and the first numeric one, once per mesh.
        dict(name="setup_g3_64_k2", kind="setup", grid="g3", N=64, k=2, theta=True),
        # New values on a kept pattern, every time or Newton step.
        dict(name="refactor_p27_50_k1", kind="refactor", grid="p27", N=50, k=1, theta=True),
        # One preconditioner application inside a user's own Krylov method.
        dict(name="apply_g3_64_k2", kind="apply", grid="g3", N=64, k=2, theta=True,
             transpose=False),
        # The transposed application, for adjoint and bi-orthogonal methods.
        dict(name="apply_t_g2_256_k2", kind="apply", grid="g2", N=256, k=2, theta=True,
             transpose=True),
        # The incomplete inverses built from kept factors, and one application.
        dict(name="iilu_band_160k_k1", kind="iilu", grid="band", N=160000, hw=2000, k=1,
             theta=False),
        # GMRES on kept factors, the largest grid.
        dict(name="gmres_p27_90_k0", kind="gmres", grid="p27", N=90, k=0, m=50, theta=False,
             prec="ilu"),
        # GMRES with the incomplete inverses: cheap applications, many iterations.
        dict(name="gmres_iilu_g3_64_k2", kind="gmres", grid="g3", N=64, k=2, m=50, theta=False,
             prec="iilu"),
        # BiCGSTAB on kept factors.
        dict(name="bicgstab_p27_50_k1", kind="bicgstab", grid="p27", N=50, k=1, theta=False,
             prec="ilu"),
        # Many independent systems in one launch: value sets on one grid and uneven grids.
        dict(name="batch_g3_32_k1", kind="batch", grid="g3", N=32, k=1, m=30, theta=True,
             sets=256, uneven=32),
        # Forward and backward through a solve: gradients of the values and right-hand side.
        dict(name="adjoint_g2_256_k2", kind="adjoint", grid="g2", N=256, k=2, m=30, theta=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["solve", "setup", "refactor", "apply", "apply", "iilu", "gmres",
                           "gmres", "bicgstab", "batch", "adjoint"])
        grid = rng.choice(["g2", "g3", "p27", "band"])
        c = dict(kind=kind, grid=grid, k=rng.choice([0, 1, 1, 2, 2]), theta=rng.random() < 0.5)
        if kind == "batch":
            c.update(grid="g3", N=rng.randint(10, 34), k=rng.choice([0, 1, 1]), m=30, theta=True,
                     sets=_log_int(rng, 16, 256), uneven=rng.choice([0, rng.randint(1, 32)]))
        elif kind == "adjoint":
            c.update(grid="g2", N=_log_int(rng, 24, 256), m=30, theta=True)
        elif grid == "g2":
            c["N"] = _log_int(rng, 24, 300)
        elif grid == "g3":
            c["N"] = _log_int(rng, 10, 72)
        elif grid == "p27":
            c.update(N=_log_int(rng, 10, 90), k=min(c["k"], 1))
        else:
            c.update(N=_log_int(rng, 4000, 160000), hw=_log_int(rng, 100, 2000), theta=False)
        if kind in ("solve", "gmres"):
            c["m"] = rng.choice([30, 50])
        if kind == "apply":
            c["transpose"] = rng.random() < 0.4
        if kind in ("gmres", "bicgstab"):
            c["prec"] = rng.choice(["ilu", "ilu", "iilu"])
        if kind == "solve" and c["theta"]:
            c["theta"] = False
        if c.get("prec") == "iilu" and c["theta"]:
            c["theta"] = False  # the incomplete inverses suit the constant-coefficient grids
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _rand(seed, tag, n, lo=-1.0, hi=1.0):
    g = torch.Generator(device="cpu")
    g.manual_seed(1000003 * seed + tag)
    return lo + (hi - lo) * torch.rand(n, generator=g, dtype=torch.float64)


def _stencil27(N, dev):
    n = N ** 3
    idx = torch.arange(n, device=dev)
    x, y, z = idx % N, (idx // N) % N, idx // (N * N)
    cols = []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                ok = ((x + dx >= 0) & (x + dx < N) & (y + dy >= 0) & (y + dy < N) &
                      (z + dz >= 0) & (z + dz < N))
                cols.append(torch.where(ok, idx + dx + N * dy + N * N * dz, -1))
    C = torch.stack(cols, dim=1)
    keep = C >= 0
    rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(keep.sum(dim=1), 0)
    return rp, C, keep


def _grid_values(pat, theta, beta, dev):
    return W.fd_values(pat, theta if theta is not None
                       else torch.ones(pat.n, dtype=torch.float64, device=dev), beta)


def _theta(seed, tag, n, dev):
    lo, hi = np.log(0.1), np.log(10.0)
    return torch.exp(_rand(seed, tag, n, lo, hi)).to(dev)


def _matrix(case, seed):
    """(rowptr, colind, vals) on the device."""
    dev, g, N = _device(), case["grid"], case["N"]
    if g == "band":  # one random pattern of the size; the seed draws the values
        A = W.random_band(N, 9, case["hw"], 77)
        ci = torch.from_numpy(A.colind).to(dev).reshape(N, 10)
        v = _rand(seed, 1, 10 * N).to(dev).reshape(N, 10)
        on = ci == torch.arange(N, device=dev)[:, None]
        diag = 1.2 * torch.where(on, 0.0, v.abs()).sum(dim=1)
        v = torch.where(on, diag[:, None], v)
        return torch.from_numpy(A.rowptr).to(dev), ci.reshape(-1), v.reshape(-1)
    if g == "p27":
        rp, C, keep = _stencil27(N, dev)
        V = torch.full(C.shape, -1.0, dtype=torch.float64, device=dev)
        V[:, 13] = 26.0
        if case["theta"]:  # random weights, rows still weakly dominant
            w = _rand(seed, 1, C.numel(), 0.5, 1.5).to(dev).reshape(C.shape)
            diag = w.sum(dim=1) - w[:, 13]
            V = V * w
            V[:, 13] = diag
        return rp, C[keep].to(torch.int32), V[keep].contiguous()
    d = 2 if g == "g2" else 3
    pat = W.fd_pattern(N, d)
    theta = _theta(seed, 1, pat.n, dev) if case["theta"] else None
    beta = (20.0, 20.0) if d == 2 else (50.0, 50.0, 50.0)
    v = _grid_values(pat, theta, beta, dev)
    return torch.from_numpy(pat.rowptr).to(dev), torch.from_numpy(pat.colind).to(dev), v


def _matvec(rp, ci, v, x):
    """A x by rows of equal padded length (a fixed order on any machine)."""
    w = int((rp[1:] - rp[:-1]).max())
    q = rp[:-1, None] + torch.arange(w, device=rp.device)[None, :]
    ok = q < rp[1:, None]
    q = torch.where(ok, q, 0)
    return torch.where(ok, v[q] * x[ci[q].long()], 0.0).sum(dim=1)


def _system(case, seed):
    rp, ci, v = _matrix(case, seed)
    x = _rand(seed, 2, rp.numel() - 1).to(rp.device)
    return rp, ci, v, x, _matvec(rp, ci, v, x)


def _batch_shapes(case):
    """Sides of the uneven grids, half to five quarters of N."""
    g = torch.Generator().manual_seed(case["N"])
    lo, hi = max(4, case["N"] // 2), max(5, case["N"] * 5 // 4)
    return torch.randint(lo, hi + 1, (case["uneven"],), generator=g).tolist()


def _batch_system(N, seed, tag):
    dev = _device()
    pat = W.fd_pattern(N, 3)
    beta = [float(t) for t in _rand(seed, 10 * tag + 3, 3, 0.0, 30.0)]
    v = _grid_values(pat, _theta(seed, 10 * tag + 1, pat.n, dev), beta, dev)
    return pat, v, _rand(seed, 10 * tag + 2, pat.n).to(dev)


def prepare(case, seed):
    kind, k = case["kind"], case["k"]
    st = {"case": case}
    if kind == "batch":
        return _prepare_batch(case, seed, st)
    if kind in ("solve", "gmres", "bicgstab", "adjoint"):
        st["rp"], st["ci"], st["v"], _, st["b"] = _system(case, seed)
    else:
        st["rp"], st["ci"], st["v"] = _matrix(case, seed)
    n = st["rp"].numel() - 1
    if kind == "adjoint":
        st["solver"] = P.IlukSolver(st["rp"], st["ci"], k, restart=case["m"], rtol=RTOL)
        st["g"] = _rand(seed, 4, n).to(st["rp"].device)
        return st
    if kind in ("refactor", "apply", "iilu", "gmres", "bicgstab"):
        S = P.symbolic(st["rp"], st["ci"], k)
        st["F"] = P.numeric(S, st["v"])
        st["S"] = S
    if kind == "refactor":  # the next step's values: the first ones, perturbed
        st["v"] = st["v"] * (1.0 + _rand(seed, 5, st["v"].numel(), 0.0, 0.01)).to(st["v"].device)
    if kind in ("apply", "iilu"):
        st["p"] = _rand(seed, 6, n).to(st["rp"].device)
    if case.get("prec") == "iilu":
        st["M"] = P.iiluk_build(st["F"])
    return st


def _prepare_batch(case, seed, st):
    N, k = case["N"], case["k"]
    systems = []
    for t in range(case["sets"]):
        systems.append((N,) + _batch_system(N, seed, t + 1))
    for t, side in enumerate(_batch_shapes(case)):
        systems.append((side,) + _batch_system(side, seed, 1000 + t))
    st["x"] = torch.zeros(sum(pat.n for _, pat, _, _ in systems), dtype=torch.float64,
                          device=_device())
    pats, items, at = {}, [], 0
    for side, pat, v, xs in systems:
        if side not in pats:
            rp = torch.from_numpy(pat.rowptr).to(v.device)
            ci = torch.from_numpy(pat.colind).to(v.device)
            pats[side] = (rp, ci, P.symbolic(rp, ci, k))
        rp, ci, S = pats[side]
        items.append((S, v, _matvec(rp, ci, v, xs), st["x"][at:at + pat.n]))
        at += pat.n
    st["batch"] = P.BatchSolve(items, restart=case["m"], rtol=RTOL)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "solve":
        x, info = P.solve(st["rp"], st["ci"], st["v"], st["b"], k=case["k"], restart=case["m"],
                          rtol=RTOL)
        return [x, info.iters]
    if kind == "setup":
        S = P.symbolic(st["rp"], st["ci"], case["k"])
        F = P.numeric(S, st["v"])
        return list(S.pattern()) + [F.values()]
    if kind == "refactor":
        st["F"].refactor(st["v"])
        return [st["F"].values()]
    if kind == "apply":
        return [st["F"].apply(st["p"], transpose=case["transpose"])]
    if kind == "iilu":
        M = P.iiluk_build(st["F"])
        return [M.values(), M.apply(st["p"])]
    if kind in ("gmres", "bicgstab"):
        prec = st["M"] if case["prec"] == "iilu" else st["F"]
        if kind == "gmres":
            x, info = P.gmres(st["rp"], st["ci"], st["v"], st["b"], prec, restart=case["m"],
                              rtol=RTOL)
        else:
            x, info = P.bicgstab(st["rp"], st["ci"], st["v"], st["b"], prec, rtol=RTOL)
        return [x, info.iters]
    if kind == "batch":
        st["batch"].solve()
        return [st["x"], np.array([r.iters for r in st["batch"].results()])]
    v = st["v"].detach().requires_grad_(True)
    b = st["b"].detach().requires_grad_(True)
    x = st["solver"].solve(v, b)
    x.backward(st["g"])
    return [x.detach(), v.grad, b.grad]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _rows(case):
    return {"g2": case["N"] ** 2, "band": case["N"]}.get(case["grid"], case["N"] ** 3)


def _iters(case):
    """Rough iteration counts: grids grow with their side, the band does not."""
    if case["grid"] == "band":
        return (7, 5, 4, 3)[case["k"]] * (2 if case.get("prec") == "iilu" else 1)
    per = {"g2": 0.3, "g3": 0.4, "p27": 0.5}[case["grid"]]
    return max(5, int(per * case["N"] * (2.5 if case.get("prec") == "iilu" else 1.0)))


def _phase_work(case):
    """(bytes, flops) of: the pattern, a numeric phase, an application, an iteration."""
    n, k = _rows(case), case["k"]
    za, zf = n * ROW_A[case["grid"]], n * ROW_F[case["grid"]][k]
    half = ROW_F[case["grid"]][k] / 2.0
    sym = (4 * za + 8 * n + 5 * zf + 16 * n, 0)
    num = (12 * za + 12 * zf + 24 * n, n * (half + 2 * half * half / 2))
    app = (12 * zf + 24 * n, 2 * zf)
    its = _iters(case)
    basis = min(its, case.get("m", 2))
    step = (app[0] + 12 * za + 8 * n + 8 * n * (basis / 2 + 2),
            app[1] + 2 * za + 4 * n * (basis / 2 + 2))
    return sym, num, app, step


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0, "flops": 0}
        for side, cnt in ((case["N"], case["sets"]), (case["N"] * 7 // 8, case["uneven"])):
            w = work(dict(case, kind="solve", N=side, m=case["m"]))
            total = {q: total[q] + cnt * w[q] for q in total}
        return total
    sym, num, app, step = _phase_work(case)
    its = _iters(case)
    parts = {"setup": [(sym, 1), (num, 1)], "refactor": [(num, 1)], "apply": [(app, 1)],
             "iilu": [(num, 1), (app, 1)], "gmres": [(step, its)],
             "bicgstab": [(step, 2 * its)], "solve": [(sym, 1), (num, 1), (step, its)],
             "adjoint": [(num, 1), (step, 2 * its)]}[kind]
    return {"bytes": int(sum(w[0] * c for w, c in parts)),
            "flops": int(sum(w[1] * c for w, c in parts))}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


# ---------------------------------------------------------------------------
# The same results in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _pattern_plain(rp, ci, n, k):
    """Keys i * n + j (ascending) of the entries of level <= k: an entry of level
    p comes from two entries (i, h), (h, j), h < min(i, j), whose levels sum to
    p - 1."""
    rows = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
    key = rows * n + ci.long()
    lev = torch.zeros_like(key)
    for p in range(1, k + 1):
        i, j = key // n, key % n
        low = torch.nonzero(j < i).squeeze(1)
        first = torch.searchsorted(key, j[low] * n + j[low] + 1)
        cnt = torch.searchsorted(key, (j[low] + 1) * n) - first
        src = torch.repeat_interleave(low, cnt)
        at = torch.arange(src.numel(), device=key.device) - torch.repeat_interleave(
            torch.cumsum(cnt, 0) - cnt, cnt) + torch.repeat_interleave(first, cnt)
        hit = lev[src] + lev[at] + 1 == p
        new = torch.unique(i[src[hit]] * n + j[at[hit]])
        pos = torch.searchsorted(key, new).clamp(max=key.numel() - 1)
        new = new[key[pos] != new]
        key, order = torch.sort(torch.cat([key, new]))
        lev = torch.cat([lev, torch.full_like(new, p)])[order]
    return key


def _levels_plain(n, i, j):
    """Depth of every row when row i waits for rows j."""
    depth = torch.zeros(n, dtype=torch.int64, device=i.device)
    while True:
        d = depth.clone()
        d.scatter_reduce_(0, i, depth[j] + 1, "amax")
        if torch.equal(d, depth):
            return depth
        depth = d


def _expand(first, cnt):
    own = torch.repeat_interleave(torch.arange(cnt.numel(), device=cnt.device), cnt)
    return own, (torch.arange(own.numel(), device=cnt.device) -
                 (torch.cumsum(cnt, 0) - cnt)[own] + first[own])


class _Plain:
    """ILU(k) by rows of equal depth."""

    def __init__(self, rp, ci, v, k):
        self.n = n = rp.numel() - 1
        self.key = _pattern_plain(rp, ci, n, k)
        self.i, self.j = self.key // n, self.key % n
        rows = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
        self.val = torch.zeros(self.key.numel(), dtype=torch.float64, device=rp.device)
        self.val[torch.searchsorted(self.key, rows * n + ci.long())] = v
        ar = torch.arange(n + 1, device=rp.device)
        self.ptr = torch.searchsorted(self.key, ar * n)
        self.diag = torch.searchsorted(self.key, ar[:-1] * n + ar[:-1])
        low, up = self.j < self.i, self.j > self.i
        self.order = {}
        for name, sel in (("fwd", low), ("bwd", up)):
            depth = _levels_plain(n, self.i[sel], self.j[sel])
            idx = torch.argsort(depth, stable=True)
            cuts = torch.cumsum(torch.bincount(depth), 0).cpu().tolist()
            self.order[name] = [idx[a:b] for a, b in zip([0] + cuts[:-1], cuts)]

    def factor(self):
        n, key, j, val = self.n, self.key, self.j, self.val
        for r in self.order["fwd"]:
            nl = self.diag[r] - self.ptr[r]
            for q in range(int(nl.max())):
                at = (self.ptr[r] + q)[nl > q]
                h = j[at]
                val[at] = val[at] / val[self.diag[h]]
                own, src = _expand(self.diag[h] + 1, self.ptr[h + 1] - self.diag[h] - 1)
                want = self.i[at][own] * n + j[src]
                pos = torch.searchsorted(key, want).clamp(max=key.numel() - 1)
                ok = key[pos] == want
                val[pos[ok]] -= val[at][own][ok] * val[src[ok]]
        return self

    def _sum(self, r, first, cnt, x, mat):
        own, at = _expand(first, cnt)
        out = torch.zeros(r.numel(), dtype=torch.float64, device=x.device)
        return out.index_add_(0, own, mat[at] * x[self.j[at]])

    def solve(self, p):
        x = p.clone()
        for r in self.order["fwd"]:
            x[r] -= self._sum(r, self.ptr[r], self.diag[r] - self.ptr[r], x, self.val)
        for r in self.order["bwd"]:
            x[r] = (x[r] - self._sum(r, self.diag[r] + 1, self.ptr[r + 1] - self.diag[r] - 1, x,
                                     self.val)) / self.val[self.diag[r]]
        return x

    def solve_t(self, p):
        """U^T then L^T: a column's value is known once its row is; scattered on."""
        x = p.clone()
        for r in reversed(self.order["bwd"]):
            x[r] = x[r] / self.val[self.diag[r]]
            own, at = _expand(self.diag[r] + 1, self.ptr[r + 1] - self.diag[r] - 1)
            x.index_add_(0, self.j[at], -self.val[at] * x[r][own])
        for r in reversed(self.order["fwd"]):
            own, at = _expand(self.ptr[r], self.diag[r] - self.ptr[r])
            x.index_add_(0, self.j[at], -self.val[at] * x[r][own])
        return x


def _block_solve(rp, ci, v, b, N, transpose):
    """A x = b (or A^T x = b) for a 2D grid: block tridiagonal elimination."""
    n = N * N
    rows = torch.repeat_interleave(torch.arange(n, device=rp.device), rp[1:] - rp[:-1])
    cols = ci.long()
    if transpose:
        rows, cols = cols, rows
    B = torch.zeros(3, N, N, N, dtype=torch.float64, device=rp.device)
    B[cols // N - rows // N + 1, rows // N, rows % N, cols % N] = v
    y, D = [], []
    for t in range(N):
        d, r = B[1, t], b[t * N:(t + 1) * N]
        if t:
            f = torch.linalg.solve(D[-1], torch.cat([B[2, t - 1], y[-1][:, None]], dim=1))
            d, r = d - B[0, t] @ f[:, :N], r - B[0, t] @ f[:, N]
        D.append(d)
        y.append(r)
    x = [None] * N
    for t in reversed(range(N)):
        r = y[t] if t == N - 1 else y[t] - B[2, t] @ x[t + 1]
        x[t] = torch.linalg.solve(D[t], r)
    return torch.cat(x)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "gmres", "bicgstab"):
        return [_system(case, seed)[3], None]
    if kind == "batch":
        xs = [_batch_system(case["N"], seed, t + 1)[2] for t in range(case["sets"])]
        xs += [_batch_system(s, seed, 1000 + t)[2]
               for t, s in enumerate(_batch_shapes(case))]
        return [torch.cat(xs), None]
    if kind == "adjoint":
        rp, ci, v, xs, b = _system(case, seed)
        g = _rand(seed, 4, xs.numel()).to(xs.device)
        x = _block_solve(rp, ci, v, b, case["N"], False)
        lam = _block_solve(rp, ci, v, g, case["N"], True)
        rows = torch.repeat_interleave(torch.arange(xs.numel(), device=xs.device),
                                       rp[1:] - rp[:-1])
        return [x, -lam[rows] * x[ci.long()], lam]
    if case["grid"] == "band" or kind == "iilu":
        return None  # thousands of levels of a few rows each: minutes row by row
    rp, ci, v = _matrix(case, seed)
    if kind == "refactor":
        v = v * (1.0 + _rand(seed, 5, v.numel(), 0.0, 0.01)).to(v.device)
    F = _Plain(rp, ci, v, case["k"]).factor()
    if kind == "setup":
        return [None, None, None, None, F.val]  # the pattern: whole numbers
    if kind == "refactor":
        return [F.val]
    p = _rand(seed, 6, F.n).to(v.device)
    return [F.solve_t(p) if case["transpose"] else F.solve(p)]
