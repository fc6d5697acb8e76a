"""The work that users of this framework have it do, as timed cases.

Each case is one pass through a public entry point of paper_2111_09512_gb300
on a matrix of the kinds the repository works with, made here from the seed:
7-point Poisson, cut-cell-like 7-point pressure operators (density jumps and
cut volume fractions) and 27-point operators on a perturbed hex lattice, from
sizes that stay in L2 to sizes of several million rows, cubes and uneven
boxes.  `exact` restates the result in plain 64-bit torch: ILU(0) by
iterating its defining equations on the stencil to their fixed point, ILUT
(small systems) row by row, the sweeps, the exact solves and flexible GMRES.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2111_09512_gb300 as silu

DEV = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # one application on a small system with several interleaved right-hand
        # sides (velocity components and a scalar); everything stays in L2
        dict(name="smooth_poisson32_r4", path="smooth", kind="poisson7", nx=32, ny=32, nz=32, factor="ilu0", prec="fp64",
             nrhs=4, sweeps_L=5, sweeps_U=5, scale="row"),
        # the paper's smallest PeleLM size (about 14 thousand rows) with ILUT: launches and latency count
        dict(name="smooth_cutcell24_ilut", path="smooth", kind="cutcell7", nx=24, ny=24, nz=24, factor="ilut", prec="fp64",
             nrhs=1, sweeps_L=10, sweeps_U=10, scale="row"),
        # the benchmark's workload: 2.1M rows, ILUT(1e-3, 10), 20 Richardson terms
        dict(name="smooth_cutcell128_ilut", path="smooth", kind="cutcell7", nx=128, ny=128, nz=128, factor="ilut",
             prec="fp64", nrhs=1, sweeps_L=10, sweeps_U=10, scale="row"),
        # the 27-point mesh operator with FP32 factors and sweeps, 110M entries
        dict(name="smooth_hex160_fp32", path="smooth", kind="hex27", nx=160, ny=160, nz=160, factor="ilu0", prec="fp32",
             nrhs=1, sweeps_L=3, sweeps_U=3, scale="row"),
        # three velocity components at once on an uneven box (columns split 2 + 1)
        dict(name="smooth_cutcell_box_r3", path="smooth", kind="cutcell7", nx=101, ny=97, nz=89, factor="ilu0",
             prec="fp64", nrhs=3, sweeps_L=10, sweeps_U=10, scale="row"),
        # the comparison path: exact level-ordered triangular solves
        dict(name="direct_cutcell96", path="direct", kind="cutcell7", nx=96, ny=96, nz=96, factor="ilu0", prec="fp64",
             nrhs=1),
        # a small pressure solve to 1e-8, as the solve server runs many of
        dict(name="fgmres_poisson32", path="fgmres", kind="poisson7", nx=32, ny=32, nz=32, factor="ilu0", prec="fp64",
             sweeps_L=5, sweeps_U=5, tol=1e-8, maxit=1000),
        # a mid-size 27-point solve with a fixed budget of two restart cycles, FP32 factors
        dict(name="fgmres_hex96_fp32", path="fgmres", kind="hex27", nx=96, ny=96, nz=96, factor="ilu0", prec="fp32",
             sweeps_L=3, sweeps_U=3, tol=1e-14, maxit=60),
        # one AMG V-cycle, the finest level smoothed by FP32 ILU(0) sweeps
        dict(name="vcycle_cutcell128_fp32", path="vcycle", kind="cutcell7", nx=128, ny=128, nz=128, factor="ilu0",
             prec="fp32", sweeps_L=5, sweeps_U=5),
        # many independent systems of uneven size (edges 8 to 64) in one batch
        dict(name="batch48_smooth_fp32", path="batch_smooth", kind="cutcell7", count=48, sizes=3, factor="ilu0", prec="fp32",
             sweeps_L=3, sweeps_U=3),
        # the batched solver, one restart cycle
        dict(name="batch24_fgmres_fp32", path="batch_fgmres", kind="cutcell7", count=24, sizes=4, factor="ilu0", prec="fp32",
             sweeps_L=5, sweeps_U=5, maxit=20),
        # the ILUT Schur complement smoother over eight row blocks
        dict(name="schur_hex64_p8", path="schur", kind="hex27", nx=64, ny=64, nz=64, factor="ilut", prec="fp64", parts=8,
             sweeps_L=3, sweeps_U=3),
    ]


def _edges(rng, lo, hi):
    """Three edges of a box spread over the logarithm of [lo, hi], uneven about half of the time."""
    e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.4:
        n = int(round(e))
        return n, n, n
    return tuple(max(lo, min(hi, int(round(e * rng.uniform(0.8, 1.2))))) for _ in range(3))


def draw(rng):
    path = rng.choice(["smooth"] * 6 + ["direct", "fgmres", "fgmres", "vcycle", "batch_smooth", "batch_fgmres", "schur"])
    prec = rng.choice(["fp64", "fp32"])
    if path in ("batch_smooth", "batch_fgmres"):
        c = dict(path=path, kind="cutcell7", count=rng.randint(3, 40 if path == "batch_smooth" else 20),
                 sizes=rng.randint(100, 10_000), factor="ilu0", prec=prec, sweeps_L=rng.randint(2, 6), sweeps_U=rng.randint(2, 6))
        if path == "batch_fgmres":
            c["maxit"] = rng.randint(5, 20)
        return c
    kind = rng.choice(["poisson7", "cutcell7", "cutcell7", "hex27"])
    top = {"smooth": 120, "direct": 80, "fgmres": 96, "vcycle": 96, "schur": 48}[path]
    nx, ny, nz = _edges(rng, 12, top)
    factor = "ilu0"
    if path == "schur" or (path in ("smooth", "fgmres") and nx * ny * nz <= 300_000 and rng.random() < 0.4):
        factor = "ilut"
    c = dict(path=path, kind=kind, nx=nx, ny=ny, nz=nz, factor=factor, prec=prec)
    if path == "smooth":
        c.update(nrhs=rng.choice([1, 1, 1, 2, 3, 4, 5, 8]), sweeps_L=rng.randint(2, 10), sweeps_U=rng.randint(2, 10),
                 scale=rng.choice(["row", "row", "row", "rowcol"]))
    elif path == "direct":
        c.update(nrhs=rng.choice([1, 1, 2, 4]))
    else:
        c.update(sweeps_L=rng.randint(2, 6), sweeps_U=rng.randint(2, 6))
        if path == "fgmres":
            c.update(tol=1e-14, maxit=rng.randint(10, 45))
        if path == "schur":
            c.update(parts=rng.choice([4, 8, 16]))
    return c


TAU, FILL = 1e-3, 10  # ILUT(1e-3, 10)


# ------------------------------------------------------------------ matrices

OFF7 = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)]
OFF27 = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _at(P, d, shape):
    """The entries at offset d from every point of a field padded by one layer on each side."""
    nz, ny, nx = shape
    return P[1 + d[0]:1 + d[0] + nz, 1 + d[1]:1 + d[1] + ny, 1 + d[2]:1 + d[2] + nx]


def _pad(t, fill=0.0):
    return torch.nn.functional.pad(t, (1, 1, 1, 1, 1, 1), value=fill)


def stencil(kind, nx, ny, nz, seed):
    """(offsets in column order, {offset: values (nz, ny, nx)}); 0 where the neighbour lies outside."""
    shape = (nz, ny, nx)
    g = _gen(seed)
    f64 = dict(dtype=torch.float64, device=DEV)
    inside = _pad(torch.ones(shape, **f64))
    if kind == "poisson7":
        return OFF7, {d: (6.0 * torch.ones(shape, **f64) if d == (0, 0, 0) else -_at(inside, d, shape)) for d in OFF7}
    if kind == "cutcell7":
        rho = torch.exp(2.0 * torch.randn(shape, generator=g, **f64))
        edge = torch.zeros(shape, dtype=torch.bool, device=DEV)
        for ax in range(3):
            edge.select(ax, 0).fill_(True)
            edge.select(ax, shape[ax] - 1).fill_(True)
        cut = edge & (torch.rand(shape, generator=g, **f64) < 0.1)
        vf = torch.where(cut, 10.0 ** (-8.0 * torch.rand(shape, generator=g, **f64)), torch.ones(shape, **f64))
        prho, pvf = _pad(rho, 1.0), _pad(vf, 0.0)
        A, diag = {}, torch.zeros(shape, **f64)
        for d in OFF7:
            if d == (0, 0, 0):
                continue
            face = torch.minimum(vf, _at(pvf, d, shape)) * (2.0 / (rho + _at(prho, d, shape)))
            own = _at(inside, d, shape)
            diag += torch.where(own > 0, face, vf * (2.0 / rho))
            A[d] = -face * own
        A[(0, 0, 0)] = diag
        return OFF7, A
    # 27-point weighted graph Laplacian on a jittered lattice with a ring of fixed outside nodes
    full = (nz + 2, ny + 2, nx + 2)
    c = torch.exp(1.5 * torch.randn(full, generator=g, **f64))
    pos = [torch.arange(full[ax], **f64).reshape([-1 if k == ax else 1 for k in range(3)])
           + 0.5 * torch.rand(full, generator=g, **f64) - 0.25 for ax in range(3)]
    mid = (0, 0, 0)
    A, diag = {}, torch.zeros(shape, **f64)
    for d in OFF27:
        if d == mid:
            continue
        dist = sum((_at(p, d, shape) - _at(p, mid, shape)) ** 2 for p in pos)
        w = torch.sqrt(_at(c, d, shape) * _at(c, mid, shape)) / dist
        diag += w
        A[d] = -w * _at(inside, d, shape)
    A[mid] = diag
    return OFF27, A


def csr(offs, A, nx, ny, nz):
    """Host CSR arrays (columns ascending in each row) of a stencil operator."""
    shape = (nz, ny, nx)
    n = nx * ny * nz
    inside = _pad(torch.ones(shape, dtype=torch.bool, device=DEV), False)
    mask = torch.stack([_at(inside, d, shape).reshape(-1) for d in offs], 1)
    step = torch.tensor([(d[0] * ny + d[1]) * nx + d[2] for d in offs], dtype=torch.int32, device=DEV)
    cols = torch.arange(n, dtype=torch.int32, device=DEV)[:, None] + step[None, :]
    vals = torch.stack([A[d].reshape(-1) for d in offs], 1)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(mask.sum(1), 0)
    return rp.cpu().numpy(), cols[mask].cpu().numpy(), vals[mask].cpu().numpy()


def _matrix(case, seed):
    offs, A = stencil(case["kind"], case["nx"], case["ny"], case["nz"], seed)
    return csr(offs, A, case["nx"], case["ny"], case["nz"])


def _batch_edges(case):
    """The edges of a batch's systems, uniform on 8..64 ("sizes" numbers the mix)."""
    return np.random.RandomState(int(case["sizes"])).randint(8, 65, int(case["count"])).tolist()


def _vectors(case, seed, n):
    """b uniform on [-1, 1) and, for the smoothers, a nonzero iterate x of the same kind."""
    g = _gen(int(seed) + 7919)
    nrhs = int(case.get("nrhs", 1))
    size = (n,) if nrhs == 1 else (n, nrhs)
    b = 2.0 * torch.rand(size, generator=g, dtype=torch.float64, device=DEV) - 1.0
    x = 2.0 * torch.rand(size, generator=g, dtype=torch.float64, device=DEV) - 1.0
    return b, x


# ---------------------------------------------------------------- the passes

def prepare(case, seed):
    path = case["path"]
    prec = silu.FP32 if case["prec"] == "fp32" else silu.FP64
    ctx = silu.Context(0, torch.cuda.current_stream())
    if path in ("batch_smooth", "batch_fgmres"):
        systems = []
        for k, e in enumerate(_batch_edges(case)):
            offs, A = stencil(case["kind"], e, e, e, int(seed) + 1000 * (k + 1))
            systems.append(csr(offs, A, e, e, e))
        B = silu.Batch(ctx, systems, case["factor"], prec=prec)
        b, x = _vectors(case, seed, B.n)
        return dict(case=case, B=B, b=b, x=x)
    M = silu.silu_mat_create(ctx, *_matrix(case, seed))
    tau, fill = (TAU, FILL) if case["factor"] == "ilut" else (0.0, 0)
    scale = silu.SCALE_ROWCOL if case.get("scale") == "rowcol" else silu.SCALE_ROW
    if path == "schur":  # the smoother keeps ILUT factors of its interior blocks; the handle itself needs only ILU(0)
        F = silu.ilu_setup(ctx, M, "ilu0", prec=prec)
        F.schur_setup(int(case["parts"]), TAU, FILL)
        F.schur_set_interface_prec(silu.SCHUR_IFACE_DIAG)
    else:
        F = silu.ilu_setup(ctx, M, case["factor"], tau=tau, fill=fill, scale=scale, prec=prec)
    if path == "vcycle":
        F.amg_setup(theta=0.25, coarse_size=400)
    F.reserve(int(case.get("nrhs", 1)), 30 if path == "fgmres" else 0)
    b, x = _vectors(case, seed, F.n)
    return dict(case=case, F=F, b=b, x=x)


def run(state):
    c, b, x = state["case"], state["b"], state["x"]
    path = c["path"]
    if path == "smooth":
        silu.ilu_smooth(state["F"], x, b, c["sweeps_L"], c["sweeps_U"])
        return x
    if path == "direct":
        silu.direct_trisolve(state["F"], x, b)
        return x
    if path == "fgmres":
        x.zero_()
        _, its, rel = silu.fgmres_solve(state["F"], x, b, tol=c["tol"], restart=30, maxit=c["maxit"],
                                        sweeps_L=c["sweeps_L"], sweeps_U=c["sweeps_U"])
        return [x, its, rel]
    if path == "vcycle":
        state["F"].amg_vcycle(x, b, c["sweeps_L"], c["sweeps_U"])
        return x
    if path == "batch_smooth":
        silu.silu_batch_smooth(state["B"], x, b, c["sweeps_L"], c["sweeps_U"])
        return x
    if path == "batch_fgmres":
        x.zero_()
        _, its, rel = silu.silu_batch_fgmres(state["B"], x, b, tol=1e-14, restart=20, maxit=c["maxit"],
                                             sweeps_L=c["sweeps_L"], sweeps_U=c["sweeps_U"])
        return [x, its, rel]
    state["F"].schur_smooth(x, b, c["sweeps_L"], c["sweeps_U"])
    return x


def work(case):
    """Every matrix and vector that a pass needs read once, its result written once; two flops per entry and use."""
    path = case["path"]
    if path in ("batch_smooth", "batch_fgmres"):
        n = sum(e ** 3 for e in _batch_edges(case))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    per_row = 27.0 if case["kind"] == "hex27" else 7.0
    nnz_a = per_row * n
    side = (per_row - 1) / 2 * n if case["factor"] == "ilu0" else (8.0 if case["kind"] != "hex27" else 10.0) * n
    vb = 4 if case["prec"] == "fp32" else 8
    factors = 2 * (side * (vb + 4) + 4 * n)
    a_bytes = nnz_a * 12 + 4 * n
    R = case.get("nrhs", 1)
    mL, mU = case.get("sweeps_L", 1), case.get("sweeps_U", 1)
    sweeps = 2.0 * ((mL - 1) + (mU - 1)) * side * R
    if path == "smooth" or path == "batch_smooth":
        return dict(bytes=a_bytes + factors + 8 * n + 24 * n * R, flops=2 * nnz_a * R + sweeps)
    if path == "direct":
        return dict(bytes=nnz_a * 12 + 4 * n + 2 * (side * 12 + 4 * n) + 8 * n + 24 * n * R,
                    flops=2 * nnz_a * R + 4 * side * R)
    if path in ("fgmres", "batch_fgmres"):
        its = min(case["maxit"], 50)
        # a basis vector and a preconditioned vector per iteration, each written once and read once at the end
        return dict(bytes=a_bytes + factors + 8 * n + 16 * n + its * 32.0 * n,
                    flops=its * (2 * nnz_a + sweeps + 4.0 * n * min(its, 30)))
    if path == "vcycle":
        return dict(bytes=2.5 * a_bytes + factors + 8 * n + 24 * n, flops=2 * (2 * nnz_a + sweeps) + 8 * nnz_a)
    return dict(bytes=2 * a_bytes + factors + 8 * n + 24 * n, flops=4 * nnz_a + 3 * sweeps)


# ------------------------------------------------------- 64-bit restatements

class _Stencil:
    """A stencil operator and its ILU(0) in plain 64-bit torch."""

    def __init__(self, kind, nx, ny, nz, seed):
        self.shape = (nz, ny, nx)
        self.n = nx * ny * nz
        self.levels = 4 * (nx + 2 * ny + 4 * nz)
        self.offs, self.A = stencil(kind, nx, ny, nz, seed)
        self._factor()

    def _factor(self):
        mid = (0, 0, 0)
        offs, A, sh = self.offs, self.A, self.shape
        have = set(offs)
        low, up = [d for d in offs if d < mid], [d for d in offs if d > mid]
        P = {d: _pad(A[d], 1.0 if d == mid else 0.0) for d in offs}  # L below, U from the diagonal up, padded
        for d in low:
            _at(P[d], mid, sh).copy_(A[d] / _at(P[mid], d, sh))
        add = lambda a, b: (a[0] + b[0], a[1] + b[1], a[2] + b[2])  # noqa: E731
        terms = {d: [(e, f) for e in low for f in up if add(e, f) == d] for d in have}
        # l_ij u_jj = a_ij - sum l_ik u_kj and u_ij = a_ij - sum l_ik u_kj, iterated in column order until nothing
        # changes; row i depends on earlier rows alone, so it is exact after as many rounds as there are levels
        for it in range(self.levels):
            moved = torch.zeros((), dtype=torch.float64, device=DEV)
            for d in offs:
                s = A[d].clone()
                for e, f in terms[d]:
                    s.addcmul_(_at(P[e], mid, sh), _at(P[f], e, sh), value=-1.0)
                if d < mid:
                    s /= _at(P[mid], d, sh)
                if d == mid:
                    moved = ((s - _at(P[d], mid, sh)).abs() / s.abs()).max()
                _at(P[d], mid, sh).copy_(s)
            if it % 4 == 3 and float(moved) < 1e-16:
                break
        self.d = _at(P[mid], mid, sh).clone()
        self.L = {d: _at(P[d], mid, sh).clone() for d in low}
        self.U = {d: _at(P[d], mid, sh) / self.d for d in up}

    def _sum(self, T, v):
        out = torch.zeros(self.shape, dtype=torch.float64, device=DEV)
        p = _pad(v)
        for d, t in T.items():
            out.addcmul_(t, _at(p, d, self.shape))
        return out

    def mul(self, v):
        return self._sum(self.A, v.reshape(self.shape)).reshape(-1)

    def apply(self, r, mL, mU):
        """m_L + m_U Richardson terms on r."""
        r = r.reshape(self.shape)
        y = r
        for _ in range(mL - 1):
            y = r - self._sum(self.L, y)
        c = y / self.d
        v = c
        for _ in range(mU - 1):
            v = c - self._sum(self.U, v)
        return v.reshape(-1)

    def solve(self, r):
        """U^{-1} L^{-1} r: the same terms until they no longer change (the strict triangles are nilpotent)."""
        def until(T, c):
            v = c
            for it in range(self.levels):
                nxt = c - self._sum(T, v)
                if it % 8 == 7 and bool((nxt == v).all()):
                    break
                v = nxt
            return v
        return until(self.U, until(self.L, r.reshape(self.shape)) / self.d).reshape(-1)


def _fgmres(S, b, x, tol, restart, maxit, mL, mU):
    """Flexible GMRES with modified Gram-Schmidt and Givens rotations; (x, iterations, true relative residual)."""
    bnorm = float(b.norm())
    its = 0
    while True:
        r = b - S.mul(x)
        beta = float(r.norm())
        if beta / bnorm <= tol or its >= maxit:
            return x, its, beta / bnorm
        V, Z = [r / beta], []
        H = np.zeros((restart + 1, restart))
        g = np.zeros(restart + 1)
        g[0] = beta
        rot = []
        for j in range(restart):
            z = S.apply(V[j], mL, mU)
            w = S.mul(z)
            Z.append(z)
            hs = []
            for i in range(j + 1):
                h = torch.dot(w, V[i])
                w = w - h * V[i]
                hs.append(h)
            hs.append(w.norm())
            col = torch.stack(hs).cpu().numpy()
            V.append(w / hs[-1])
            for i, (c, s) in enumerate(rot):
                col[i], col[i + 1] = c * col[i] + s * col[i + 1], -s * col[i] + c * col[i + 1]
            den = math.hypot(col[j], col[j + 1])
            c, s = col[j] / den, col[j + 1] / den
            rot.append((c, s))
            H[:j, j] = col[:j]
            H[j, j] = den
            g[j + 1] = -s * g[j]
            g[j] = c * g[j]
            its += 1
            if abs(g[j + 1]) <= tol * bnorm or its >= maxit:
                break
        k = len(Z)
        y = np.linalg.solve(np.triu(H[:k, :k]), g[:k])
        for i in range(k):
            x = x + float(y[i]) * Z[i]


def _ilut(rp, ci, va, tau, fill):
    """Row-by-row ILUT with dual threshold (relative to the row's 2-norm), pivoting off: rows of L and U as dicts."""
    rp, ci, va = rp.tolist(), ci.tolist(), va.tolist()
    L, U = [], []
    for i in range(len(rp) - 1):
        w = {ci[p]: va[p] for p in range(rp[i], rp[i + 1])}
        ti = tau * math.sqrt(sum(va[p] * va[p] for p in range(rp[i], rp[i + 1])))
        todo = sorted(j for j in w if j < i)
        kept = {}
        while todo:
            k = todo.pop(0)
            wk = w.pop(k) / U[k][k]
            if abs(wk) < ti:
                continue
            kept[k] = wk
            fresh = False
            for j, u in U[k].items():
                if j == k:
                    continue
                if j not in w:
                    w[j] = 0.0
                    if j < i:
                        todo.append(j)
                        fresh = True
                w[j] -= wk * u
            if fresh:
                todo.sort()
        most = lambda d: dict(sorted(sorted(d.items(), key=lambda t: (-abs(t[1]), t[0]))[:fill]))  # noqa: E731
        low = most({j: v for j, v in kept.items() if abs(v) >= ti})
        upper = most({j: v for j, v in w.items() if j > i and abs(v) >= ti})
        L.append(low)
        U.append({i: w[i], **upper})
    return L, U


def _dict_rows(rows, n):
    at = [(i, j, v) for i, row in enumerate(rows) for j, v in row.items()]
    idx = torch.tensor([[a[0] for a in at], [a[1] for a in at]], dtype=torch.int64)
    return torch.sparse_coo_tensor(idx, torch.tensor([a[2] for a in at], dtype=torch.float64), (n, n)).coalesce()


def _smooth_ilut(case, seed, b, x):
    rp, ci, va = _matrix(case, seed)
    n = len(rp) - 1
    L, U = _ilut(rp, ci, va, TAU, FILL)
    d = torch.tensor([U[i][i] for i in range(n)], dtype=torch.float64)[:, None]
    T = _dict_rows(L, n)
    S = _dict_rows([{j: v / U[i][i] for j, v in U[i].items() if j != i} for i in range(n)], n)
    A = torch.sparse_coo_tensor(torch.stack([torch.from_numpy(np.repeat(np.arange(n), np.diff(rp))),
                                             torch.from_numpy(ci.astype(np.int64))]), torch.from_numpy(va), (n, n))
    xs, r = x.cpu().reshape(n, -1), b.cpu().reshape(n, -1)
    r = r - torch.sparse.mm(A, xs)
    y = r
    for _ in range(case["sweeps_L"] - 1):
        y = r - torch.sparse.mm(T, y)
    c = y / d
    v = c
    for _ in range(case["sweeps_U"] - 1):
        v = c - torch.sparse.mm(S, v)
    return (xs + v).reshape(x.shape)


def exact(case, seed):
    path = case["path"]
    if path in ("vcycle", "schur"):  # their hierarchies and ILUT blocks take minutes in plain Python
        return None
    if path in ("batch_smooth", "batch_fgmres"):
        edges = _batch_edges(case)
        n = sum(e ** 3 for e in edges)
        b, x = _vectors(case, seed, n)
        xs, rels, at = [], [], 0
        for k, e in enumerate(edges):
            S = _Stencil(case["kind"], e, e, e, int(seed) + 1000 * (k + 1))
            bk, xk = b[at:at + S.n], x[at:at + S.n]
            at += S.n
            if path == "batch_smooth":
                xs.append(xk + S.apply(bk - S.mul(xk), case["sweeps_L"], case["sweeps_U"]))
            else:
                xk, _, rel = _fgmres(S, bk, torch.zeros_like(bk), 1e-14, 20, case["maxit"], case["sweeps_L"],
                                     case["sweeps_U"])
                xs.append(xk)
                rels.append(rel)
        return torch.cat(xs) if path == "batch_smooth" else [torch.cat(xs), None, np.array(rels)]
    n = case["nx"] * case["ny"] * case["nz"]
    b, x = _vectors(case, seed, n)
    if case["factor"] == "ilut":
        if path != "smooth" or n > 16_000:
            return None
        return _smooth_ilut(case, seed, b, x)
    S = _Stencil(case["kind"], case["nx"], case["ny"], case["nz"], seed)
    if path == "fgmres":
        x, _, rel = _fgmres(S, b, torch.zeros_like(b), case["tol"], 30, case["maxit"], case["sweeps_L"],
                            case["sweeps_U"])
        return [x, None, rel]
    out = torch.empty_like(x).reshape(n, -1)
    bb, xx = b.reshape(n, -1), x.reshape(n, -1)
    for k in range(out.shape[1]):
        r = bb[:, k] - S.mul(xx[:, k])
        out[:, k] = xx[:, k] + (S.solve(r) if path == "direct" else S.apply(r, case["sweeps_L"], case["sweeps_U"]))
    return out.reshape(x.shape)
