"""Performance cases: the calls a user of the library makes, through its public Python API.

Three kinds of work: applying a relaxation (as a smoother or as a preconditioner of one's own
Krylov method), applying the multigrid cycle, and solving systems (GMRES, CG, packs of small
systems).  Matrices are the model problems the library is meant for -- 5- and 7-point Laplacians,
Poisson problems with lognormal coefficients, upwind convection-diffusion, Q1 elasticity -- and
unstructured matrices with uneven rows.  They are built here on the GPU, so the reference values of
exact() do not depend on the library.
"""
import math

import numpy as np
import torch

import paper_2104_01196_gb300 as gs2

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one symmetric sweep on a small grid (a coarse solver's smoother, a
        # small subdomain's preconditioner), where launches and latency are all there is
        _apply("apply-laplace2d-64", "laplace2d", 64, "symmetric", inner=1),
        # a smoother in lower precision on mechanics: long rows (up to 81 entries) of interleaved
        # unknowns, damped, two inner sweeps, FP32 triangles
        _apply("apply-elastic-40-fp32", "elastic", 40, "symmetric", inner=2, omega=0.8,
               precision="fp32"),
        # a preconditioner apply on an unstructured matrix of uneven, unsorted rows, odd size
        _apply("apply-ragged-300007", "ragged", 300007, "symmetric", inner=1),
        # the whole sweep in single precision on a large transport problem
        _apply("apply-convdiff-150-fp32sweep", "convdiff3d", 150, "symmetric", inner=1,
               precision="fp32_sweep"),
        # exact Gauss-Seidel by triangular solves, the baseline every GS2 user compares with
        dict(name="gs-laplace3d-100", op="gs", matrix="laplace3d", size=100,
             direction="symmetric", omega=1.0),
        # multicolour Gauss-Seidel with over-relaxation on an odd grid
        dict(name="mtgs-convdiff-127", op="mtgs", matrix="convdiff3d", size=127,
             direction="symmetric", omega=1.1),
        # one multigrid cycle with the GS2 smoother, as a preconditioner of one's own solver
        dict(name="amg-poisson3d-80", op="amg", matrix="poisson3d", size=80,
             direction="symmetric"),
        # a small system solved to tolerance (an inner solve, a request of a service)
        _gmres("gmres-laplace2d-64", "laplace2d", 64, "forward", 1e-8),
        # an ordinary solve: a middle-sized transport problem
        _gmres("gmres-convdiff-57", "convdiff3d", 57, "symmetric", 1e-8),
        # the largest: the benchmark's problem on a 160^3 grid (n = 4.1M)
        _gmres("gmres-convdiff-160", "convdiff3d", 160, "symmetric", 1e-8),
        # conjugate gradients on a large symmetric problem
        dict(name="cg-laplace3d-110", op="cg", matrix="laplace3d", size=110, tol=1e-8),
        # many small uneven systems at once
        dict(name="pack-48", op="pack", count=48, low=1000, high=16000, tol=1e-8),
    ]


def _apply(name, matrix, size, direction, inner, omega=1.0, precision="fp64"):
    c = dict(op="apply", matrix=matrix, size=size, direction=direction, inner=inner, omega=omega,
             precision=precision)
    return dict(c, name=name) if name else c


def _gmres(name, matrix, size, direction, tol):
    c = dict(op="gmres", matrix=matrix, size=size, direction=direction, tol=tol, restart=30)
    return dict(c, name=name) if name else c


def _size(rng, low, high):
    """Log-uniform, every residue as likely as another."""
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "gs", "mtgs", "amg", "gmres", "gmres", "cg",
                     "pack"])
    if op == "apply":
        matrix = rng.choice(["laplace2d", "laplace3d", "convdiff3d", "elastic", "ragged"])
        low, high = {"laplace2d": (20, 1500), "laplace3d": (10, 150), "convdiff3d": (10, 150),
                     "elastic": (6, 40), "ragged": (1000, 500000)}[matrix]
        return _apply(None, matrix, _size(rng, low, high),
                      rng.choice(["forward", "backward", "symmetric"]), rng.choice([1, 1, 2, 3]),
                      0.8 if matrix == "elastic" else rng.choice([1.0, 0.9]),
                      rng.choice(["fp64", "fp64", "fp32", "fp16", "fp32_sweep"]))
    if op in ("gs", "mtgs"):
        matrix = rng.choice(["laplace2d", "laplace3d", "convdiff3d"])
        low, high = (20, 700) if matrix == "laplace2d" else (10, 127)
        return dict(op=op, matrix=matrix, size=_size(rng, low, high),
                    direction=rng.choice(["forward", "backward", "symmetric"]),
                    omega=rng.choice([1.0, 1.1]))
    if op == "amg":
        return dict(op="amg", matrix=rng.choice(["laplace3d", "poisson3d"]),
                    size=_size(rng, 16, 80), direction="symmetric")
    if op == "gmres":
        matrix = rng.choice(["laplace2d", "convdiff3d", "convdiff3d"])
        return _gmres(None, matrix, _size(rng, *((20, 90) if matrix == "laplace2d" else (12, 150))),
                      rng.choice(["forward", "symmetric"]), rng.choice([1e-6, 1e-8]))
    if op == "cg":
        return dict(op="cg", matrix="laplace3d", size=_size(rng, 12, 110), tol=1e-8)
    return dict(op="pack", count=rng.randint(8, 48), low=1000, high=_size(rng, 2000, 16000),
                tol=1e-8)


# ---------------------------------------------------------------------------
# matrices: (rowptr int64, col int32, val float64) on the GPU
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7fffffffffff)
    return g


def _uniform(n, g):
    """U[-1, 1), the benchmark's right-hand sides and solutions."""
    return 2.0 * torch.rand(n, dtype=F64, device=DEV, generator=g) - 1.0


def _from_slots(mask, cols, vals):
    rp = torch.zeros(mask.shape[0] + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(mask.sum(1), 0, out=rp[1:])
    return rp, cols[mask].to(torch.int32), vals[mask]


def _grid(dims, coef):
    """Rows of a 5- or 7-point operator, x fastest, Dirichlet nodes eliminated, columns ascending.
    coef(d, side) is the entry towards the neighbour in direction d; coef(None, 0) the diagonal."""
    nx, ny, nz = dims
    n = nx * ny * nz
    i = torch.arange(n, device=DEV)
    at, stride, top = (i % nx, i // nx % ny, i // (nx * ny)), (1, nx, nx * ny), dims
    sides = [(d, -1) for d in (2, 1, 0)] + [(None, 0)] + [(d, 1) for d in (0, 1, 2)]
    sides = [(d, s) for d, s in sides if d is None or top[d] > 1]
    mask = torch.ones(n, len(sides), dtype=torch.bool, device=DEV)
    cols = torch.empty(n, len(sides), dtype=torch.int64, device=DEV)
    vals = torch.empty(n, len(sides), dtype=F64, device=DEV)
    for q, (d, s) in enumerate(sides):
        if d is not None:
            mask[:, q] = at[d] > 0 if s < 0 else at[d] < top[d] - 1
        cols[:, q] = i if d is None else i + s * stride[d]
        vals[:, q] = coef(d, s)
    return _from_slots(mask, cols, vals)


def _laplace(dims):
    side = sum(2.0 for t in dims if t > 1)
    return _grid(dims, lambda d, s: side if d is None else -1.0)


def _faces(kappa, dims):
    """Harmonic means of the cells' coefficients at each face, the cell's own at the boundary."""
    k = kappa.reshape(dims[2], dims[1], dims[0])
    out = {}
    for d in range(3):
        if dims[d] == 1:
            continue
        axis = 2 - d
        for s in (-1, 1):
            nb = torch.roll(k, -s, axis)
            edge = [slice(None)] * 3
            edge[axis] = slice(-1, None) if s == 1 else slice(0, 1)
            nb[tuple(edge)] = k[tuple(edge)]
            out[d, s] = (2.0 * k * nb / (k + nb)).reshape(-1)
    return out


def _poisson(dims, g):
    """-div(kappa grad u), kappa lognormal(0, 1) cell by cell."""
    n = dims[0] * dims[1] * dims[2]
    f = _faces(torch.exp(torch.randn(n, dtype=F64, device=DEV, generator=g)), dims)
    total = sum(f.values())
    return _grid(dims, lambda d, s: total if d is None else -f[d, s])


def _convdiff(dims, g):
    """First-order upwind convection-diffusion with mass term, wind rotating about the axis,
    lognormal cell Peclet numbers in [0.1, 10]."""
    nx, ny, nz = dims
    n = nx * ny * nz
    i = torch.arange(n, device=DEV)
    x, y = (i % nx + 0.5) / nx, (i // nx % ny + 0.5) / ny
    w = torch.stack([-(y - 0.5), x - 0.5, torch.full_like(x, 0.2)]).to(F64)
    w = w / w.norm(dim=0)
    pe = torch.exp(torch.randn(n, dtype=F64, device=DEV, generator=g) * (math.log(10.0) / 2))
    p = [2.0 * pe.clamp(0.1, 10.0) * w[d] for d in range(3)]
    diag = 1.0 + sum(2.0 + p[d].abs() for d in range(3) if dims[d] > 1)

    def coef(d, s):
        if d is None:
            return diag
        return -1.0 - torch.where(p[d] > 0 if s < 0 else p[d] < 0, p[d].abs(), 0.0)
    return _grid(dims, coef)


def _q1_stiffness(h, young=1.0, nu=0.3):
    """24 x 24 stiffness of a trilinear cube of side h, 2 x 2 x 2 Gauss points."""
    lam, mu = young * nu / ((1 + nu) * (1 - 2 * nu)), young / (2 * (1 + nu))
    D = np.zeros((6, 6))
    D[:3, :3] = lam
    D[range(3), range(3)] += 2 * mu
    D[range(3, 6), range(3, 6)] = mu
    s = np.array([[a & 1, a >> 1 & 1, a >> 2 & 1] for a in range(8)]) * 2.0 - 1.0
    K = np.zeros((24, 24))
    for q in range(8):
        f = 1.0 + s * (s[q] / math.sqrt(3.0))
        dn = np.stack([s[:, 0] * f[:, 1] * f[:, 2], f[:, 0] * s[:, 1] * f[:, 2],
                       f[:, 0] * f[:, 1] * s[:, 2]], 1) / 8.0 / (h / 2.0)
        B = np.zeros((6, 24))
        for c in range(3):
            B[c, c::3] = dn[:, c]
        for r, (c, d) in enumerate(((0, 1), (1, 2), (0, 2))):
            B[3 + r, c::3] = dn[:, d]
            B[3 + r, d::3] = dn[:, c]
        K += B.T @ D @ B * (h / 2.0) ** 3
    return K


def _elastic(nodes):
    """Q1 elasticity on nodes^3 nodes, three unknowns a node interleaved, the face x = 0 clamped
    (identity rows, its couplings removed)."""
    K = torch.from_numpy(_q1_stiffness(1.0 / (nodes - 1))).to(DEV).reshape(8, 3, 8, 3)
    n = nodes ** 3
    i = torch.arange(n, device=DEV)
    at = (i % nodes, i // nodes % nodes, i // (nodes * nodes))
    corner = [(a & 1, a >> 1 & 1, a >> 2 & 1) for a in range(8)]
    block = torch.zeros(n, 27, 3, 3, dtype=F64, device=DEV)
    for a in range(8):  # node i is corner a of the element whose first node is at - corner[a]
        inside = torch.ones(n, dtype=torch.bool, device=DEV)
        for d in range(3):
            first = at[d] - corner[a][d]
            inside &= (first >= 0) & (first < nodes - 1)
        for b in range(8):
            o = [corner[b][d] - corner[a][d] + 1 for d in range(3)]
            block[:, o[2] * 9 + o[1] * 3 + o[0]] += torch.where(inside[:, None, None],
                                                                K[a, :, b, :], 0.0)
    there = torch.empty(n, 27, dtype=torch.bool, device=DEV)
    cols = torch.empty(n, 27, dtype=torch.int64, device=DEV)
    free = at[0] > 0
    for q in range(27):
        o = (q % 3 - 1, q // 3 % 3 - 1, q // 9 - 1)
        there[:, q] = free & (at[0] + o[0] > 0)
        for d in range(3):
            there[:, q] &= (at[d] + o[d] >= 0) & (at[d] + o[d] < nodes)
        cols[:, q] = i + o[0] + o[1] * nodes + o[2] * nodes * nodes
    there[~free, 13] = True
    block[~free, 13] = torch.eye(3, dtype=F64, device=DEV)
    mask = there[:, None, :, None].expand(n, 3, 27, 3).clone()
    eye = torch.eye(3, dtype=torch.bool, device=DEV)
    mask[~free, :, 13, :] = eye
    cols = (3 * cols[:, None, :, None] + torch.arange(3, device=DEV)).expand(n, 3, 27, 3)
    vals = block.permute(0, 2, 1, 3)
    return _from_slots(mask.reshape(3 * n, 81), cols.reshape(3 * n, 81), vals.reshape(3 * n, 81))


def _ragged(n, g):
    """An unstructured nonsymmetric matrix: lognormal row lengths (1 to 64 entries, about 11 on
    average), neighbours scattered near the diagonal with wrap-around, unsorted, diagonally
    dominant."""
    length = torch.exp(2.0 + 0.8 * torch.randn(n, dtype=F64, device=DEV, generator=g))
    length = length.clamp(0, 63).to(torch.int64)
    gap = torch.randint(1, 9, (n, 63), device=DEV, generator=g)
    off = torch.cumsum(gap, 1)
    off = off - torch.gather(off, 1, (length // 2).clamp(max=62)[:, None])
    off = off + (off >= 0).to(torch.int64)  # never the diagonal
    i = torch.arange(n, device=DEV)[:, None]
    cols = torch.cat([(i + off) % n, i], 1)
    vals = 2.0 * torch.rand(n, 64, dtype=F64, device=DEV, generator=g) - 1.0
    mask = torch.cat([torch.arange(63, device=DEV)[None, :] < length[:, None],
                      torch.ones(n, 1, dtype=torch.bool, device=DEV)], 1)
    vals[:, 63] = 0.5 + 1.1 * torch.where(mask[:, :63], vals[:, :63].abs(), 0.0).sum(1)
    return _from_slots(mask, cols, vals)


def _matrix(kind, size, seed):
    g = _gen(seed + 7919)
    if kind == "laplace2d":
        return _laplace((size, size, 1))
    if kind == "laplace3d":
        return _laplace((size, size, size))
    if kind == "poisson3d":
        return _poisson((size, size, size), g)
    if kind == "convdiff3d":
        return _convdiff((size, size, size), g)
    if kind == "elastic":
        return _elastic(size)
    return _ragged(size, g)


def _pack_systems(case, seed):
    """(matrix, b) of each system of a pack, on the GPU: sizes log-uniform (the same for every
    seed), kinds mixed."""
    r = np.random.RandomState(case["count"] * 100003 + case["high"])
    out = []
    for s in range(case["count"]):
        n = math.exp(r.uniform(math.log(case["low"]), math.log(case["high"])))
        g = _gen(seed * 1000 + s)
        c = max(2, round(n ** (1 / 3)))
        kind = r.randint(3)
        if kind == 0:
            A = _poisson((max(2, round(math.sqrt(n))),) * 2 + (1,), g)
        else:
            A = (_poisson if kind == 1 else _convdiff)((c, c, c), g)
        out.append((A, _times(A, _uniform(A[0].shape[0] - 1, g))))
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    if op == "pack":
        systems = _pack_systems(case, seed)
        h = gs2.pack_setup([tuple(t.cpu().numpy() for t in A) for A, _ in systems])
        b = torch.cat([b for _, b in systems])
        return dict(case=case, h=h, b=b, x=torch.zeros_like(b), p=_params(case))
    A = _matrix(case["matrix"], case["size"], seed)
    precision = case.get("precision", "fp64")
    h = gs2.gs2_setup(A, precisions=() if precision == "fp64" else (precision,))
    b, x = _vectors(case, A, seed)
    if op == "amg":
        h.amg_setup()
    return dict(case=case, h=h, b=b, x=x, p=_params(case))


def _vectors(case, A, seed):
    """b = A x_true, and the x that the call starts from: zero for a solve, some iterate for a
    smoother."""
    g = _gen(seed)
    n = A[0].shape[0] - 1
    b = _times(A, _uniform(n, g))
    zero = case["op"] in ("gmres", "cg", "pack", "amg")
    return b, torch.zeros_like(b) if zero else 0.1 * _uniform(n, g)


def _params(case):
    op = case["op"]
    if op == "apply":
        return gs2.params("gs2", inner=case["inner"], omega=case["omega"],
                          direction=case["direction"], precision=case["precision"])
    if op == "amg":
        return gs2.params("amg", direction=case["direction"])
    return gs2.params("gs2", direction=case.get("direction", "symmetric"))


def run(s):
    case, h, b, x = s["case"], s["h"], s["b"], s["x"]
    op = case["op"]
    if op == "apply":  # smooths x in place
        return gs2.gs2_apply_ex(h, b, x, s["p"])
    if op == "gs":
        return gs2.gs_apply(h, b, x, 1, case["omega"], case["direction"])
    if op == "mtgs":
        return gs2.mtgs_apply(h, b, x, 1, case["omega"], case["direction"])
    if op == "amg":
        return gs2.amg_vcycle(h, b, x, s["p"])
    x.zero_()
    if op == "pack":
        infos = gs2.pack_gmres(h, b, x, 30, case["tol"], 5000, s["p"])
        return dict(x=x, iters=np.array([i.iters for i in infos]))
    if op == "cg":
        info = gs2.cg_solve(h, b, x, case["tol"], 5000, s["p"])
    else:
        info = gs2.gmres_solve(h, b, x, case["restart"], case["tol"], 5000, s["p"])
    return dict(x=x, iters=info.iters)


# ---------------------------------------------------------------------------
# work: every matrix entry (value and column), b, the starting x and the result once, and the
# operations of one pass over the matrix's entries per sweep; of a solve, whose number of
# iterations is not known beforehand, the operations of one iteration
# ---------------------------------------------------------------------------

def _sizes(case):
    """(rows, stored entries); of ragged matrices and packs the expected values."""
    if case["op"] == "pack":
        lo, hi = case["low"], case["high"]
        n = case["count"] * (hi - lo) / max(1e-9, math.log(hi / lo))
        return n, 6.1 * n
    s, kind = case["size"], case["matrix"]
    if kind == "ragged":
        return s, 10.5 * s
    if kind == "laplace2d":
        return s * s, 5 * s * s - 4 * s
    if kind == "elastic":
        return 3 * s ** 3, 9 * (3 * s - 2) ** 2 * (3 * (s - 1) - 2) + 3 * s * s
    return s ** 3, 7 * s ** 3 - 6 * s * s


def work(case):
    n, nnz = _sizes(case)
    sweeps = 2 if case.get("direction", "symmetric") == "symmetric" else 1
    inner = case.get("inner", 1)
    # a half sweep: the residual and `inner` passes over one triangle
    flops = sweeps * (2 * nnz + inner * nnz)
    if case["op"] in ("gs", "mtgs"):
        flops = sweeps * 2 * nnz
    return {"bytes": 12.0 * nnz + 8.0 * n * (2 if case["op"] == "amg" else 3),
            "flops": float(flops)}


# ---------------------------------------------------------------------------
# exact: the same in plain 64-bit torch
# ---------------------------------------------------------------------------

def _times(A, x):
    rp, ci, va = A
    M = torch.sparse_csr_tensor(rp, ci.to(torch.int64), va, size=(rp.shape[0] - 1,) * 2)
    return M @ x


class _Split:
    """A = L + D + U with products by each part."""

    def __init__(self, A):
        rp, ci, va = A
        self.n = n = rp.shape[0] - 1
        rows = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
        cols = ci.to(torch.int64)

        def part(mask):
            count = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
            count[1:] = torch.cumsum(torch.bincount(rows[mask], minlength=n), 0)
            return torch.sparse_csr_tensor(count, cols[mask], va[mask], size=(n, n))
        self.A = torch.sparse_csr_tensor(rp, cols, va, size=(n, n))
        self.L, self.U = part(cols < rows), part(cols > rows)
        self.d = torch.zeros(n, dtype=F64, device=DEV)
        self.d[rows[cols == rows]] = va[cols == rows]

    def gs2(self, b, x, direction, inner=1, omega=1.0):
        order = {"forward": (self.L,), "backward": (self.U,), "symmetric": (self.L, self.U)}
        for T in order[direction]:
            r = (b - self.A @ x) / self.d
            g = r
            for _ in range(inner):
                g = r - omega * (T @ g) / self.d
            x = x + omega * g
        return x

    def rows_in_turn(self, groups, b, x, omega):
        """Gauss-Seidel / SOR: group after group of mutually independent rows (the rows of a group
        as slots of a padded row list)."""
        x = x.clone()
        for rows, cols, vals in groups:
            s = (vals * x[cols]).sum(1)  # the diagonal included
            x[rows] += omega * (b[rows] - s) / self.d[rows]
        return x


def _groups(A, number):
    """Rows with equal `number`, ascending, each as (rows, columns, values) padded to 7 slots."""
    rp, ci, va = A
    length = rp[1:] - rp[:-1]
    order = torch.argsort(number, stable=True)
    slot = torch.arange(int(length.max()), device=DEV)
    out = []
    for rows in torch.split(order, torch.bincount(number).tolist()):
        at = rp[rows][:, None] + slot
        there = slot < length[rows][:, None]
        at = torch.where(there, at, 0)
        out.append((rows, ci[at].to(torch.int64), torch.where(there, va[at], 0.0)))
    return out


def _solve_gmres(S, b, precond, m, tol, most):
    x, norm, iters = torch.zeros_like(b), float(b.norm()), 0
    while True:
        r = b - S.A @ x
        beta = float(r.norm())
        if beta <= tol * norm or iters >= most:
            return x, iters
        V = torch.zeros(m + 1, S.n, dtype=F64, device=DEV)
        V[0] = r / beta
        H, cs, sn = np.zeros((m + 1, m)), np.zeros(m), np.zeros(m)
        g = np.zeros(m + 1)
        g[0], k = beta, 0
        while k < m and iters < most:
            w = S.A @ precond(V[k])
            h = V[:k + 1] @ w
            w = w - h @ V[:k + 1]
            again = V[:k + 1] @ w
            w = w - again @ V[:k + 1]
            hn = w.norm()
            V[k + 1] = w / hn
            col = torch.cat([h + again, hn[None]]).cpu().numpy()
            for q in range(k):
                col[q], col[q + 1] = (cs[q] * col[q] + sn[q] * col[q + 1],
                                      -sn[q] * col[q] + cs[q] * col[q + 1])
            d = math.hypot(col[k], col[k + 1])
            cs[k], sn[k] = col[k] / d, col[k + 1] / d
            col[k], col[k + 1] = d, 0.0
            H[:k + 2, k] = col
            g[k + 1], g[k] = -sn[k] * g[k], cs[k] * g[k]
            k, iters = k + 1, iters + 1
            if abs(g[k]) <= tol * norm:
                break
        y = np.linalg.solve(H[:k, :k], g[:k])
        x = x + precond(torch.from_numpy(y).to(DEV) @ V[:k])


def _solve_cg(S, b, precond, tol, most):
    x, r, norm = torch.zeros_like(b), b.clone(), float(b.norm())
    z = precond(r)
    p, rz = z, r @ z
    for it in range(1, most + 1):
        q = S.A @ p
        alpha = rz / (p @ q)
        x, r = x + alpha * p, r - alpha * q
        if float(r.norm()) <= tol * norm:
            return x, it
        z = precond(r)
        new = r @ z
        p, rz = z + (new / rz) * p, new
    return x, most


def exact(case, seed):
    op = case["op"]
    if op == "amg":  # (would need a second implementation of the hierarchy)
        return None
    if op == "pack":
        xs, its = [], []
        for A, b in _pack_systems(case, seed):
            S = _Split(A)
            x, it = _solve_gmres(S, b, lambda v: S.gs2(v, torch.zeros_like(v), "symmetric"), 30,
                                 case["tol"], 5000)
            xs.append(x)
            its.append(it)
        return dict(x=torch.cat(xs), iters=np.array(its))
    A = _matrix(case["matrix"], case["size"], seed)
    b, x = _vectors(case, A, seed)
    S = _Split(A)
    if op == "apply":
        return S.gs2(b, x, case["direction"], case["inner"], case["omega"])
    if op in ("gs", "mtgs"):
        # a row's place in the sweep: the wavefront of the triangular solve (all neighbours behind
        # it come earlier), or its colour (these grids' first-fit colouring is red-black)
        i, s = torch.arange(S.n, device=DEV), case["size"]
        front = i % s + i // s % s + (i // (s * s) if case["matrix"] != "laplace2d" else 0)
        groups = _groups(A, front if op == "gs" else front % 2)
        if case["direction"] in ("forward", "symmetric"):
            x = S.rows_in_turn(groups, b, x, case["omega"])
        if case["direction"] in ("backward", "symmetric"):
            x = S.rows_in_turn(groups[::-1], b, x, case["omega"])
        return x
    d = case.get("direction", "symmetric")
    precond = lambda v: S.gs2(v, torch.zeros_like(v), d)  # noqa: E731
    if op == "cg":
        x, it = _solve_cg(S, b, precond, case["tol"], 5000)
    else:
        x, it = _solve_gmres(S, b, precond, case["restart"], case["tol"], 5000)
    return dict(x=x, iters=it)
