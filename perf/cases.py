"""Workloads of the sparse operator library, as a user's program runs them:
SpMV applies, COO assembly, Krylov solves, batched solves and the ILU(0)
operator, through the Python binding of the C ABI.

``listed()`` names the workloads, ``draw(rng)`` gives more of the same
ranges, ``prepare`` builds inputs and handles on the GPU from a seed,
``run`` is one pass, ``work`` its least bytes and flops, and ``exact`` the
result in 64 bits by plain torch.
"""
import math

import numpy as np
import torch

import paper_2510_08230_gb300 as gk

DEV = "cuda"
L2_BYTES = 126e6  # a solve whose matrix fits on the chip need not read it again
VALUE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
VECTOR = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}


# ------------------------------------------------------------------ cases

def listed():
    return [
        # One product with the 64 x 64 Laplacian, the smallest system of the
        # benchmark: the cost of a call.
        dict(name="apply_csr_f64_lap2d_64", op="apply", matrix="lap2d", nx=64, ny=64, nz=1,
             fmt="csr", dtype="f64"),
        # The SpMV sweep's stencil in the library's default format.
        dict(name="apply_csr_f64_lap3d_256", op="apply", matrix="lap3d", nx=256, ny=256, nz=256,
             fmt="csr", dtype="f64"),
        # A stencil on a ragged box in the padded format, single precision
        # (the matrix of a refinement's inner solve).
        dict(name="apply_sellp_f32_lap3d_ragged", op="apply", matrix="lap3d", nx=201, ny=255,
             nz=190, fmt="sellp", dtype="f32"),
        # Residual r = b - A x on the sweep's skewed matrix (graphs, networks).
        dict(name="residual_csr_f64_powerlaw_4m", op="residual", matrix="powerlaw", n=1 << 22,
             mean=16, fmt="csr", dtype="f64"),
        # Assembly of a matrix from unordered triplets with duplicates, then
        # its first product.
        dict(name="assemble_coo_f64_powerlaw", op="assemble", matrix="powerlaw", n=500_009,
             mean=16, fmt="csr", dtype="f64"),
        # One small CG solve (the configuration quoted in solves per second).
        dict(name="cg_f64_lap2d_64", op="solve", matrix="lap2d", nx=64, ny=64, nz=1, fmt="csr",
             dtype="f64", method="cg", precond="none", mixed=0, tol=1e-10),
        # A request of the serving mix: ten to the fifth rows, in cache.
        dict(name="cg_f64_lap3d_serving", op="solve", matrix="lap3d", nx=49, ny=51, nz=47,
             fmt="csr", dtype="f64", method="cg", precond="jacobi", mixed=0, tol=1e-10),
        # Variable-coefficient diffusion on 128^3: Jacobi-CG in double
        # precision, and refined from single precision.
        dict(name="cg_f64_diffusion_128", op="solve", matrix="diffusion", nx=128, ny=128, nz=128,
             fmt="csr", dtype="f64", method="cg", precond="jacobi", mixed=0, tol=1e-10),
        dict(name="cg_mixed_diffusion_128", op="solve", matrix="diffusion", nx=128, ny=128,
             nz=128, fmt="csr", dtype="f64", method="cg", precond="jacobi", mixed=1, tol=1e-10),
        # GMRES(30) on the same operator.
        dict(name="gmres_f64_diffusion_128", op="solve", matrix="diffusion", nx=128, ny=128,
             nz=128, fmt="csr", dtype="f64", method="gmres", precond="jacobi", mixed=0,
             tol=1e-10),
        # Many independent small systems of uneven size in one call.
        dict(name="batched_cg_f64_2048", op="batched", count=2048, n_hi=4096, dtype="f64",
             tol=1e-10),
        # ILU(0) as an operator: both substitutions on the 128^3 stencil.
        dict(name="ilu_apply_f64_diffusion_128", op="ilu", matrix="diffusion", nx=128, ny=128,
             nz=128, fmt="csr", dtype="f64"),
    ]


def _log_int(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """A box of about n points, n log-uniform in [lo, hi], its sides uneven."""
    side = _log_int(rng, lo, hi) ** (1.0 / 3.0)
    return {k: max(3, int(round(side * rng.uniform(0.85, 1.15)))) for k in ("nx", "ny", "nz")}


def draw(rng):
    kind = rng.choice(["apply", "apply", "skewed", "assemble", "solve", "solve", "batched",
                       "ilu"])
    if kind == "apply":
        c = dict(op=rng.choice(["apply", "residual"]), fmt=rng.choice(["csr", "ell", "sellp", "coo"]),
                 dtype=rng.choice(["f64", "f32", "bf16"]))
        if rng.random() < 0.25:
            return dict(c, matrix="lap2d", nx=_log_int(rng, 20, 2500), ny=_log_int(rng, 20, 2500),
                        nz=1)
        return dict(c, matrix="lap3d", **_box(rng, 2_000, 10_000_000))
    if kind == "skewed":
        return dict(op=rng.choice(["apply", "residual"]), matrix="powerlaw",
                    n=_log_int(rng, 20_000, 3_000_000), mean=rng.choice([8, 16, 24]),
                    fmt=rng.choice(["csr", "coo"]), dtype=rng.choice(["f64", "f32"]))
    if kind == "assemble":
        return dict(op="assemble", matrix="powerlaw", n=_log_int(rng, 5_000, 400_000),
                    mean=rng.choice([8, 16]), fmt="csr", dtype=rng.choice(["f64", "f32"]))
    if kind == "solve":
        method = rng.choice(["cg", "cg", "gmres", "bicgstab"])
        c = dict(op="solve", fmt="csr", dtype="f64", method=method, precond="jacobi",
                 mixed=rng.choice([0, 1]) if method != "bicgstab" else 0, tol=1e-10)
        hi = 300_000 if method == "gmres" else 1_200_000
        if rng.random() < 0.25:
            return dict(c, matrix="banded", n=_log_int(rng, 2_000, 200_000),
                        half=rng.randint(5, 64))
        return dict(c, matrix=rng.choice(["lap3d", "diffusion"]), **_box(rng, 3_000, hi))
    if kind == "batched":
        dtype = rng.choice(["f64", "f32"])
        return dict(op="batched", count=_log_int(rng, 8, 1500), n_hi=rng.choice([1024, 2500, 4096]),
                    dtype=dtype, tol=1e-10 if dtype == "f64" else 1e-5)
    return dict(op="ilu", matrix="diffusion", fmt="csr", dtype=rng.choice(["f64", "f32"]),
                **_box(rng, 5_000, 1_500_000))


# ------------------------------------------------------------------ matrices

class Csr:
    """CSR arrays on the GPU: int32 indices, float64 values."""

    def __init__(self, n, row_ptr, col, val):
        self.n, self.row_ptr, self.col, self.val = n, row_ptr, col, val

    def rows(self):
        return torch.repeat_interleave(torch.arange(self.n, device=DEV),
                                       torch.diff(self.row_ptr.long()))


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _pack(n, table):
    """CSR of per-row candidate entries [(column offset, present, value)], in
    ascending column order."""
    idx = torch.arange(n, device=DEV, dtype=torch.int32)
    present = torch.stack([p for _, p, _ in table], 1)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(present.sum(1), 0, out=row_ptr[1:])
    col = torch.stack([idx + off for off, _, _ in table], 1)[present]
    val = torch.stack([v for _, _, v in table], 1)[present]
    return Csr(n, row_ptr.int(), col, val)


def _neighbours(nx, ny, nz):
    """(offset, axis, side, inside) of the stencil's neighbours, x fastest,
    offsets ascending; `inside` is a flat mask."""
    at = {2: torch.arange(nx, device=DEV).view(1, 1, -1).expand(nz, ny, nx),
          1: torch.arange(ny, device=DEV).view(1, -1, 1).expand(nz, ny, nx),
          0: torch.arange(nz, device=DEV).view(-1, 1, 1).expand(nz, ny, nx)}
    size, step = {2: nx, 1: ny, 0: nz}, {2: 1, 1: nx, 0: nx * ny}
    axes = (0, 1, 2) if nz > 1 else (1, 2)
    out = [(-step[a], a, -1, (at[a] > 0).reshape(-1)) for a in axes]
    return out + [(step[a], a, 1, (at[a] < size[a] - 1).reshape(-1)) for a in reversed(axes)]


def _laplacian(nx, ny, nz):
    """5- or 7-point Dirichlet Laplacian (nz = 1: two-dimensional)."""
    n = nx * ny * nz
    near = _neighbours(nx, ny, nz)
    minus, all_ = torch.full((n,), -1.0, dtype=torch.float64, device=DEV), torch.ones(
        n, dtype=torch.bool, device=DEV)
    table = [(off, inside, minus) for off, _, _, inside in near]
    table.insert(len(near) // 2, (0, all_, torch.full_like(minus, float(len(near)))))
    return _pack(n, table)


def _diffusion(nx, ny, nz, g):
    """7-point diffusion: log-normal cell coefficients (sigma 1), harmonic
    face coefficients, Dirichlet boundary."""
    n = nx * ny * nz
    k = torch.exp(torch.randn((nz, ny, nx), generator=g, dtype=torch.float64, device=DEV))
    diag = torch.zeros(n, dtype=torch.float64, device=DEV)
    table = []
    for off, axis, side, inside in _neighbours(nx, ny, nz):
        other = torch.roll(k, -side, axis)
        face = (2.0 * k * other / (k + other)).reshape(-1)
        diag += torch.where(inside, face, k.reshape(-1))
        table.append((off, inside, -face))
    table.insert(3, (0, torch.ones_like(table[0][1]), diag))
    return _pack(n, table)


def _powerlaw(n, mean, g):
    """Zipf(1.8) row lengths of the given mean, the longest 4096 (less on
    small matrices), uniformly random distinct columns, N(0,1) values."""
    top = min(4096, n // 4)
    p = torch.arange(1, top + 1, dtype=torch.float64, device=DEV) ** -1.8
    u = torch.rand(n, generator=g, dtype=torch.float64, device=DEV)
    z = (torch.searchsorted(torch.cumsum(p / p.sum(), 0), u) + 1).clamp_(1, top).double()
    lo, hi = 0.01, 1000.0
    for _ in range(60):
        c = 0.5 * (lo + hi)
        length = (c * z).round().clamp(1, top)
        m = float(length.mean())
        if abs(m - mean) <= 0.001 * mean:
            break
        lo, hi = (c, hi) if m < mean else (lo, c)
    length = length.long()
    length[int(torch.randint(0, n, (1,), generator=g, device=DEV))] = top
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length, 0, out=row_ptr[1:])
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), length)
    span = n - length + 1
    key = (torch.rand(rows.numel(), generator=g, dtype=torch.float64, device=DEV)
           * span[rows]).long()
    key = torch.sort(rows * n + torch.minimum(key, span[rows] - 1)).values - rows * n
    col = (key + torch.arange(rows.numel(), device=DEV) - row_ptr[rows]).int()
    val = torch.randn(rows.numel(), generator=g, dtype=torch.float64, device=DEV)
    return Csr(n, row_ptr.int(), col, val)


def _banded(n, half, g):
    """Symmetric band, off-diagonals U[-1,0], diagonal 1.1 x the absolute row
    sum."""
    off = -torch.rand((n, half), generator=g, dtype=torch.float64, device=DEV)
    idx = torch.arange(n, device=DEV)
    total = torch.zeros(n, dtype=torch.float64, device=DEV)
    upper, lower = [], []
    for d in range(1, half + 1):
        right = off[:, d - 1]
        left = torch.roll(right, d)
        upper.append((d, idx + d < n, right))
        lower.append((-d, idx >= d, left))
        total -= torch.where(idx + d < n, right, 0.0) + torch.where(idx >= d, left, 0.0)
    return _pack(n, lower[::-1] + [(0, idx >= 0, 1.1 * total)] + upper)


def _matrix(case, g):
    kind = case["matrix"]
    if kind in ("lap2d", "lap3d"):
        return _laplacian(case["nx"], case["ny"], case["nz"])
    if kind == "diffusion":
        return _diffusion(case["nx"], case["ny"], case["nz"], g)
    if kind == "banded":
        return _banded(case["n"], case["half"], g)
    return _powerlaw(case["n"], case["mean"], g)


def _uniform(n, g, dtype=torch.float64):
    return (2.0 * torch.rand(n, generator=g, dtype=torch.float64, device=DEV) - 1.0).to(dtype)


def _handle(m, fmt, dtype):
    val = m.val.to(VALUE[dtype])
    A = gk.Matrix(gk.gk_matrix_create_csr(m.n, m.n, m.col.numel(), m.row_ptr, m.col, val, dtype))
    if fmt == "csr":
        return A
    B = A.convert(fmt)
    A.close()
    return B


def _triplets(case, g):
    """The matrix's entries in random order, one in fifty of them split in
    two."""
    m = _matrix(case, g)
    rows = m.rows().int()
    twice = torch.rand(rows.numel(), generator=g, device=DEV) < 0.02
    val = torch.where(twice, 0.5 * m.val, m.val).to(VALUE[case["dtype"]])
    row, col, val = (torch.cat([a, a[twice]]) for a in (rows, m.col, val))
    order = torch.randperm(row.numel(), generator=g, device=DEV)
    return m.n, row[order].contiguous(), col[order].contiguous(), val[order].contiguous()


def _rectangles(case, seed):
    """Grid sides and diagonal shifts of a batch: n_target ~ U{64..n_hi},
    width U{8..64} (the case's own), shift U[0,1] (from the seed)."""
    size, rng = np.random.default_rng(case["n_hi"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        target, a = int(size.integers(64, case["n_hi"] + 1)), int(size.integers(8, 65))
        out.append((a, int(min(max(round(target / a), 1), case["n_hi"] // a)),
                    float(rng.uniform(0.0, 1.0))))
    return out


def _rectangle_csr(a, b, shift):
    """Host CSR arrays of the a x b 5-point Laplacian plus shift."""
    n = a * b
    i = np.arange(n, dtype=np.int32)
    x, y = i % a, i // a
    present = np.stack([y > 0, x > 0, i >= 0, x < a - 1, y < b - 1], 1)
    col = (i[:, None] + np.array([-a, -1, 0, 1, a], dtype=np.int32))[present]
    val = np.broadcast_to(np.array([-1.0, -1.0, 4.0 + shift, -1.0, -1.0]), (n, 5))[present]
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    np.cumsum(present.sum(1), out=row_ptr[1:])
    return row_ptr, col, val


# ------------------------------------------------------------------ passes

def prepare(case, seed):
    g = _generator(seed)
    op, dtype = case["op"], case["dtype"]
    vec = VECTOR[dtype]
    if op == "assemble":
        n, row, col, val = _triplets(case, g)
        return dict(case=case, n=n, row=row, col=col, val=val, b=_uniform(n, g, vec),
                    y=torch.empty(n, dtype=vec, device=DEV))
    if op == "batched":
        value = np.float64 if dtype == "f64" else np.float32
        handles, sizes = [], []
        for a, b, shift in _rectangles(case, seed):
            rp, col, val = _rectangle_csr(a, b, shift)
            handles.append(gk.Matrix(gk.gk_matrix_create_csr(a * b, a * b, col.size, rp, col,
                                                             val.astype(value), dtype)))
            sizes.append(a * b)
        rhs = _uniform(sum(sizes), g, vec)
        x = torch.zeros_like(rhs)
        return dict(case=case, matrices=handles, rhs=rhs, x=x, A=[h.handle for h in handles],
                    bs=list(rhs.split(sizes)), xs=list(x.split(sizes)))
    m = _matrix(case, g)
    A = _handle(m, case["fmt"], dtype)
    b = _uniform(m.n, g, vec)
    s = dict(case=case, A=A, b=b, y=torch.zeros(m.n, dtype=vec, device=DEV))
    if op == "residual":
        s["x"] = _uniform(m.n, g, vec)
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "apply":
        s["A"].apply(s["b"], s["y"])
    elif op == "residual":
        s["y"].copy_(s["b"])
        s["A"].apply_adv(-1.0, s["x"], 1.0, s["y"])
    elif op == "assemble":
        A = gk.Matrix(gk.gk_matrix_create_coo(s["n"], s["n"], s["row"].numel(), s["row"],
                                              s["col"], s["val"], c["dtype"]))
        A.apply(s["b"], s["y"])
        nnz = A.nnz
        A.close()
        return s["y"], nnz
    elif op == "solve":
        s["y"].zero_()
        s["A"].solve(s["b"], s["y"], method=c["method"], precond=c["precond"], tol=c["tol"],
                     max_iters=20000, krylov_dim=30, mixed=c["mixed"])
    elif op == "batched":
        s["x"].zero_()
        gk.gk_solve_batched(s["A"], s["bs"], s["xs"],
                            gk.make_opts(method="cg", precond="jacobi", tol=c["tol"],
                                         max_iters=5000))
        return s["x"]
    else:
        s["A"].precond_apply(s["b"], s["y"], kind="ilu")
    return s["y"]


# ------------------------------------------------------------------ least work

def _counts(case):
    """Rows and entries of the case's matrix."""
    kind = case["matrix"]
    if kind == "powerlaw":
        return case["n"], case["n"] * case["mean"]
    if kind == "banded":
        h = case["half"]
        return case["n"], case["n"] * (2 * h + 1) - h * (h + 1)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    faces = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
    return nx * ny * nz, nx * ny * nz + 2 * faces


def _iterations(case):
    """About how many iterations a solve takes (measured on each family)."""
    if case["matrix"] == "banded":
        return 130
    side = max(case["nx"], case["ny"], case["nz"])
    per_side = {"lap2d": 3.5, "lap3d": 2.4, "diffusion": 4.7}[case["matrix"]]
    if case["method"] == "gmres":
        return per_side * side * (1.0 + side / 64.0)
    return per_side * side * (0.65 if case["method"] == "bicgstab" else 1.0)


def work(case):
    """Bytes and flops of one pass: inputs read once and outputs written
    once.  A solve reads its matrix once, or once per iteration where it does
    not fit on the chip."""
    size = SIZE[case["dtype"]]
    vec = 8 if case["dtype"] == "f64" else 4
    if case["op"] == "batched":
        n = case["count"] * (64 + case["n_hi"]) / 2
        its = 75 if case["dtype"] == "f64" else 35
        return {"bytes": n * (5 * (size + 4) + 4 + 2 * vec), "flops": n * its * 2 * (5 + 6)}
    n, nnz = _counts(case)
    matrix = nnz * (size + 4) + 4 * (n + 1)
    if case["op"] == "assemble":
        return {"bytes": 1.02 * nnz * (size + 8) + matrix + 2 * n * vec, "flops": 2 * nnz}
    if case["op"] == "solve":
        its = _iterations(case)
        low = 0.5 if case["mixed"] else 1.0
        per = (0.67 if case["mixed"] else 1.0) * matrix
        extra = 15 * 2 * 2 * n if case["method"] == "gmres" else 6 * 2 * n
        products = 2 if case["method"] == "bicgstab" else 1
        once = matrix + 2 * n * vec
        again = 0 if matrix < L2_BYTES else its * products * (per + 6 * low * n * vec)
        return {"bytes": once + again, "flops": its * (products * 2 * nnz + extra)}
    if case["op"] == "ilu":
        return {"bytes": matrix + 3 * n * vec, "flops": 2 * nnz}
    vectors = 3 if case["op"] == "residual" else 2
    return {"bytes": matrix + vectors * n * vec, "flops": 2 * nnz}


# ------------------------------------------------------------------ 64 bits

def _product(rows, col, val, x, n):
    y = torch.zeros(n, dtype=torch.float64, device=DEV)
    return y.index_add_(0, rows, val.double() * x.double()[col.long()])


def _solution(m, b):
    """A x = b by Jacobi-CG in 64 bits, restarted from its residual until
    that stands still."""
    A = torch.sparse_csr_tensor(m.row_ptr.long(), m.col.long(), m.val, size=(m.n, m.n))
    rows = m.rows()
    dinv = 1.0 / m.val[rows == m.col]
    x = torch.zeros_like(b)
    for goal in (1e-10, 1e-6, 1e-4):
        r = b - A @ x
        stop = float(r.norm()) * goal
        z = dinv * r
        p, rz, d = z.clone(), r @ z, torch.zeros_like(x)
        for k in range(20000):
            q = A @ p
            alpha = rz / (p @ q)
            d += alpha * p
            r -= alpha * q
            if k % 20 == 19 and not float(r.norm()) > stop:
                break
            z = dinv * r
            rz, old = r @ z, rz
            p = z + (rz / old) * p
        x += d
    return x


def _separable(case, seed, rhs):
    """The batch's solutions in the Laplacian's eigenbasis."""
    basis = {}

    def modes(k):
        if k not in basis:
            j = torch.arange(1, k + 1, dtype=torch.float64, device=DEV)
            basis[k] = (math.sqrt(2.0 / (k + 1)) * torch.sin(math.pi * j[:, None] * j / (k + 1)),
                        2.0 - 2.0 * torch.cos(math.pi * j / (k + 1)))
        return basis[k]

    out, at = [], 0
    for a, b, shift in _rectangles(case, seed):
        if case["dtype"] == "f32":
            shift = float(np.float32(4.0 + shift)) - 4.0
        (sa, la), (sb, lb) = modes(a), modes(b)
        f = rhs[at:at + a * b].double().view(b, a)
        at += a * b
        out.append((sb @ ((sb @ f @ sa) / (lb[:, None] + la + shift)) @ sa).reshape(-1))
    return torch.cat(out)


def _ilu(case, m, r):
    """z = U^-1 L^-1 r of the 7-point matrix's ILU(0), one diagonal plane of
    the grid after the other.  No fill lies on the pattern, so only the
    pivots change: u_ii = a_ii - sum of a_ik a_ki / u_kk."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n, rows, col = m.n, m.rows(), m.col.long()
    offs = [nx * ny, nx, 1]
    low = [torch.zeros(n, dtype=torch.float64, device=DEV) for _ in offs]
    up = [torch.zeros(n, dtype=torch.float64, device=DEV) for _ in offs]
    for d, lo, hi in zip(offs, low, up):
        at = col == rows - d
        lo[rows[at]] = m.val[at]
        at = col == rows + d
        hi[rows[at]] = m.val[at]
    u = m.val[col == rows].clone()
    idx = torch.arange(n, device=DEV)
    level = idx % nx + (idx // nx) % ny + idx // (nx * ny)
    planes = list(torch.split(torch.argsort(level, stable=True),
                              torch.bincount(level).tolist()))
    y = torch.zeros(n, dtype=torch.float64, device=DEV)
    z = torch.zeros_like(y)
    for i in planes:
        t = r.double()[i]
        for d, lo, hi in zip(offs, low, up):
            k = (i - d).clamp(min=0)
            f = lo[i] / u[k]
            u[i] -= f * hi[k]
            t = t - f * y[k]
        y[i] = t
    for i in reversed(planes):
        t = y[i]
        for d, hi in zip(offs, up):
            t = t - hi[i] * z[(i + d).clamp(max=n - 1)]
        z[i] = t / u[i]
    return z


def exact(case, seed):
    s = prepare(case, seed)
    op, dtype = case["op"], case["dtype"]
    if op == "assemble":
        return _product(s["row"].long(), s["col"], s["val"], s["b"], s["n"]), None
    if op == "batched":
        return _separable(case, seed, s["rhs"])
    m = _matrix(case, _generator(seed))
    if op == "solve":
        return _solution(m, s["b"])
    m.val = m.val.to(VALUE[dtype]).double()
    if op == "ilu":
        return _ilu(case, m, s["b"])
    if op == "residual":
        return s["b"].double() - _product(m.rows(), m.col, m.val, s["x"], m.n)
    return _product(m.rows(), m.col, m.val, s["b"], m.n)
