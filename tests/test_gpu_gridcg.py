"""The persistent grid-wide kernels of CG and GMRES (the automatic engine on
matrices that solve on an ELL layout) against the multi-kernel engine
(engine=1) and the oracle: every shared-memory mode, odd sizes, both ends of
their range."""
import numpy as np
import pytest

import oracle
import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _solve(A, b, dtype, **kw):
    import torch
    bt = torch.from_numpy(b).to(torch_dev(), torch.float64 if dtype == "f64" else torch.float32)
    x = torch.zeros_like(bt)
    info = A.solve(bt, x, **dict(dict(method="cg"), **kw))
    return x.cpu().numpy().astype(np.float64), info


# name: matrix, what it reaches (152 blocks; rows a block keeps per mode)
FIXED = {
    "mode0_first": lambda: W.laplacian_2d(129, 128),      # 16,512 rows
    "mode0_odd": lambda: W.laplacian_3d(31, 29, 37),      # 33,263 rows, a virtual pair row
    "mode0_large": lambda: W.laplacian_2d(601, 599),
    "mode1_wide": lambda: W.banded_spd(40001, 60, 3),     # 121 entries a row
    "mode1": lambda: W.laplacian_1d(900001),
    "half_limit": lambda: W.laplacian_2d(608, 512),       # 2,048 rows a block
    "half_mode1": lambda: W.banded_spd(60001, 12, 4),     # 25 entries a row
    "half_last": lambda: W.laplacian_1d(152 * 3392),      # FP64: the last half grid of CG
    "full_first": lambda: W.laplacian_1d(152 * 3520 + 1),
    "mode2": lambda: W.laplacian_1d(1200001),             # FP64 only: 7,936 rows a block
}


@pytest.mark.parametrize("name", list(FIXED))
@pytest.mark.parametrize("dtype,precond", [("f64", "jacobi"), ("f64", None), ("f32", "jacobi")])
def test_fixed_iterations_equal_multi_kernel(name, dtype, precond):
    """30 iterations from the same start: the same recurrence and row sums,
    the dot products in another order.  A dot of n terms of either order is
    within n eps of the exact one relative to its absolute sum, in practice
    sqrt(n) eps; 30 iterations amplify that by at most ~10^3."""
    m = FIXED[name]()
    A = gk.Matrix.from_csr(m, dtype)
    b = W.uniform_vector(m.n, 3)
    kw = dict(precond=precond, tol=1e-30, max_iters=30)
    x1, i1 = _solve(A, b, dtype, engine=1, **kw)
    x0, i0 = _solve(A, b, dtype, **kw)
    assert i0["return"] == i1["return"] == gk.GK_NOT_CONVERGED
    assert i0["iters"] == i1["iters"] == 30 and i0["spmv_format"] == i1["spmv_format"] == gk.GK_ELL
    eps = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    tol = 1e3 * np.sqrt(m.n) * eps
    assert np.linalg.norm(x0 - x1) <= tol * np.linalg.norm(x1)
    assert abs(i0["rel_res_true"] - i1["rel_res_true"]) <= tol * (1 + i1["rel_res_true"])
    assert abs(i0["rel_res_recurrence"] - i1["rel_res_recurrence"]) <= tol * (
        1 + i1["rel_res_recurrence"])
    A.close()


@pytest.mark.parametrize("name,m", [("mode0_first", 30), ("mode0_odd", 7), ("mode1_wide", 64),
                                    ("mode1", 33), ("mode2", 9), ("half_limit", 31),
                                    ("half_mode1", 12)])
@pytest.mark.parametrize("dtype,precond", [("f64", "jacobi"), ("f64", None), ("f32", "jacobi")])
def test_gmres_fixed_steps_equal_multi_kernel(name, m, dtype, precond):
    """m + 5 Arnoldi steps (a restart among them; up to 64 columns, with and
    without the matrix in shared memory): orthogonalised twice, so the steps
    of either engine are within a few n eps of exact ones relative to the
    cycle's residual; a factor 10^3 as for CG."""
    mat = FIXED[name]()
    A = gk.Matrix.from_csr(mat, dtype)
    b = W.uniform_vector(mat.n, 3)
    kw = dict(method="gmres", precond=precond, tol=1e-30, max_iters=m + 5, krylov_dim=m)
    x1, i1 = _solve(A, b, dtype, engine=1, **kw)
    x0, i0 = _solve(A, b, dtype, **kw)
    assert i0["return"] == i1["return"] == gk.GK_NOT_CONVERGED
    assert (i0["iters"], i0["restarts"]) == (i1["iters"], i1["restarts"]) == (m + 5, 1)
    eps = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    tol = 1e3 * np.sqrt(mat.n) * eps
    assert np.linalg.norm(x0 - x1) <= tol * np.linalg.norm(x1)
    for key in ("rel_res_true", "rel_res_recurrence"):
        assert abs(i0[key] - i1[key]) <= tol * (1 + i1[key])
    A.close()


@pytest.mark.parametrize("method", ["cg", "gmres"])
@pytest.mark.parametrize("mixed", [0, 1, 2, 3])
@pytest.mark.parametrize("name", ["lap2d", "diff3d"])
def test_converges_like_multi_kernel(name, mixed, method):
    """To a true 1e-10, plain and refined (the inner solves run on the same
    kernel), from a nonzero start; twice, with the same bits."""
    import torch
    m = W.laplacian_2d(131) if name == "lap2d" else W.diffusion_3d(30)
    A = gk.Matrix.from_csr(m)
    b = W.uniform_vector(m.n, 5)
    bt = torch.from_numpy(b).to(torch_dev())
    out = []
    for engine in (1, 0, 0):
        x = torch.from_numpy(0.1 * W.uniform_vector(m.n, 6)).to(torch_dev())
        info = A.solve(bt, x, method=method, precond="jacobi", tol=1e-10, max_iters=40000,
                       mixed=mixed, engine=engine)
        assert info["return"] == gk.GK_OK, info
        assert oracle.true_rel_residual(m, b, x.cpu().numpy()) <= 1e-10
        out.append((x.cpu().numpy(), info))
    assert np.array_equal(out[1][0], out[2][0])
    if not mixed:
        assert abs(out[0][1]["iters"] - out[1][1]["iters"]) <= max(
            3 if method == "cg" else 30, 0.1 * out[0][1]["iters"])
    A.close()


@pytest.mark.parametrize("method", ["cg", "gmres"])
def test_edges(method):
    """b = 0, an exact initial guess, a negative definite matrix (a breakdown
    of CG), NaN, an iteration cap of one, and a zero diagonal: the
    multi-kernel engine's outcomes."""
    import torch
    dev = torch_dev()
    m = W.laplacian_2d(130)
    A = gk.Matrix.from_csr(m)
    neg = gk.Matrix.from_csr(W.CSR(m.n, m.n, m.row_ptr, m.col_idx, -m.values))
    ones = torch.ones(m.n, dtype=torch.float64, device=dev)
    exact = torch.empty_like(ones)
    A.apply(ones, exact)
    nan = ones.clone()
    nan[7] = float("nan")
    for M, b, x0, kw in ((A, torch.zeros_like(ones), ones, {}), (A, exact, ones, {}),
                         (neg, ones, 0 * ones, {}), (A, nan, 0 * ones, {}),
                         (A, ones, 0 * ones, dict(max_iters=1))):
        res = []
        for engine in (1, 0):
            x = x0.clone()
            info = M.solve(b, x, method=method, tol=1e-10, engine=engine,
                           **dict(dict(max_iters=99), **kw))
            res.append((info, x.cpu().numpy()))
        (i1, x1), (i0, x0_) = res
        assert (i0["return"], i0["status"], i0["iters"]) == (i1["return"], i1["status"], i1["iters"])
        assert np.allclose(x0_, x1, rtol=1e-9, atol=1e-12, equal_nan=True)
    v = m.values.copy()
    v[m.row_ptr[5]:m.row_ptr[6]] = 0.0
    Z = gk.Matrix.from_csr(W.CSR(m.n, m.n, m.row_ptr, m.col_idx, v))
    info = Z.solve(ones, 0 * ones, method=method, precond="jacobi", max_iters=9)
    assert info["return"] == gk.GK_ERR_ZERO_DIAG
    for M in (A, neg, Z):
        M.close()


def test_solves_at_once_equal_alone():
    """Grids that share the GPU (half blocks), that fill it (full blocks) and
    refinements, from six threads: bit-identical to the same solve alone."""
    import threading
    import torch
    work = [(W.laplacian_2d(131, 130), "cg", 0), (W.laplacian_3d(48, 50, 49), "cg", 0),
            (W.laplacian_2d(130, 133), "gmres", 0), (W.laplacian_2d(640, 639), "cg", 0),
            (W.laplacian_2d(51, 40), "gmres", 1), (W.laplacian_3d(40, 41, 39), "cg", 1)]
    dev = torch_dev()
    jobs = []
    for m, method, mixed in work:
        A = gk.Matrix.from_csr(m, "f64")
        b = torch.from_numpy(W.uniform_vector(m.n, 5)).to(dev)
        jobs.append((A, b, dict(method=method, precond="jacobi", tol=1e-30, max_iters=200,
                                mixed=mixed)))
    torch.cuda.synchronize()

    def run(i, out):
        A, b, kw = jobs[i]
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            x = torch.zeros_like(b)
        info = A.solve(b, x, s, **kw)
        s.synchronize()
        out[i] = (x.cpu(), info["iters"], info["return"])

    alone, at_once = {}, {}
    for i in range(len(jobs)):
        run(i, alone)
    for _ in range(3):
        ts = [threading.Thread(target=run, args=(i, at_once)) for i in range(len(jobs))]
        [t.start() for t in ts]
        [t.join() for t in ts]
        for i in range(len(jobs)):
            assert torch.equal(alone[i][0], at_once[i][0]) and alone[i][1:] == at_once[i][1:], i
    for A, _, _ in jobs:
        A.close()
