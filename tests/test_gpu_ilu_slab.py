"""The slab mode of the ILU(0) substitutions (consecutive rows on one SM,
values across slab boundaries through L2): bit for bit the oracle's
substitution, the other modes' bits in FP32 and for signalling NaNs, and an
error status when a wait runs out."""
import numpy as np
import pytest

import oracle
import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu

# what each reaches: slabs of one row; slabs shorter and longer than the
# farthest dependency; slabs of whole planes; more slabs than SMs are left to
# one; rows a level up to the thread count and past it; dependencies two
# levels back; a remainder slab
CASES = {
    "one_row": lambda: W.laplacian_1d(1),
    "lap1d_33": lambda: W.laplacian_1d(33),
    "lap1d_7000": lambda: W.laplacian_1d(7000),
    "lap2d_37x29": lambda: W.laplacian_2d(37, 29),
    "lap2d_700x300": lambda: W.laplacian_2d(700, 300),
    "lap2d_3x5000": lambda: W.laplacian_2d(3, 5000),
    "convdiff_45": lambda: W.convection_diffusion_2d(45),
    "diff3d_12": lambda: W.diffusion_3d(12, seed=5),
    "lap3d_33x35x70": lambda: W.laplacian_3d(33, 35, 70),
    "lap3d_90x90x8": lambda: W.laplacian_3d(90, 90, 8),
    "banded_2": lambda: W.banded_spd(5001, 2, 7),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("case", list(CASES))
def test_apply_and_triangular_solves_bit_exact(monkeypatch, case):
    import torch
    monkeypatch.setenv("GK_ILU_CHUNK", "slab")
    dev = torch_dev()
    m = CASES[case]()
    A = gk.Matrix.from_csr(m, "f64")
    lu = oracle.ilu0(m)
    rng = np.random.default_rng(31)
    for rep in range(3):
        r = rng.uniform(-1, 1, m.n)
        rt = torch.from_numpy(r).to(dev)
        zt = torch.full_like(rt, float("nan"))
        A.precond_apply(rt, zt, "ilu")
        torch.cuda.synchronize()
        want = oracle.ilu0_apply(m, lu, r)
        assert np.array_equal(zt.cpu().numpy().view(np.uint64), want.view(np.uint64)), rep
    A.close()


@pytest.mark.parametrize("case", ["lap1d_33", "lap2d_37x29", "lap3d_33x35x70"])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_same_bits_as_chunks(monkeypatch, case, dtype):
    """FP32 and FP64, with signalling NaNs among the inputs; the triangular
    solves of A itself as well."""
    import torch
    dev = torch_dev()
    m = CASES[case]()
    vt = torch.float64 if dtype == "f64" else torch.float32
    ut = np.uint64 if dtype == "f64" else np.uint32
    r = W.uniform_vector(m.n, 17).astype(np.float64 if dtype == "f64" else np.float32)
    r.view(ut)[[m.n // 2, m.n - 1]] = ut(0x7FF0000000000005 if dtype == "f64" else 0x7F800005)
    outs = {}
    for mode in ("32", "slab"):
        monkeypatch.setenv("GK_ILU_CHUNK", mode)
        A = gk.Matrix.from_csr(m, dtype)
        rt = torch.from_numpy(r).to(dev)
        got = []
        zt = torch.zeros(m.n, dtype=vt, device=dev)
        A.precond_apply(rt, zt, "ilu")
        got.append(zt.cpu().numpy().view(ut))
        for upper in (0, 1):
            for unit in (0, 1):
                zt = torch.zeros(m.n, dtype=vt, device=dev)
                A.triangular_solve(rt, zt, upper=upper, unit_diagonal=unit)
                torch.cuda.synchronize()
                got.append(zt.cpu().numpy().view(ut))
        outs[mode] = got
        A.close()
    for a, b in zip(outs["32"], outs["slab"]):
        assert np.array_equal(a, b)


def test_times_out_then_recovers(monkeypatch):
    """A budget shorter than a copy of records runs out (waits on other slabs
    take the default at least); blocks leave after their copies have landed
    and the next apply is exact.  Solves in a captured graph likewise."""
    import torch
    monkeypatch.setenv("GK_ILU_CHUNK", "slab")
    m = W.laplacian_3d(24)
    A = gk.Matrix.from_csr(m, "f64")
    dev = torch_dev()
    r = W.uniform_vector(m.n, 8)
    rt = torch.from_numpy(r).to(dev)
    zt = torch.zeros_like(rt)
    want = oracle.ilu0_apply(m, oracle.ilu0(m), r)
    for _ in range(2):
        A.precond_apply(rt, zt, "ilu")
        torch.cuda.synchronize()
        assert np.array_equal(zt.cpu().numpy(), want)
        assert gk.gk_precond_apply(A.handle, "ilu", 0, rt, zt, 1) == gk.GK_ERR_TIMEOUT
    xt = torch.zeros_like(rt)
    info = A.solve(rt, xt, method="cg", precond="ilu", tol=1e-10, max_iters=500, wait_budget_ns=1)
    assert info["return"] == gk.GK_ERR_TIMEOUT, info
    for method in ("cg", "gmres", "bicgstab"):
        xt.zero_()
        info = A.solve(rt, xt, method=method, precond="ilu", tol=1e-10, max_iters=500)
        assert info["return"] == gk.GK_OK, info
        assert oracle.true_rel_residual(m, r, xt.cpu().numpy()) <= 1e-10
    A.close()


def test_at_once_equal_alone(monkeypatch):
    """Launches that share the SMs: 64 or more slabs each, from four threads."""
    import threading
    import torch
    monkeypatch.setenv("GK_ILU_CHUNK", "slab")
    dev = torch_dev()
    jobs = []
    for m in (W.laplacian_3d(40), W.laplacian_2d(300, 200), W.laplacian_3d(36), W.laplacian_2d(64)):
        A = gk.Matrix.from_csr(m, "f64")
        r = torch.from_numpy(W.uniform_vector(m.n, 3)).to(dev)
        z = torch.zeros_like(r)
        A.precond_apply(r, z, "ilu")
        jobs.append((A, r, z.clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    same = [True] * len(jobs)

    def run(i):
        A, r, want, s = jobs[i]
        with torch.cuda.stream(s):
            z = torch.zeros_like(r)
        for _ in range(10):
            A.precond_apply(r, z, "ilu", stream=s)
            s.synchronize()
            same[i] = same[i] and torch.equal(z, want)

    ts = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert all(same), same
    for A, *_ in jobs:
        A.close()
