"""Which kernel the automatic engine takes, on both sides of every line, by the
block size it reports (512 and 1024: the persistent kernel's half and full
blocks, 0: the multi-kernel engine), and what the result then is against the
multi-kernel engine (engine=1)."""
import numpy as np
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu

SMS = 152  # of the GPU this library is written for; the sizes below follow from it


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    ensure_built()
    assert torch.cuda.get_device_properties(0).multi_processor_count == SMS


def _compare(m, dtype, threads, its=12, fmt=None, **kw):
    import torch
    A = gk.Matrix.from_csr(m, dtype)
    if fmt:
        B = A.convert(fmt)
        A.close()
        A = B
    b = torch.from_numpy(W.uniform_vector(m.n, 3)).to(
        torch_dev(), torch.float64 if dtype == "f64" else torch.float32)
    out = []
    for engine in (1, 0):
        x = torch.zeros_like(b)
        info = A.solve(b, x, precond="jacobi", tol=1e-30, max_iters=its, engine=engine, **kw)
        out.append((x.cpu().numpy().astype(np.float64), info))
    A.close()
    (x1, i1), (x0, i0) = out
    assert i1["block_threads"] == 0 and i0["block_threads"] == threads
    assert i0["return"] == i1["return"] and i0["iters"] == i1["iters"]
    # as in the fixed-iteration comparisons: sqrt(n) eps a dot, amplified by
    # at most 10^3 over the iterations
    eps = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    assert np.linalg.norm(x0 - x1) <= 1e3 * np.sqrt(m.n) * eps * np.linalg.norm(x1)


# a half block holds four vectors of 3,456 rows in FP64 and 6,912 in FP32; a
# full one four of 6,976 or two of 13,952 in FP64
@pytest.mark.parametrize("dtype,rows,threads", [
    ("f64", 3456, 512), ("f64", 3457, 1024), ("f64", 6976, 1024), ("f64", 6977, 1024),
    ("f64", 13952, 1024), ("f64", 13953, 0), ("f32", 6912, 512), ("f32", 6913, 1024),
    ("f32", 13952, 1024), ("f32", 13953, 1024)])
def test_cg_blocks(dtype, rows, threads):
    _compare(W.laplacian_1d(SMS * (rows // 64 * 64) + rows % 64), dtype, threads, method="cg")


# half blocks to 4,096 rows and 131,072 entries a block, full ones while w fits
@pytest.mark.parametrize("rows,band,m,threads", [
    (4096, 1, 30, 512), (4097, 1, 30, 1024), (1024, 60, 12, 512), (1025, 60, 12, 1024),
    (27648, 1, 4, 1024), (27649, 1, 4, 0)])
def test_gmres_blocks(rows, band, m, threads):
    n = SMS * (rows // 64 * 64) + rows % 64
    mat = W.laplacian_1d(n) if band == 1 else W.banded_spd(n, band, 3)
    _compare(mat, "f64", threads, method="gmres", krylov_dim=m)


@pytest.mark.parametrize("n,threads", [(1023, 0), (1024, 512), (2001, 512)])
def test_gmres_smallest(n, threads):
    _compare(W.laplacian_1d(n), "f64", threads, method="gmres")


@pytest.mark.parametrize("n,its", [(1, 1), (31, 4), (513, 12), (16385, 12)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_cg_smallest(n, its, dtype):
    """An ELL handle takes the persistent kernel at every size (a CSR one runs
    on a cluster up to 16,384 rows)."""
    _compare(W.laplacian_1d(n), dtype, 512, its=its, fmt="ell", method="cg")


@pytest.mark.parametrize("method", ["cg", "gmres"])
@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("name,threads", [("staged", 512), ("from_l2", 512), ("full", 1024)])
def test_16_bit_values(name, threads, dtype, method):
    """16-bit values solved directly: rows in shared memory, rows read from
    L2 with half and with full blocks."""
    m = {"staged": lambda: W.laplacian_2d(130, 133),
         "from_l2": lambda: W.banded_spd(40001, 60, 3),
         "full": lambda: W.laplacian_3d(131, 130, 129)}[name]()
    _compare(m, dtype, threads, method=method)


@pytest.mark.parametrize("mixed", [1, 2, 3])
@pytest.mark.parametrize("method", ["cg", "gmres"])
def test_refinement_reports_its_inner_solves(mixed, method):
    import torch
    m = W.laplacian_2d(130, 133)
    A = gk.Matrix.from_csr(m)
    b = torch.from_numpy(W.uniform_vector(m.n, 3)).to(torch_dev())
    for engine, threads in ((0, 512), (1, 0)):
        x = torch.zeros_like(b)
        info = A.solve(b, x, method=method, precond="jacobi", tol=1e-9, max_iters=20000,
                       mixed=mixed, engine=engine)
        assert info["return"] == gk.GK_OK and info["block_threads"] == threads
    A.close()
