"""The persistent grid kernels under a wait budget that runs out: every block
leaves, and the solve is the multi-kernel engine's, from the caller's initial
guess and bit for bit, since that engine waits for nothing here.  A budget of
one nanosecond is shorter than any hand-off between blocks; no wait is on a
value that never comes."""
import time

import numpy as np
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu

# half blocks with the matrix in shared memory, full blocks, and (FP64 CG) full
# blocks that keep x in global memory
MATRICES = {
    "half": lambda: W.laplacian_2d(130, 133),
    "full": lambda: W.laplacian_1d(152 * 3520 + 1),
    "x_in_global": lambda: W.laplacian_1d(1200001),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("method", ["cg", "gmres"])
@pytest.mark.parametrize("dtype,mixed", [("f64", 0), ("f32", 0), ("f64", 1)])
@pytest.mark.parametrize("name", list(MATRICES))
def test_budget_runs_out_then_multi_kernel(name, dtype, mixed, method):
    import torch
    m = MATRICES[name]()
    A = gk.Matrix.from_csr(m, dtype)
    vt = torch.float64 if dtype == "f64" else torch.float32
    b = torch.from_numpy(W.uniform_vector(m.n, 3)).to(torch_dev(), vt)
    x0 = 0.1 * torch.from_numpy(W.uniform_vector(m.n, 4)).to(torch_dev(), vt)

    def solve(**kw):
        x = x0.clone()
        t = time.perf_counter()
        info = A.solve(b, x, method=method, precond="jacobi", tol=1e-30, max_iters=40, mixed=mixed,
                       **kw)
        torch.cuda.synchronize()
        keys = ("return", "iters", "restarts", "outer_iters", "rel_res_true", "rel_res_recurrence")
        return x.cpu().numpy(), tuple(info[k] for k in keys), time.perf_counter() - t

    grid = solve()
    multi = solve(engine=1)
    short = solve(wait_budget_ns=1)
    assert short[2] < 1.0, short[2]  # the waits gave up, far below the 2 s default
    assert short[1] == multi[1]
    assert np.array_equal(short[0], multi[0])
    again = solve()  # nothing is left behind
    generous = solve(wait_budget_ns=5_000_000_000)
    for other in (again, generous):
        assert other[1] == grid[1] and np.array_equal(other[0], grid[0])
    A.close()
