"""One handle that serves plain and refined solves in turn: the copies in
other value types and the solver's layout stay apart.  Refinement with
FP16-stored inner solves must run on the FP16 copy every time, as on a fresh
handle, and FP64 solves must stay on the FP64 values."""
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


def _arrow(n):
    """Symmetric, diagonally dominant, a full first row and column: no padded
    layout is admissible, so the solver stays on the CSR arrays."""
    rng = np.random.default_rng(11)
    off = rng.uniform(-1.0, 1.0, n - 1) / n
    rp = np.concatenate([[0], n + 2 * np.arange(n, dtype=np.int64)]).astype(np.int32)
    ci = np.empty(n + 2 * (n - 1), np.int32)
    v = np.empty(ci.size)
    ci[:n], v[0], v[1:n] = np.arange(n), 3.0, off
    ci[n::2], ci[n + 1::2] = 0, np.arange(1, n)
    v[n::2], v[n + 1::2] = off, rng.uniform(2.0, 3.0, n - 1)
    return W.CSR(n, n, rp, ci, v)


@pytest.mark.parametrize("name,layout", [("arrow", gk.GK_CSR), ("lap2d", gk.GK_ELL)])
@pytest.mark.parametrize("mixed", [1, 2, 3])
def test_refined_and_plain_solves_in_turn(name, layout, mixed):
    import torch
    m = _arrow(20000) if name == "arrow" else W.laplacian_2d(130, 131)
    b = W.uniform_vector(m.n, 5)
    bt = torch.from_numpy(b).to(torch_dev())

    def solve(A, mx):
        x = torch.zeros_like(bt)
        info = A.solve(bt, x, method="cg", precond="jacobi", tol=1e-10, max_iters=4000, mixed=mx)
        assert info["return"] == gk.GK_OK, info
        assert info["spmv_format"] == layout, info
        assert oracle.true_rel_residual(m, b, x.cpu().numpy()) <= 1e-10
        keys = ("iters", "restarts", "outer_iters", "rel_res_true")
        return x.cpu().numpy(), tuple(info[k] for k in keys)

    want = {}
    for mx in (0, mixed):  # each on a handle of its own
        A = gk.Matrix.from_csr(m)
        want[mx] = solve(A, mx)
        A.close()
    assert want[mixed][1][2] >= 1  # refined, not handed to FP64
    for order in ((0, mixed, mixed, 0, mixed), (mixed, mixed, 0, mixed, 0)):
        A = gk.Matrix.from_csr(m)
        for mx in order:
            x, info = solve(A, mx)
            assert info == want[mx][1], (order, mx)
            assert np.array_equal(x, want[mx][0]), (order, mx)
        A.close()
