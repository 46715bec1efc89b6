"""The slab mode's waits on other slabs take the caller's budget."""
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


def test_wait_on_other_slabs_keeps_the_budget(monkeypatch):
    """700 x 300 points: some 300 levels lie before the last slab's first, none
    of which takes less than the 0.3 us of its dependent operations, so its
    block waits for longer than 50 us; a copy of a level's records lands well
    within that.  The budget runs out there and nowhere on a value that never
    comes, and the next application is exact."""
    import torch
    monkeypatch.setenv("GK_ILU_CHUNK", "slab")
    m = W.laplacian_2d(700, 300)
    A = gk.Matrix.from_csr(m, "f64")
    r = W.uniform_vector(m.n, 8)
    rt = torch.from_numpy(r).to(torch_dev())
    zt = torch.zeros_like(rt)
    want = oracle.ilu0_apply(m, oracle.ilu0(m), r)
    for budget, status in ((0, gk.GK_OK), (50_000, gk.GK_ERR_TIMEOUT), (1_000_000_000, gk.GK_OK)):
        zt.zero_()
        assert gk.gk_precond_apply(A.handle, "ilu", 0, rt, zt, budget) == status, budget
        torch.cuda.synchronize()
        assert (A.describe()["device_error"] != 0) == (status != gk.GK_OK)
        if status == gk.GK_OK:
            assert np.array_equal(zt.cpu().numpy(), want)
    for upper in (False, True):
        A.triangular_solve(rt, zt, upper=upper)
        st = gk.lib().gk_triangular_solve(A.handle, int(upper), 0, rt.data_ptr(), zt.data_ptr(),
                                          50_000, gk._stream(None))
        assert st == gk.GK_ERR_TIMEOUT
        A.triangular_solve(rt, zt, upper=upper)
        torch.cuda.synchronize()
        assert np.array_equal(zt.cpu().numpy(), oracle.trsv(m, r, upper=upper))
    A.close()
