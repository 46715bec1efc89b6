"""The first ILU(0) application to a new matrix: where the slab mode qualifies,
no other mode is built or timed; on both sides of the size from which it is
tried, the oracle's bits."""
import time

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


def _first(m, rt, zt):
    import torch
    A = gk.Matrix.from_csr(m, "f64")
    torch.cuda.synchronize()
    t = time.perf_counter()
    A.precond_apply(rt, zt, "ilu")
    torch.cuda.synchronize()
    t = time.perf_counter() - t
    A.close()
    return t


def test_first_application_times_slabs_alone(monkeypatch):
    """300 x 200 points: trials of the chunked kernels, at up to 40 ms an
    application, would make the first one take three times as long as with the
    slab mode forced."""
    import torch
    m = W.laplacian_2d(300, 200)
    rt = torch.from_numpy(W.uniform_vector(m.n, 3)).to(torch_dev())
    zt = torch.zeros_like(rt)
    forced, auto = [], []
    for _ in range(4):
        monkeypatch.setenv("GK_ILU_CHUNK", "slab")
        forced.append(_first(m, rt, zt))
        monkeypatch.delenv("GK_ILU_CHUNK")
        auto.append(_first(m, rt, zt))
    assert min(auto) <= 1.5 * min(forced), (auto, forced)


@pytest.mark.parametrize("case", ["lap1d_128", "lap1d_129", "lap2d_8x16", "lap2d_43x3", "banded_130",
                                  "wide_levels"])
def test_automatic_mode_bit_exact(case):
    import torch
    m = {"lap1d_128": lambda: W.laplacian_1d(128), "lap1d_129": lambda: W.laplacian_1d(129),
         "lap2d_8x16": lambda: W.laplacian_2d(8, 16), "lap2d_43x3": lambda: W.laplacian_2d(43, 3),
         "banded_130": lambda: W.banded_spd(130, 5, 3),
         "wide_levels": lambda: W.laplacian_3d(60, 60, 60)}[case]()
    lu = oracle.ilu0(m)
    A = gk.Matrix.from_csr(m, "f64")
    for k in range(3):
        r = W.uniform_vector(m.n, 3 + k)
        rt = torch.from_numpy(r).to(torch_dev())
        zt = torch.zeros_like(rt)
        A.precond_apply(rt, zt, "ilu")
        torch.cuda.synchronize()
        assert np.array_equal(zt.cpu().numpy(), oracle.ilu0_apply(m, lu, r))
    A.close()
