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


def _chains(n, k):
    """k interleaved chains: row i depends on row i - k alone."""
    i = np.arange(n)
    table = np.stack([i - k, i, i + k], 1)
    keep = (table >= 0) & (table < n)
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    vals = np.tile([-1.0, 4.0, -1.0], (n, 1))[keep]
    return W.CSR(n, n, rp, table[keep].astype(np.int32), vals)


def test_dependencies_that_all_cross_slabs(monkeypatch):
    """Every row's one dependency lies in another slab, so each level waits for
    one: the window mode is faster, and is what the automatic choice runs."""
    import torch
    m = _chains(60000, 5000)
    r = W.uniform_vector(m.n, 3)
    rt = torch.from_numpy(r).to(torch_dev())
    zt = torch.zeros_like(rt)
    want = oracle.ilu0_apply(m, oracle.ilu0(m), r)
    took = {}
    for mode in ("win", "slab", "auto"):
        if mode == "auto":
            monkeypatch.delenv("GK_ILU_CHUNK")
        else:
            monkeypatch.setenv("GK_ILU_CHUNK", mode)
        A = gk.Matrix.from_csr(m, "f64")
        times = []
        for _ in range(8):
            A.precond_apply(rt, zt, "ilu")
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(20):
                A.precond_apply(rt, zt, "ilu")
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        took[mode] = min(times)
        assert np.array_equal(zt.cpu().numpy(), want), mode
        A.close()
    assert took["auto"] <= 1.2 * min(took["win"], took["slab"]), took


@pytest.mark.parametrize("case", ["chains", "lap1d_128", "lap1d_129", "lap2d_8x16", "lap2d_43x3", "banded_130",
                                  "wide_levels"])
def test_automatic_mode_bit_exact(case):
    import torch
    m = {"chains": lambda: _chains(3001, 400), "lap1d_128": lambda: W.laplacian_1d(128), "lap1d_129": lambda: W.laplacian_1d(129),
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
