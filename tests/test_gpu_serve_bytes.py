"""The serving loop's estimate of what an ILU(0) solve keeps on the device is
no less than what it keeps."""
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from paper_2510_08230_gb300.serve import ilu_bytes
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu

GRAIN = 2 << 20  # the device hands memory out in pieces of 2 MB


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("name", ["lap3d_100", "lap2d_1000", "banded"])
def test_ilu_bytes_cover_what_is_kept(name):
    import torch
    m = {"lap3d_100": lambda: W.laplacian_3d(100), "lap2d_1000": lambda: W.laplacian_2d(1000),
         "banded": lambda: W.banded_spd(50000, 20, 3)}[name]()
    A = gk.Matrix.from_csr(m, "f64")
    r = torch.from_numpy(W.uniform_vector(m.n, 3)).to(torch_dev())
    z = torch.zeros_like(r)
    warm = gk.Matrix.from_csr(W.laplacian_3d(20))  # the kernels' code and stacks
    warm.precond_apply(r[:8000], z[:8000], "ilu")
    A.apply(r, z)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    A.precond_apply(r, z, "ilu")
    torch.cuda.synchronize()
    kept = free - torch.cuda.mem_get_info()[0]
    assert kept <= ilu_bytes(m, False) + 16 * GRAIN, (kept, ilu_bytes(m, False))
    A.close()
    warm.close()
