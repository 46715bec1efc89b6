"""Solves that fill the GPU take turns; the time a solve queues for the others
is not device time of its own."""
import threading
import time

import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_device_ms_leaves_the_queue_out():
    """Four solves on full-size grids, which run one at a time: their device
    times add up to no more than the wall clock (with the queue counted they
    would come to about 2.5 times it)."""
    import torch
    m = W.laplacian_1d(1200001)
    As = [gk.Matrix.from_csr(m) for _ in range(4)]
    b = torch.from_numpy(W.uniform_vector(m.n, 3)).to(torch_dev())
    streams = [torch.cuda.Stream() for _ in As]
    xs = [torch.zeros_like(b) for _ in As]
    torch.cuda.synchronize()
    ms = [0.0] * len(As)

    def run(i):
        with torch.cuda.stream(streams[i]):
            xs[i].zero_()
        ms[i] = As[i].solve(b, xs[i], streams[i], method="cg", precond="jacobi", tol=1e-30,
                            max_iters=2000)["device_ms"]

    for i in range(len(As)):  # what a first solve builds
        run(i)
    ts = [threading.Thread(target=run, args=(i,)) for i in range(len(As))]
    t0 = time.perf_counter()
    [t.start() for t in ts]
    [t.join() for t in ts]
    wall = (time.perf_counter() - t0) * 1e3
    assert all(t > 0 for t in ms)
    assert sum(ms) <= 1.2 * wall, (ms, wall)
    for A in As:
        A.close()
