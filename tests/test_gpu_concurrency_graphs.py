"""First solves on the multi-kernel engine from several threads at once: each
captures its CUDA graphs while the others capture theirs, upload and destroy
matrices.  engine=1, since the automatic engine takes most of these solves to
kernels that capture nothing."""
import threading

import numpy as np
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built
from test_gpu_concurrency import CASES, _solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def test_captures_at_once_equal_sequential():
    import torch
    cases = [(c(), dict(kw, engine=1)) for c, kw in CASES]
    seq = {}
    for i, (m, kw) in enumerate(cases):
        _solve(m, kw, torch.cuda.Stream(), seq, i, None)
        assert seq[i][0]["block_threads"] == 0  # no persistent kernel
    for rep in range(3):
        par, stop = {}, threading.Event()
        start = threading.Barrier(len(cases) + 1)

        def churn():
            start.wait()
            k = 0
            while not stop.is_set():
                gk.Matrix.from_csr(W.laplacian_2d(64 + k % 7)).close()
                k += 1

        ths = [threading.Thread(target=_solve, args=(m, kw, torch.cuda.Stream(), par, i, start))
               for i, (m, kw) in enumerate(cases)]
        ch = threading.Thread(target=churn)
        for t in ths + [ch]:
            t.start()
        for t in ths:
            t.join(300)
        stop.set()
        ch.join(60)
        for i in range(len(cases)):
            info, x = par[i]
            assert info["return"] == gk.GK_OK, (rep, i, info)
            assert info["iters"] == seq[i][0]["iters"], (rep, i)
            assert np.array_equal(x, seq[i][1]), (rep, i)
