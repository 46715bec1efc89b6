"""Products of one CSR matrix on several streams at once.  The products of a
matrix without rows longer than 1024 entries share nothing but the matrix,
whichever kernel its plan picks: streams have carry buffers of their own,
those that come too late and captured products do without."""
import numpy as np
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import TOL, assert_rows_close, ensure_built, oracle_apply, torch_dev, vec_dtype

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _rows(lengths, ncols, seed):
    rng = np.random.default_rng(seed)
    lengths = np.asarray(lengths)
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    col = rng.integers(0, ncols, int(rp[-1])).astype(np.int32)
    return W.CSR(len(lengths), ncols, rp, col, rng.standard_normal(int(rp[-1])))


def _lengths(kind):
    rng = np.random.default_rng(23)
    if kind == "exponential":  # rows of 8 entries on average, some empty
        return np.minimum(rng.exponential(8.0, 1_500_000).astype(np.int64), 1024)
    if kind == "long":         # rows over many units of 256 entries
        return rng.integers(0, 1025, 20_000)
    return np.minimum(rng.zipf(1.8, 300_000), 1024)


@pytest.mark.parametrize("kind", ["exponential", "long", "zipf"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_products_at_once(kind, dtype):
    """Seven streams, more than have buffers, and a captured graph beside them;
    every product within the tolerance of the oracle, and on the streams with
    buffers the one it is alone, bit for bit."""
    import torch
    m = _rows(_lengths(kind), 400_000, 3)
    A = gk.Matrix.from_csr(m, dtype)
    assert A.desc["spmv_kernel"] == 2
    dev, vt = torch_dev(), vec_dtype(dtype)
    streams = [torch.cuda.Stream() for _ in range(7)]
    xs = [torch.from_numpy(W.uniform_vector(m.ncols, 3 + k)).to(dev, vt) for k in range(8)]
    y0 = torch.from_numpy(W.uniform_vector(m.n, 9)).to(dev, vt)
    ys = [y0.clone() for _ in xs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        A.apply_adv(-0.5, xs[7], 1.5, ys[7])

    def all_at_once(wait):
        for y in ys:
            y.copy_(y0)
        torch.cuda.synchronize()
        for x, y, s in zip(xs, ys, streams):
            A.apply_adv(-0.5, x, 1.5, y, s)
            if wait:
                s.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        return [y.clone() for y in ys]

    want = all_at_once(True)
    for x, w in zip(xs, want):
        ref, scale = oracle_apply(m, x.cpu().numpy(), -0.5, 1.5, y0.cpu().numpy(), dtype)
        assert_rows_close(w.cpu().numpy(), ref, scale, TOL[dtype], f"{kind} {dtype}")
    for _ in range(10):
        for got, w in zip(all_at_once(False), want):
            assert torch.equal(got, w)
    A.close()


# Rows of exactly 1024 entries against one of 1025 (which has one carry buffer
# for all streams), and rows that reach across units of 256 entries by 1 entry
# and more, from one unit to several.
def _across(width, heads):
    """Rows of at most 1024 entries; a row begins k entries before each
    multiple of width, k from heads, and ends at most 1024 later."""
    lengths, at = [], 0
    for b, k in enumerate(heads, 1):
        rest = b * width - k - at
        while rest > 0:
            lengths.append(min(rest, 1000))
            rest -= lengths[-1]
        lengths.append(k + 1 + (7 * k) % max(1, min(1024 - k, 100)))
        at = b * width - k + lengths[-1]
    return lengths


HEADS = {
    "whole_units": [1024] * 9,
    "one_entry_early": [255] + [1024] * 4 + [1],
    "one_entry_late": [257] + [1024] * 4 + [3],
    "last_unit": [100, 1000],
    "limit": [1024, 7, 0, 0, 900, 1024, 33] * 2,
    "past_limit": [1025, 7, 0, 0, 900, 1024, 33] * 2,
    "across_units": _across(256, range(1, 120)),
    "across_blocks": _across(2048, range(1, 45)),
    "far_across_blocks": _across(2048, range(900, 1024, 7)),
    "short_rows": [1, 2, 3, 0, 5, 64, 9] * 150,
}


@pytest.mark.parametrize("name", list(HEADS))
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16", "f16"])
def test_rows_across_units(monkeypatch, name, dtype):
    import torch
    monkeypatch.setenv("GK_CSR_KERNEL", "2")
    m = _rows(HEADS[name], 3000, 5)
    A = gk.Matrix.from_csr(m, dtype)
    assert A.desc["spmv_kernel"] == 2
    x, y0 = W.uniform_vector(m.ncols, 6), W.uniform_vector(m.n, 7)
    xt = torch.from_numpy(x).to(torch_dev(), vec_dtype(dtype))
    streams = [torch.cuda.Stream() for _ in range(5)]
    for s in streams:  # the last one comes too late for a buffer
        A.apply(xt, torch.empty(m.n, dtype=xt.dtype, device=xt.device), s)
    late = streams[-1]
    for alpha, beta in ((1.0, 0.0), (2.5, 0.0), (-1.0, 1.0), (0.5, -2.0)):
        ref, scale = oracle_apply(m, x, alpha, beta, y0 if beta else None, dtype)
        for stream in [None] + ([late] if max(HEADS[name]) <= 1024 else []):
            yt = torch.from_numpy(y0).to(torch_dev(), vec_dtype(dtype))
            torch.cuda.synchronize()
            A.apply_adv(alpha, xt, beta, yt, stream)
            torch.cuda.synchronize()
            assert_rows_close(yt.cpu().numpy(), ref, scale, TOL[dtype],
                              f"{name} {dtype} {alpha} {beta}")
    A.close()
