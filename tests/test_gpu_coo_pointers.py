"""gk_matrix_create_coo on device triplets at addresses below their types'
alignment: such arrays are copied before a kernel reads them."""
import ctypes

import numpy as np
import pytest

import paper_2510_08230_gb300 as gk
from paper_2510_08230_gb300 import workloads as W
from gpu_util import ensure_built, torch_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _at(a, offset):
    """The bytes of an array on the device, `offset` past an allocation's start."""
    import torch
    raw = torch.from_numpy(np.frombuffer(a.tobytes(), np.uint8).copy())
    buf = torch.empty(raw.numel() + 64, dtype=torch.uint8, device=torch_dev())
    buf[offset:offset + raw.numel()] = raw.to(buf.device)
    return buf, buf.data_ptr() + offset


@pytest.mark.parametrize("offsets", [(0, 0, 0), (1, 0, 0), (0, 2, 0), (0, 0, 4), (3, 2, 1), (4, 4, 8)])
@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
def test_triplets_at_any_address(offsets, dtype):
    import torch
    m = W.power_law(3001, max_len=700, seed=6)
    rng = np.random.default_rng(2)
    perm = rng.permutation(m.nnz)
    row = np.repeat(np.arange(m.n), m.row_lengths())[perm].astype(np.int32)
    col, val = m.col_idx[perm].astype(np.int32), m.values[perm]
    if dtype == "f64":
        values = val
    else:
        values = val.astype(np.float32)
        if dtype == "bf16":  # truncated: any valid bfloat16 will do
            values = (values.view(np.uint32) >> 16).astype(np.uint16)
    keep, ptr = zip(*(_at(a, o) for a, o in zip((row, col, values), offsets)))
    torch.cuda.synchronize()
    h = ctypes.c_void_p()
    dt = {"f64": gk.GK_F64, "f32": gk.GK_F32, "bf16": gk.GK_BF16}[dtype]
    st = gk.lib().gk_matrix_create_coo(m.n, m.ncols, m.nnz, *ptr, dt, gk.GK_MEM_DEVICE,
                                       gk._stream(None), ctypes.byref(h))
    assert st == gk.GK_OK
    rp, ci = np.empty(m.n + 1, np.int32), np.empty(m.nnz, np.int32)
    va = np.empty(m.nnz, values.dtype)
    assert gk.lib().gk_matrix_export(h, rp.ctypes.data, None, ci.ctypes.data,
                                     va.ctypes.data) == gk.GK_OK
    order = np.lexsort((col, row))  # the matrix has no duplicates
    assert np.array_equal(rp, m.row_ptr) and np.array_equal(ci, col[order])
    assert np.array_equal(va, values[order])
    gk.lib().gk_matrix_destroy(h)
