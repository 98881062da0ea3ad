"""The register groups of the fused sorting passes at their edges: one block and
the first sizes beyond, every count of keys per thread, and float keys that are
all ordinary or hold a single special one (the thread block with it then
compares as IEEE <=, the others by minimum and maximum or as integers).  The
kernel looks for special keys by the extremes of their bits, so NaN of either
sign and -0.0 come alone, and for doubles also what the high word cannot tell
from them: infinities and the smallest negative numbers.  Bit for bit the host
emulation of the same plan."""

import ctypes

import numpy as np
import pytest

from paper_2306_07795_gb300 import _binding as B

pytestmark = pytest.mark.gpu

KEYS = {np.float32: B.BMMC_KEY_F32, np.float64: B.BMMC_KEY_F64, np.int32: B.BMMC_KEY_I32,
        np.uint64: B.BMMC_KEY_U64}


def _keys(dtype, count, special, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    if not np.issubdtype(dtype, np.floating):
        info = np.iinfo(dtype)
        x = g.integers(info.min, info.max, size=count, dtype=dtype, endpoint=True)
        x[g.integers(0, count, 4)] = info.min
        x[g.integers(0, count, 4)] = info.max
        return x
    x = g.standard_normal(count).astype(dtype)
    x[g.integers(0, count, 8)] = 0.0
    x[g.integers(0, count, 4)] = np.finfo(dtype).smallest_subnormal
    x[g.integers(0, count, 4)] = -np.finfo(dtype).max
    if dtype == np.float32:  # ordinary keys in 4 bytes
        x[g.integers(0, count, 2)] = np.inf
        x[g.integers(0, count, 2)] = -np.inf
        x[g.integers(0, count, 2)] = -np.finfo(dtype).smallest_subnormal
    if special is not None:
        x[g.integers(0, count)] = special
    return x


SPECIAL = [np.nan, np.copysign(np.nan, -1.0), -0.0]
SPECIAL64 = SPECIAL + [np.inf, -np.inf, -np.finfo(np.float64).smallest_subnormal]


def test_keys_are_as_ordinary_as_they_say():
    """What the kernel takes for special, restated: no key without `special`,
    one with."""
    for dtype, special in [(np.float32, v) for v in [None] + SPECIAL] + \
            [(np.float64, v) for v in [None] + SPECIAL64]:
        x = _keys(dtype, 1 << 8, special, 1)
        odd = np.isnan(x) | ((x == 0) & np.signbit(x))
        if dtype == np.float64:
            odd |= np.isinf(x) | ((x < 0) & (x > -2.0 ** -1042))
        assert odd.sum() == (0 if special is None else 1)


@pytest.mark.parametrize("dtype,special", [(np.float32, None)] +
                         [(np.float32, v) for v in SPECIAL] + [(np.float64, None)] +
                         [(np.float64, v) for v in SPECIAL64] +
                         [(np.int32, None), (np.uint64, None)])
@pytest.mark.parametrize("n,b,block_log2", [(7, 0, 0), (8, 0, 0), (9, 0, 0), (11, 0, 0), (12, 0, 0),
                                            (13, 0, 0), (13, 0, 16), (14, 0, 16), (15, 1, 15),
                                            (8, 6, 0), (20, 0, 0)])
def test_groups(n, b, block_log2, dtype, special):
    import torch
    x = _keys(dtype, 1 << (n + b), special, n * 10 + b)
    h = B.bmmc_sort_plan_create(n, b, KEYS[dtype], block_log2)
    want = np.empty_like(x)
    B.bmmc_sort_plan_emulate(h, ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(want.ctypes.data))
    d = torch.from_numpy(x.view(np.int32 if x.itemsize == 4 else np.int64).copy()).cuda()
    y = torch.full_like(d, -1)
    ws = torch.empty(max(16, B.bmmc_sort_workspace_bytes(h)), dtype=torch.uint8, device="cuda")
    B.bmmc_sort_execute(h, d.data_ptr(), y.data_ptr(), ws.data_ptr(),
                        torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    B.bmmc_sort_plan_destroy(h)
    got = y.cpu().numpy().view(dtype)
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))


@pytest.mark.parametrize("n,b", [(5, 10), (10, 6), (10, 10)])
@pytest.mark.parametrize("dtype", [np.int32, np.uint64])
def test_rows_without_workspace(n, b, dtype):
    """Rows that fit a thread block are one pass: no workspace, and one that is
    passed all the same is left alone."""
    import torch
    x = _keys(dtype, 1 << (n + b), None, n + b)
    h = B.bmmc_sort_plan_create(n, b, KEYS[dtype])
    assert B.bmmc_sort_workspace_bytes(h) == 0
    d = torch.from_numpy(x.view(np.int32 if x.itemsize == 4 else np.int64).copy()).cuda()
    y, z, ws = (torch.full_like(d, -1) for _ in range(3))
    s = torch.cuda.current_stream().cuda_stream
    B.bmmc_sort_execute(h, d.data_ptr(), y.data_ptr(), None, s)
    B.bmmc_sort_execute(h, d.data_ptr(), z.data_ptr(), ws.data_ptr(), s)
    torch.cuda.synchronize()
    B.bmmc_sort_plan_destroy(h)
    want = np.sort(x.reshape(1 << b, 1 << n), axis=1).reshape(-1)
    assert np.array_equal(y.cpu().numpy().view(dtype), want)
    assert torch.equal(y, z)
    assert bool((ws == -1).all())
