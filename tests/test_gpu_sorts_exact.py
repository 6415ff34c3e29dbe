"""The radix sorts against numpy's stable sort, keys and values, at the edges of
their forms: one block (4,096 keys), the cluster (163,840; 262,144 with the
count on the device), three kernels a pass, and at even and odd pass counts
(the result of an odd number is copied back)."""
import ctypes as C

import numpy as np
import pytest
import torch

import native_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sort_case(tmp_path_factory):
    torch.cuda.set_device(0)
    m = native_build.load("sorts", tmp_path_factory.mktemp("native"), objects=True)
    m.sort_case.argtypes = [C.c_void_p, C.c_void_p, C.c_int64, C.c_int, C.c_int, C.c_int,
                            C.c_void_p, C.c_void_p]
    return m.sort_case


def _check(sort_case, n, count, key_bytes, vals, lo, bits, seed):
    g = np.random.default_rng(seed)
    dt = np.uint64 if key_bytes == 8 else np.uint32
    keys = g.integers(0, 2**min(bits + 5, 8 * key_bytes), n, dtype=dt, endpoint=False)
    keys[g.integers(0, n, n // 3)] = keys[0]  # equal keys: the order must be stable
    v = np.arange(n, dtype=np.uint32)
    dk = torch.from_numpy(keys.view(np.uint8)).cuda()
    dv = torch.from_numpy(v.view(np.int32)).cuda()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    dn = None if count is None else torch.tensor([count], dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    rc = sort_case(dk.data_ptr(), dv.data_ptr() if vals else None, n, key_bytes, lo, bits,
                   None if dn is None else dn.data_ptr(), err.data_ptr())
    assert rc == 0
    m = n if count is None else min(count, n)
    # whole 8-bit digits from lo until `bits` is reached (a last, partial digit
    # takes the bits above it along; the library's keys have none there)
    width = min(8 * -(-(bits - lo) // 8), 8 * key_bytes - lo)
    field = (keys[:m] >> dt(lo)) & dt((1 << width) - 1)
    order = np.argsort(field, kind="stable")
    assert np.array_equal(dk.cpu().numpy().view(dt)[:m], keys[:m][order])
    if vals:
        assert np.array_equal(dv.cpu().numpy().view(np.uint32)[:m], v[:m][order])


@pytest.mark.parametrize("vals", [False, True])
@pytest.mark.parametrize("key_bytes,lo,bits", [(8, 0, 48), (8, 0, 40), (8, 8, 48), (8, 3, 40),
                                               (8, 0, 64), (4, 0, 32), (4, 0, 24)])
@pytest.mark.parametrize("n", [2, 4096, 4097, 163840, 163841, 300001])
def test_host_count(sort_case, n, key_bytes, lo, bits, vals):
    _check(sort_case, n, None, key_bytes, vals, lo, bits, n + bits + lo)


@pytest.mark.parametrize("vals", [False, True])
@pytest.mark.parametrize("lo,bits", [(0, 48), (1, 41)])
@pytest.mark.parametrize("cap", [5000, 163841, 262144, 262145])
@pytest.mark.parametrize("count", [0, 1, 4096, 4097, 163841, 262144, 10**6])
def test_device_count(sort_case, cap, count, lo, bits, vals):
    _check(sort_case, cap, count, 8, vals, lo, bits, cap + count + lo)
