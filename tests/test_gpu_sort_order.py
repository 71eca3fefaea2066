"""The two device sorts of csrc/mt_dedup.cu are stable: the batched split's
second key and the tip list of the mixed tier rest on it.  Called directly
(a few lines linked with the library's own objects), with many equal keys, at
sizes on both sides of the one-launch sort's limit of 40960, over part of the
key's bits, and with the count on the device."""
from __future__ import annotations

import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHIM = r"""
#include "mt_internal.h"
extern "C" size_t sort_temp(int64_t n) { return mt::radix_temp_bytes(n); }
extern "C" int sort_pairs(uint64_t* k, uint32_t* v, uint64_t* ka, uint32_t* va, int64_t n, void* t,
                          const unsigned long long* n_dev) {
  return (int)mt::radix_sort_pairs(k, v, ka, va, n, t, (cudaStream_t)0, n_dev);
}
extern "C" int sort_bits(uint64_t* k, uint32_t* v, uint64_t* ka, uint32_t* va, int64_t n, void* t, int b, int e,
                         int* in_alt) {
  bool a = false;
  const int rc = (int)mt::radix_sort_bits(k, v, ka, va, n, t, b, e, &a, (cudaStream_t)0);
  *in_alt = a;
  return rc;
}
"""


@pytest.fixture(scope="module")
def sorts(tmp_path_factory):
    from paper_2402_06083_gb300 import build as b
    b.build()
    d = tmp_path_factory.mktemp("sort")
    src, lib = str(d / "shim.cu"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([b.nvcc(), *b.ARCH, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-I", b.INCLUDE, "-I", b.SRC, "-shared",
                    "-cudart", "shared", src, *sorted(glob.glob(os.path.join(b.OUT, "*.o"))), "-o", lib], check=True)
    L = ctypes.CDLL(lib)
    vp = ctypes.c_void_p
    L.sort_temp.restype, L.sort_temp.argtypes = ctypes.c_size_t, [ctypes.c_int64]
    L.sort_pairs.argtypes = [vp, vp, vp, vp, ctypes.c_int64, vp, vp]
    L.sort_bits.argtypes = [vp, vp, vp, vp, ctypes.c_int64, vp, ctypes.c_int, ctypes.c_int, vp]
    return L


def _buffers(L, keys):
    import torch
    k = torch.from_numpy(keys.view(np.int64).copy()).cuda()
    v = torch.arange(keys.size, dtype=torch.int32, device="cuda")
    return k, v, torch.empty_like(k), torch.empty_like(v), torch.empty(L.sort_temp(keys.size), dtype=torch.uint8,
                                                                        device="cuda")


def _keys(n, seed):
    """A few hundred values that differ in one byte at a time."""
    r = np.random.RandomState(seed)
    return (r.randint(0, 6, n).astype(np.uint64) << (8 * r.randint(0, 8, n)).astype(np.uint64)) | \
        (np.uint64(1) << np.uint64(63)) * (r.randint(0, 2, n).astype(np.uint64))


SIZES = [2, 31, 33, 1025, 8191, 8193, 32769, 40959, 40960, 40961, 100003]


@pytest.mark.parametrize("n", SIZES)
def test_whole_keys(sorts, n):
    import torch
    keys = _keys(n, n)
    for live in (n, n - n // 3, 1, 0):
        k, v, ka, va, t = _buffers(sorts, keys)
        nd = torch.tensor([live], dtype=torch.int64, device="cuda")
        assert sorts.sort_pairs(k.data_ptr(), v.data_ptr(), ka.data_ptr(), va.data_ptr(), n, t.data_ptr(),
                                nd.data_ptr() if live < n else None) == 0
        torch.cuda.synchronize()
        order = np.argsort(keys[:live], kind="stable")
        assert np.array_equal(v.cpu().numpy()[:live], order)
        assert np.array_equal(k.cpu().numpy().view(np.uint64)[:live], keys[order])


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("bits", [(0, 40), (8, 24), (16, 24)])
def test_part_of_the_bits(sorts, n, bits):
    import torch
    keys = _keys(n, n + 1)
    k, v, ka, va, t = _buffers(sorts, keys)
    alt = ctypes.c_int(0)
    assert sorts.sort_bits(k.data_ptr(), v.data_ptr(), ka.data_ptr(), va.data_ptr(), n, t.data_ptr(), bits[0], bits[1],
                           ctypes.byref(alt)) == 0
    torch.cuda.synchronize()
    if alt.value:
        k, v = ka, va
    part = (keys >> np.uint64(bits[0])) & np.uint64((1 << (bits[1] - bits[0])) - 1)
    order = np.argsort(part, kind="stable")
    assert np.array_equal(v.cpu().numpy(), order)
    assert np.array_equal(k.cpu().numpy().view(np.uint64), keys[order])
