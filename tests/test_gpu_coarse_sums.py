"""The coarsest product's row sums: as exact as FP64 sums in the same order, whatever the
storage type of the cycle, and finite or infinite where those are."""
import ctypes as C
import math

import numpy as np
import pytest

from native import host_library

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdint>
struct CUstream_st;
struct __nv_bfloat16;
namespace dm {
template <typename T>
void dense_coarse_solve(const double*, const float*, int, const int*, const unsigned char*, const T*, T*, CUstream_st*);
}
extern "C" int solve(int bf16, const float* M, int n, const int* list, const void* f, void* x) {
    try {
        if (bf16) dm::dense_coarse_solve<__nv_bfloat16>(nullptr, M, n, list, nullptr, (const __nv_bfloat16*)f, (__nv_bfloat16*)x, nullptr);
        else dm::dense_coarse_solve<float>(nullptr, M, n, list, nullptr, (const float*)f, (float*)x, nullptr);
    } catch (...) { return 1; }
    return 0;
}
"""


@pytest.fixture(scope="module")
def product(dm, tmp_path_factory):
    import torch
    lib = host_library(SOURCE, tmp_path_factory.mktemp("solve"))

    def run(M, f, dtype):
        n = M.shape[0]
        Md = torch.from_numpy(np.ascontiguousarray(M, dtype=np.float32)).cuda()
        fd = torch.from_numpy(f).cuda().to(dtype).contiguous()
        x = torch.zeros(n, dtype=dtype, device="cuda")
        lst = torch.arange(n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        p = lambda t: C.c_void_p(t.data_ptr())
        assert lib.solve(int(dtype == torch.bfloat16), p(Md), n, p(lst), p(fd), p(x)) == 0
        torch.cuda.synchronize()
        return x.double().cpu().numpy()
    return run


def _fp64_rows(M, f):
    """Row sums as one FP64 chain per lane of a warp and a tree over the lanes (the products are exact)."""
    n = M.shape[1]
    pad = -n % 32
    t = np.pad(M.astype(np.float64) * f.astype(np.float64), ((0, 0), (0, pad))).reshape(len(M), -1, 32)
    s = np.zeros((len(M), 32))
    for c in range(t.shape[1]):
        s = s + t[:, c]
    for o in (16, 8, 4, 2, 1):
        s = s[:, :o] + s[:, o:2 * o]
    return s[:, 0]


@pytest.mark.parametrize("n", [34, 256, 2050])
@pytest.mark.parametrize("kind", ["float32", "bfloat16"])
def test_sums_as_exact_as_fp64(n, kind, product):
    import torch
    dtype = getattr(torch, kind)
    rng = np.random.default_rng(n)
    f = torch.from_numpy(rng.standard_normal(n)).to(dtype).float().numpy()
    f[n // 2:] = f[:n // 2]
    M = rng.standard_normal((n, n)).astype(np.float32)
    # every row's products cancel in pairs: the exact sum is zero, and what a sum leaves is its own error
    # (the result's rounding to the storage type is relative to that)
    M[:, n // 2:] = -M[:, :n // 2]
    scale = np.abs(M.astype(np.float64) * f).sum(1)
    rms = lambda v: math.sqrt(np.mean((v / scale) ** 2))
    got, ref = product(M, f, dtype), _fp64_rows(M, f)
    # the lanes' tree is the same; a lane's own sum at least as exact as an FP64 chain's
    assert rms(got) <= 1.05 * rms(ref), (rms(got), rms(ref))


@pytest.mark.parametrize("kind", ["float32", "bfloat16"])
def test_range_of_fp64_sums(kind, product):
    import torch
    n = 70
    big, tiny = 2.0**100, 2.0**-80
    M = np.zeros((n, n), dtype=np.float32)
    f = np.zeros(n, dtype=np.float32)
    f[0], f[32], f[64], f[1], f[33], f[2] = big, big, 1.0, 4.0, -4.0, tiny
    M[0, 0] = big                                          # past FP32 and BF16: infinite, not NaN
    M[1, 0], M[1, 32], M[1, 64] = big, -big, 3.0           # products past FP32 that cancel
    M[2, 1], M[2, 33] = 2.0**126, 2.0**126                 # a lane's sum that reaches FP32's end and comes back
    M[2, 64] = 5.0
    M[3, 2] = -tiny * (1 + 2.0**-6)                        # a product below FP32's smallest, whose sum is zero in FP32
    M[4, 2] = 2.0**-40 * (1 + 2.0**-6)                     # small, but a number of the storage type
    M[5, 0], M[5, 32] = big, big
    x = product(M, f, getattr(torch, kind))
    assert x[0] == math.inf and x[5] == math.inf
    assert x[1] == 3.0 and x[2] == 5.0
    assert x[3] == 0.0 and x[4] == 2.0**-120 * (1 + 2.0**-6)
    assert np.all(x[6:] == 0)
