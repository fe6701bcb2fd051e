"""The integer square root with its reciprocal (fp_convert.cuh, used by the Cholesky leaf
and the stop test) and the branch-free scaled conversion of the folds, against the host's
correctly rounded operations: every result is the same bits.

Squares and their neighbours, both parities of the exponent, significands of all ones,
subnormals, the ends of the range and infinity, for the root; carries and ties for the conversion.  The
kernels are compiled here from the header, which is what the library's kernels inline."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <stdint.h>
#include "fp_convert.cuh"
__global__ void roots(int64_t n, const double *x, double *root, double *rcp) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) omm::sw_sqrt_rcp(x[i], root[i], rcp[i]);
}
__global__ void scaled(int64_t n, const uint64_t *a, const int *e, double *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = omm::sw_u64_scaled(a[i], (i & 1) != 0, e[i]);
}
extern "C" int run_roots(int64_t n, const double *x, double *root, double *rcp) {
    roots<<<(unsigned)((n + 255) / 256), 256>>>(n, x, root, rcp);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_scaled(int64_t n, const uint64_t *a, const int *e, double *out) {
    scaled<<<(unsigned)((n + 255) / 256), 256>>>(n, a, e, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2209_05934_gb300 import build
    d = tmp_path_factory.mktemp("roots")
    src, so = d / "roots.cu", d / "roots.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    "-shared", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def test_root_and_reciprocal_are_correctly_rounded(lib):
    rng = np.random.default_rng(0)
    n = 1 << 20
    bits = (rng.integers(1, 0x7FF, n).astype(np.uint64) << np.uint64(52)) | rng.integers(0, 1 << 52, n, dtype=np.uint64)
    s = rng.integers(1 << 26, 1 << 27, 1 << 18).astype(np.float64)
    sq = np.ldexp(s * s, rng.integers(-500, 400, s.size))                     # exact squares
    ones = ((rng.integers(1, 0x7FF, 4096).astype(np.uint64) << np.uint64(52)) | np.uint64((1 << 52) - 1)).view(np.float64)
    pow2 = np.ldexp(1.0, np.arange(-1074, 1024))
    sub = rng.integers(1, 1 << 52, 1 << 16, dtype=np.uint64).view(np.float64)
    x = np.concatenate([bits.view(np.float64), sq, np.nextafter(sq, 0), np.nextafter(sq, np.inf), ones, pow2,
                        np.nextafter(pow2, 0), sub, [5e-324, np.finfo(np.float64).max, np.inf]])
    x = x[x > 0]
    t = torch.from_numpy(x).cuda()
    root, rcp = torch.empty_like(t), torch.empty_like(t)
    assert lib.run_roots(ctypes.c_int64(x.size), ptr(t), ptr(root), ptr(rcp)) == 0
    r = np.sqrt(x)
    np.testing.assert_array_equal(root.cpu().numpy().view(np.uint64), r.view(np.uint64))
    np.testing.assert_array_equal(rcp.cpu().numpy().view(np.uint64), (1.0 / r).view(np.uint64))


def test_scaled_conversion_is_correctly_rounded(lib):
    rng = np.random.default_rng(1)
    n = 1 << 19
    a = rng.integers(0, 1 << 64, n, dtype=np.uint64) >> rng.integers(0, 64, n).astype(np.uint64)
    sh = rng.integers(1, 11, n).astype(np.uint64)
    tie = (rng.integers(1 << 52, 1 << 53, n, dtype=np.uint64) << sh) | (np.uint64(1) << (sh - np.uint64(1)))
    carry = np.uint64(2 ** 64 - 1) - rng.integers(0, 1 << 12, 1 << 14, dtype=np.uint64)
    a = np.concatenate([a, tie, carry, np.array([0, 0, 1, 1, 2 ** 63, 2 ** 64 - 1], dtype=np.uint64)])
    e = rng.integers(-960, 900, a.size).astype(np.int32)
    ta, te = torch.from_numpy(a.view(np.int64)).cuda(), torch.from_numpy(e).cuda()
    out = torch.empty(a.size, dtype=torch.float64, device="cuda")
    assert lib.run_scaled(ctypes.c_int64(a.size), ptr(ta), ptr(te), ptr(out)) == 0
    ref = np.ldexp(a.astype(np.float64), e) * np.where((np.arange(a.size) & 1) & (a != 0), -1.0, 1.0)
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), ref.view(np.uint64))
