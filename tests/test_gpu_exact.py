"""csrc/exact.h against the operations that it stands for, bit for bit: the
integer conversions against the hardware's, the quotient against the division,
over every exponent, ties, carries into the next exponent, both ends of each
window, subnormals, zeros, infinities and NaN."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1005_5340_gb300 import build
from tests.libutil import ensure_library

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "exact.h"
using namespace tddft;
__global__ void wide(int n, const float *x, double *y, double *z) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  y[i] = to_f64(x[i]);
  z[i] = (double)x[i];
}
__global__ void split(int n, const double *x, __nv_bfloat16 *y, __nv_bfloat16 *z) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  split_f64(x[i], y[2 * i], y[2 * i + 1]);
  z[2 * i] = __double2bfloat16(x[i]);
  z[2 * i + 1] = __double2bfloat16(x[i] - (double)__bfloat162float(z[2 * i]));
}
__global__ void divide(int n, const double *a, const double *b, double *y, double *z) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  y[i] = quotient(a[i], b[i], 1.0 / b[i]);
  z[i] = a[i] / b[i];
}
extern "C" int run_wide(int n, const float *x, double *y, double *z) {
  wide<<<(n + 255) / 256, 256>>>(n, x, y, z);
  return cudaDeviceSynchronize();
}
extern "C" int run_split(int n, const double *x, __nv_bfloat16 *y, __nv_bfloat16 *z) {
  split<<<(n + 255) / 256, 256>>>(n, x, y, z);
  return cudaDeviceSynchronize();
}
extern "C" int run_divide(int n, const double *a, const double *b, double *y, double *z) {
  divide<<<(n + 255) / 256, 256>>>(n, a, b, y, z);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_library()
    d = tmp_path_factory.mktemp("exact")
    (d / "exact.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-cudart", "shared", "-I", build.CSRC, str(d / "exact.cu"), "-o",
                    str(d / "exact.so")], check=True)
    torch.zeros(1, device="cuda")
    return ctypes.CDLL(str(d / "exact.so"))


def call(f, outs, *xs):
    """The two results of f on the device copies of xs (outs: per-entry widths in bytes)."""
    import torch
    n = len(xs[0])
    dev = [torch.from_numpy(x).cuda() for x in xs]
    y, z = (torch.empty(n * outs, dtype=torch.uint8, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    assert f(n, *(ctypes.c_void_p(t.data_ptr()) for t in (*dev, y, z))) == 0
    return y.cpu().numpy(), z.cpu().numpy()


def float64s(rng, exponents, significands):
    """+- every exponent field with every significand, as float64."""
    e, m = np.meshgrid(exponents.astype(np.uint64), significands.astype(np.uint64))
    b = (e << np.uint64(52) | m).ravel()
    return np.concatenate([b, b | np.uint64(1 << 63)]).view(np.float64)


def significands(rng, n):
    """Random ones, those with few bits, and neighbours of ties and of carries at 8 and 16 bits."""
    top = (1 << 52) - 1
    edge = [0, 1, top, top - 1]
    for cut in range(30, 52):   # a tie when all below bit `cut` is cut off, and its neighbours
        for odd in (0, 1, 2, 3, (1 << (51 - cut)) - 1):
            base = (odd << (cut + 1) | 1 << cut) & top
            edge += [base, max(base - 1, 0), min(base + 1, top)]
    r = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    few = r & ~np.uint64((1 << 36) - 1)   # 16 bits: the low part is short, often a tie
    tie = (r & ~np.uint64((1 << 45) - 1)) | np.uint64(1 << 44)
    return np.concatenate([np.array(edge, dtype=np.uint64), r, few, tie])


def test_float32_to_float64(lib):
    rng = np.random.default_rng(1)
    m = np.concatenate([[0, 1, 2, (1 << 23) - 1, 1 << 22], rng.integers(0, 1 << 23, 2000)])
    e, mm = np.meshgrid(np.arange(256, dtype=np.uint32), m.astype(np.uint32))
    b = (e << np.uint32(23) | mm).ravel()
    x = np.concatenate([b, b | np.uint32(1 << 31)]).view(np.float32)
    y, z = call(lib.run_wide, 8, x)
    assert np.array_equal(y, z)


def test_split_of_float64(lib):
    rng = np.random.default_rng(2)
    x = float64s(rng, np.arange(1023 - 70, 1023 + 71), significands(rng, 2000))
    far = float64s(rng, np.array([0, 1, 500, 880, 900, 1150, 1151, 1500, 2046, 2047]),
                   significands(rng, 100))
    y, z = call(lib.run_split, 4, np.concatenate([x, far]))
    y, z = y.view(np.uint16), z.view(np.uint16)
    nan = lambda v: (v & 0x7FFF) > 0x7F80
    assert np.array_equal(nan(y), nan(z)) and np.array_equal(y[~nan(y)], z[~nan(z)])


def test_quotient(lib):
    rng = np.random.default_rng(3)
    a = float64s(rng, rng.integers(900, 1150, 40), significands(rng, 12000))
    b = rng.permutation(a)
    top = (1 << 52) - 1
    ends = np.array([0, 1, 399, 400, 401, 1023, 1646, 1647, 1648, 2046, 2047])
    c = float64s(rng, ends, np.array([0, 1, 12345678901234, top - 1, top]))
    p, q = np.meshgrid(c, c)
    gap = float64s(rng, np.arange(1023 - 252, 1023 + 253), np.array([0, 1, 98765432109876, top]))
    n = np.concatenate([a, p.ravel(), gap])
    d = np.concatenate([b, q.ravel(), gap[::-1]])
    y, z = call(lib.run_divide, 8, n, d)
    y, z = y.view(np.uint64), z.view(np.uint64)
    nan = np.isnan(z.view(np.float64))
    assert np.array_equal(np.isnan(y.view(np.float64)), nan) and np.array_equal(y[~nan], z[~nan])
    with np.errstate(all="ignore"):
        assert np.array_equal((n / d)[~nan].view(np.uint64), z[~nan])
