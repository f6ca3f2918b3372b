"""The double-float conversions that work on the words of their operands give the bits of the FP64 instructions for every
input (ties, carries into the next binade, powers of two with a low word of either sign, both edges of the fast range,
signed zeros, denormals, infinities, NaN, pairs that are not normalised, random patterns), and the quotient without FP64
division is within 2^-44 of it wherever it is formed."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_00947_gb300", "csrc")
KERNELS = r"""
#include "df64.cuh"
using namespace mgar;
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
__global__ void k_from(const double* x, int n, unsigned* bad) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const df a = df_from_double(x[i]), b = df_from_double_fp(x[i]);
    if (!same(a.hi, b.hi) || !same(a.lo, b.lo)) atomicAdd(bad, 1u);
  }
}
__global__ void k_to(const float2* x, int n, unsigned* bad) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const df v{x[i].x, x[i].y};
    if (__double_as_longlong(df_to_double(v)) != __double_as_longlong(df_to_double_fp(v))) atomicAdd(bad, 1u);
  }
}
// err: the relative error in units of 2^-44, or -1 where no quotient is formed
__global__ void k_quotient(const double* a, const double* b, int n, double* err) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    df p;
    if (!df_quotient(a[i], b[i], p)) { err[i] = -1.0; continue; }
    const double q = a[i] / b[i];
    err[i] = fabs((((double)p.hi - q) + (double)p.lo) / q) * 0x1p44;
  }
}
extern "C" {
int from_double(const double* x, int n, unsigned* bad) { k_from<<<512, 256>>>(x, n, bad); return cudaDeviceSynchronize(); }
int to_double(const float2* x, int n, unsigned* bad) { k_to<<<512, 256>>>(x, n, bad); return cudaDeviceSynchronize(); }
int quotient(const double* a, const double* b, int n, double* err) {
  k_quotient<<<512, 256>>>(a, b, n, err);
  return cudaDeviceSynchronize();
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("df64")
    (d / "words.cu").write_text(KERNELS)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "words.so"), str(d / "words.cu")], check=True)
    return ctypes.CDLL(str(d / "words.so"))


def doubles():
    rng = np.random.default_rng(1)
    out = [rng.integers(0, 1 << 64, 1 << 22, dtype=np.uint64)]
    # exponents across the fast range and around its ends (949 and 1149), every significand at which the 29 low bits
    # round: just below, at and just above a tie, for an even and an odd last bit, and with a carry out of the word
    low = np.array([0, 1, 2, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1], dtype=np.uint64)
    top = np.array([0, 1, 2, 3, (1 << 23) - 2, (1 << 23) - 1, 0x2AAAAA, 0x555555], dtype=np.uint64)
    sig = (top[:, None] << np.uint64(29) | low[None, :]).reshape(-1)
    exp = np.arange(2048, dtype=np.uint64) << np.uint64(52)
    v = (exp[:, None] | sig[None, :]).reshape(-1)
    out += [v, v | np.uint64(1 << 63)]
    return np.concatenate(out)


def pairs():
    rng = np.random.default_rng(2)
    n = 1 << 21
    out = [rng.integers(0, 1 << 32, (n, 2), dtype=np.uint32)]
    # normalised pairs of every size, and low words at and about half a unit of the high one
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-140, 127, n)) * rng.choice([-1.0, 1.0], n)
    hi = x.astype(np.float32)
    lo = (x - hi.astype(np.float64)).astype(np.float32)
    out.append(np.stack([hi, lo], 1).view(np.uint32))
    sig = np.array([0, 1, 2, 0x7FFFFE, 0x7FFFFF, 0x400000], dtype=np.uint32)
    exp = np.arange(256, dtype=np.uint32)
    h = (exp[:, None] << 23 | sig[None, :]).reshape(-1).astype(np.uint32)
    hf = h.view(np.float32)
    e = np.clip(h >> 23, 1, 254).astype(np.int64) - 127
    for scale in (-24, -25, -30, -52, -53, -54, -55, -77, -78):
        for m in (0.0, 1.0, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -23, 1.5, 1.25):
            lo = np.ldexp(m, e + scale).astype(np.float32)
            for a in (hf, -hf):
                for b in (lo, -lo):
                    out.append(np.stack([a, b], 1).astype(np.float32).view(np.uint32))
    return np.concatenate(out)


def test_from_double(lib):
    x = torch.tensor(doubles().view(np.int64), device=DEV)
    bad = torch.zeros(1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert lib.from_double(ctypes.c_void_p(x.data_ptr()), x.numel(), ctypes.c_void_p(bad.data_ptr())) == 0
    assert int(bad) == 0


def test_to_double(lib):
    x = torch.tensor(pairs().view(np.int32), device=DEV)
    bad = torch.zeros(1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert lib.to_double(ctypes.c_void_p(x.data_ptr()), x.shape[0], ctypes.c_void_p(bad.data_ptr())) == 0
    assert int(bad) == 0


def test_quotient(lib):
    rng = np.random.default_rng(3)
    n = 1 << 20
    a, b = (np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-70, 70, n)) * rng.choice([-1.0, 1.0], n) for _ in range(2))
    # at the limits of the exponents' difference, and operands that have no quotient here
    for d in (-101, -100, -99, 99, 100, 101):
        a, b = np.append(a, np.ldexp(1.75, d)), np.append(b, 1.25)
    for v in (0.0, -0.0, 5e-324, np.inf, np.nan):
        a, b = np.append(a, [v, 1.0]), np.append(b, [1.0, v])
    ea, eb = ((v.view(np.int64) >> 52 & 0x7FF) for v in (a, b))
    formed = (ea != 0) & (ea != 0x7FF) & (eb != 0) & (eb != 0x7FF) & (np.abs(ea - eb) <= 100)
    err = torch.empty(a.size, dtype=torch.float64, device=DEV)
    ad, bd = torch.tensor(a, device=DEV), torch.tensor(b, device=DEV)
    torch.cuda.synchronize()
    assert lib.quotient(ctypes.c_void_p(ad.data_ptr()), ctypes.c_void_p(bd.data_ptr()), a.size,
                        ctypes.c_void_p(err.data_ptr())) == 0
    e = err.cpu().numpy()
    np.testing.assert_array_equal(e >= 0, formed)
    assert e[formed].max() <= 1.0
