"""The FP32 primitives of gv_device.cuh against the operations they stand for,
bit by bit: f2d against the conversion on every float, div_rn against the
IEEE quotient, Divisor against the approximate division it shares a reciprocal
for.  The kernels are compiled from the header here."""
import ctypes as C
import os
import subprocess

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "gv_device.cuh"
using namespace gv;

__device__ __forceinline__ bool same(float a, float b) { return a == b ? signbit(a) == signbit(b) : a != a && b != b; }
__device__ __forceinline__ bool same(double a, double b) { return a == b ? signbit(a) == signbit(b) : a != a && b != b; }

// all 2^32 floats; bad[0]: how many differ, bad[1]: one of them
__global__ void k_widen(unsigned long long *bad) {
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * blockDim.x;
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; i < 1ull << 32; i += stride) {
    const float f = __uint_as_float(static_cast<unsigned>(i));
    if (!same(f2d(f), static_cast<double>(f))) {
      atomicAdd(&bad[0], 1ull);
      bad[1] = i;
    }
  }
}

// n pairs of random bits; lo, hi: the divisors' exponents (biased)
__device__ void draw(unsigned long long i, unsigned lo, unsigned hi, float &a, float &b) {
  const uint4 w = philox4x32_10(make_uint4(static_cast<unsigned>(i), static_cast<unsigned>(i >> 32), 0u, 0u), 17u, 4u);
  a = __uint_as_float(w.x);
  b = __uint_as_float((w.y & 0x807fffffu) | (lo + w.z % (hi - lo + 1u)) << 23);
  if (i % 4 == 0) b = __uint_as_float(__float_as_uint(b) | 0x007ffff0u);  // next to a power of two from below
  if (i % 4 == 1) a = __uint_as_float(__float_as_uint(a) & 0xff800007u);  // and from above
}

// div_rn over what its comment states: divisor, quotient and residual normal,
// or a special numerator or divisor, or an overflowing quotient
__global__ void k_div(unsigned long long n, unsigned long long *bad) {
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * blockDim.x;
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    float a, b;
    draw(i, 1u, 253u, a, b);
    if (i % 64 == 7) a = 0.0f * a;
    if (i % 64 == 13) a = a < 0.0f ? -INFINITY : INFINITY;
    if (i % 64 == 21) b = b < 0.0f ? -INFINITY : INFINITY;
    if (i % 64 == 33) b = 0.0f * b;
    const float q = __fdiv_rn(a, b), m = fabsf(q);
    const bool special = a == 0.0f || isinf(a) || isinf(b) || b == 0.0f || a != a;
    const bool overflow = fabs(static_cast<double>(a) / b) > 3.5e38;
    const bool normal = m >= 1.17549435e-38f && m < 1.7e38f && fabsf(a) >= 2.0e-31f;  // (residual: 2^-24 of the numerator)
    if (!(special || overflow || normal)) continue;
    atomicAdd(&bad[2], 1ull);
    if (!same(div_rn(a, b), q)) {
      atomicAdd(&bad[0], 1ull);
      bad[1] = (static_cast<unsigned long long>(__float_as_uint(a)) << 32) | __float_as_uint(b);
    }
  }
}

// Divisor against __fdividef; lo, hi as above (0: zeros and subnormals)
__global__ void k_shared(unsigned long long n, unsigned lo, unsigned hi, unsigned long long *bad) {
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * blockDim.x;
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    float a, b;
    draw(i, lo, hi, a, b);
    if (i % 8 == 3) a = 0.0f;
    atomicAdd(&bad[2], 1ull);
    if (!same(Divisor<float>(b).div(a), __fdividef(a, b))) {
      atomicAdd(&bad[0], 1ull);
      bad[1] = (static_cast<unsigned long long>(__float_as_uint(a)) << 32) | __float_as_uint(b);
    }
  }
}

extern "C" int run(int what, unsigned long long n, unsigned lo, unsigned hi, unsigned long long *bad) {
  if (what == 0) k_widen<<<1216, 256>>>(bad);
  if (what == 1) k_div<<<1216, 256>>>(n, bad);
  if (what == 2) k_shared<<<1216, 256>>>(n, lo, hi, bad);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_2005_00949_gb300 import build
    d = tmp_path_factory.mktemp("arith")
    src, out = d / "arith.cu", d / "arith.so"
    src.write_text(SOURCE)
    subprocess.check_call([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                           "-I", os.path.join(ROOT, "paper_2005_00949_gb300", "csrc"), "-shared", "-o", str(out), str(src)])
    lib = C.CDLL(str(out))
    lib.run.argtypes = [C.c_int, C.c_ulonglong, C.c_uint, C.c_uint, C.c_void_p]

    def call(what, n=0, lo=0, hi=0):
        bad = torch.zeros(3, dtype=torch.int64, device="cuda")
        assert lib.run(what, n, lo, hi, bad.data_ptr()) == 0
        return [int(x) for x in bad.cpu()]
    return call


def test_widening_is_exact_on_every_float(run):
    bad, which, _ = run(0)
    assert bad == 0, (bad, hex(which))


def test_div_rn_is_the_ieee_quotient(run):
    bad, which, checked = run(1, 1 << 28)
    assert checked > 1 << 26
    assert bad == 0, (bad, hex(which))


@pytest.mark.parametrize("lo, hi", [(1, 252), (0, 0)], ids=["normal", "subnormal"])
def test_divisor_is_the_approximate_division(run, lo, hi):
    bad, which, checked = run(2, 1 << 26, lo, hi)
    assert checked > 1 << 24
    assert bad == 0, (bad, hex(which))
