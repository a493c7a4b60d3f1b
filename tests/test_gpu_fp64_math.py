"""The short double quotients, square roots and float conversions of
`csrc/fp64_math.cuh` against the IEEE operators, bit for bit, on the device:

* quotients a / y (`div`, and `quot_raw` with a shared reciprocal), over edge
  operands (significands of ones, just above a power of two, just below;
  exponents on both sides of where the short form holds), 2^30 random ones, and
  2^30 whose quotient lies within a few ulps of a tie;
* square roots over the same edges, 2^30 random operands and 2^30 squares of
  ties, and x / 3 over 2^30;
* `widen` of all 2^32 floats, and `narrow` of every float's upper tie and the
  doubles next to it, and of 2^30 random doubles around the float range.

A small program is compiled from the header with the flags of the library's
exact and of its fast units and prints the number of mismatches of each."""
import subprocess

import pytest

from paper_1206_0919_gb300 import build as B
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "eos64.cuh"
using namespace shasta;
typedef unsigned long long u64;
enum { DIV, QUOT, SQRT, THIRD, WIDEN, NARROW, DIV_TIE, SQRT_TIE, DIV_EDGE, SQRT_EDGE, NARROW_ANY, KINDS };

__device__ u64 mix(u64 x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
__device__ double make(u64 sig, int e, int sign) {
  return __longlong_as_double((long long)((sig & 0xfffffffffffffull) | ((u64)(e + 1023) << 52) | ((u64)sign << 63)));
}
__device__ double rnd(u64 r, int lo, int hi) { return make(r, lo + (int)((r >> 53) % (u64)(hi - lo)), (int)(r >> 52 & 1)); }
__device__ double step(double x, int k) { return __longlong_as_double(__double_as_longlong(x) + k); }
__device__ bool differ(double a, double b) { return __double_as_longlong(a) != __double_as_longlong(b) && !(a != a && b != b); }
__device__ bool differf(float a, float b) { return __float_as_uint(a) != __float_as_uint(b) && !(a != a && b != b); }

__device__ const u64 kSig[] = {0, 1, 2, 3, 0x8000000000000ull, 0x8000000000001ull, 0x7ffffffffffffull, 0xfffffffffffffull,
                               0xffffffffffffeull, 0xffffffffffffdull, 0x5555555555555ull, 0x6a09e667f3bccull,
                               0x6a09e667f3bcdull, 0xfffffffe00000ull, 0x0000020000000ull};
__device__ const int kExp[] = {-1022, -1021, -901, -900, -899, -501, -500, -499, -401, -400, -399, -60, -2, -1, 0, 1, 2,
                               59, 399, 400, 401, 499, 500, 501, 810, 999, 1000, 1001, 1023};
constexpr int NS = sizeof(kSig) / sizeof(u64), NE = sizeof(kExp) / sizeof(int);

__global__ void run(int kind, u64 n, u64* bad) {
  u64 local = 0;
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const u64 r0 = mix(2 * i + ((u64)kind << 56)), r1 = mix(2 * i + 1 + ((u64)kind << 56));
    if (kind == DIV) {
      const double a = rnd(r0, -520, 520), y = rnd(r1, -420, 420);
      local += differ(f64::div(a, y), a / y);
    } else if (kind == QUOT) {
      const double a = rnd(r0, -500, 500), y = rnd(r1, -400, 400);
      local += differ(f64::quot_raw(a, y, f64::recip_raw(y)), a / y);
    } else if (kind == DIV_TIE) {
      // a within two ulps of y (q + ulp / 2); every eighth y of ones
      const double y = i & 7 ? make(r0, 0, 0) : make(~0ull, (int)(r0 % 5) - 2, 0), q = make(r1, 0, 0);
      const double a = step(fma(y, q, y * 0x1p-53), (int)(r0 >> 60) % 5 - 2);
      local += differ(f64::div(a, y), a / y) + differ(f64::quot_raw(a, y, f64::recip_raw(y)), a / y);
    } else if (kind == SQRT) {
      const double x = fabs(rnd(r0, -920, 1010));
      local += differ(f64::sqrt(x), ::sqrt(x));
    } else if (kind == SQRT_TIE) {
      const double s = make(r0, (int)(r1 % 3) - 1, 0);
      const double x = step(fma(s, s, s * 0x1p-53 * (r1 & 8 ? 2.0 : 1.0)), (int)(r1 >> 60) % 5 - 2);
      local += differ(f64::sqrt(x), ::sqrt(x)) + differ(f64::sqrt_raw(x), ::sqrt(x));
    } else if (kind == THIRD) {
      const double x = rnd(r0, -1000, 1020);
      local += differ(f64::third(x), x / 3.0) + differ(f64::third(step(0.0, (int)(i & 0xffff))), step(0.0, (int)(i & 0xffff)) / 3.0);
    } else if (kind == WIDEN) {
      const float f = __uint_as_float((unsigned)i);
      local += differ(f64::widen(f), (double)f);
    } else if (kind == NARROW) {
      const float f = __uint_as_float((unsigned)i);
      const double t = make(0, 0, 0) * (double)f;  // the tie above f, by the bit pattern of the double
      const double x = __longlong_as_double(__double_as_longlong(t) + 0x10000000ll);
      for (int k = -1; k < 2; ++k) local += differf(f64::narrow<float>(step(x, k)), (float)step(x, k));
    } else if (kind == NARROW_ANY) {
      const double x = rnd(r0, -160, 140);
      local += differf(f64::narrow<float>(x), (float)x);
    } else {
      const u64 s0 = kSig[i % NS], s1 = kSig[i / NS % NS];
      const int e0 = kExp[i / (NS * NS) % NE], e1 = kExp[i / (NS * NS * NE) % NE];
      const double a = make(s0, e0, (int)(i & 1)), y = make(s1, e1, (int)(i >> 1 & 1));
      if (kind == DIV_EDGE)
        local += differ(f64::div(a, y), a / y) + differ(f64::div(0.0, y), 0.0 / y) + differ(f64::div(a, 0.0), a / 0.0);
      else
        local += differ(f64::sqrt(a), ::sqrt(a)) + differ(f64::sqrt(i & 2 ? 0.0 : -0.0), ::sqrt(i & 2 ? 0.0 : -0.0));
    }
  }
  if (local) atomicAdd(bad, local);
}

int main() {
  u64 *bad, h[KINDS];
  if (cudaMalloc(&bad, sizeof h) != cudaSuccess || cudaMemset(bad, 0, sizeof h) != cudaSuccess) return 2;
  const u64 edge = (u64)NS * NS * NE * NE, many = 1ull << 30;
  for (int k = 0; k < KINDS; ++k)
    run<<<152 * 8, 256>>>(k, k == WIDEN || k == NARROW ? 1ull << 32 : k == DIV_EDGE || k == SQRT_EDGE ? edge : many, bad + k);
  if (cudaMemcpy(h, bad, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  for (int k = 0; k < KINDS; ++k) std::printf("%llu\n", h[k]);
  return 0;
}
"""
NAMES = ["div", "quot_raw", "sqrt", "third", "widen", "narrow at ties", "div near ties", "sqrt near ties", "div edges",
         "sqrt edges", "narrow"]


@pytest.mark.parametrize("flags", ["EXACT", "FAST"])
def test_short_forms_against_ieee(tmp_path, flags):
    require_gpu()
    src, exe = tmp_path / "ops.cu", tmp_path / "ops"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc()] + B.ARCH + B.COMMON + getattr(B, flags) + [str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.returncode
    bad = dict(zip(NAMES, map(int, r.stdout.split())))
    assert len(bad) == len(NAMES) and not any(bad.values()), bad
