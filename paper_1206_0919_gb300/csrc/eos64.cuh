// eos64.cuh -- roots of the equations of state in double for the FP64-bound
// kernels: the expressions of sweep.cuh's eos_solve and eos_table_solve with
// the quotients and roots of fp64_math.cuh (same bits).  For E in [2^-400,
// 2^400) and 0 <= M <= E.
#pragma once

#include "fp64_math.cuh"
#include "sweep.cuh"

namespace shasta {
namespace f64 {

// Floor and fraction of any x by the conversions.
static __device__ __noinline__ double split_rest(double x, int last, int& k) {
  k = __double2int_rd(x);
  k = k < 0 ? 0 : (k > last ? last : k);
  return x - (double)k;
}
// k = floor(x) held in [0, last] and x - k.  By the bit pattern inside the
// table: the two conversions and the subtraction would each take a slot of the
// double pipe, 3 of a lookup's 9 (64^3 FP64 table event: 1797 us a step, 1623 so;
// 130^3 11.5 ms, 10.2).
__device__ __forceinline__ double split(double x, int last, int& k) {
  const int ex = (hi(x) >> 20) - 1023;  // (negative x: far below 0)
  if (ex < 0 && hi(x) >= 0) {
    k = 0;
    return x;
  }
  if ((unsigned)ex < 31u) {
    const int sh = 52 - ex;
    const unsigned long long m = ((unsigned long long)bits(x) & 0xfffffffffffffull) | (1ull << 52);
    k = (int)(m >> sh);
    if (k <= last) {
      const unsigned long long r = m & ((1ull << sh) - 1);
      const int up = __clzll((long long)r) - 11;  // (r = 0: any)
      const unsigned long long f = ((r << up) & 0xfffffffffffffull) + ((unsigned long long)(1023 + ex - up) << 52);
      return __longlong_as_double((long long)(r ? f : 0ull));
    }
  }
  return split_rest(x, last, k);
}

// p(e) of the table (table_p64), rde = recip_raw(T.de).
__device__ __forceinline__ double table_at(const EosTable& T, double rde, double e) {
  const bool z = is_zero(e);
  double x;
  if ((z || within<-500, 500>(e)) && within<-400, 400>(T.de)) {
    const double q = e * rde;
    x = z ? q : fma(fma(-T.de, q, e), rde, q);
  } else {
    x = ieee_div(e, T.de);
  }
  int k;
  const double f = split(x, T.n - 2, k);
  const double a = __ldg(T.p64 + k), b = __ldg(T.p64 + k + 1);
  return a + f * (b - a);
}

// The fixed point of Sec. 3 (eos_table_solve).
__device__ __forceinline__ void table_solve(double E, double M, const EosTable& T, double& e, double& p) {
  const double rde = recip_raw(T.de);
  double v = div(M, E + table_at(T, rde, E));
  for (int it = 0; it < 200; ++it) {
    const double vn = div(M, E + table_at(T, rde, E - M * v));
    const double d = vn - v;
    v = vn;
    if ((bits(d) & ~(1ll << 63)) <= bits(1e-14)) break;
  }
  e = E - M * v;
  p = table_at(T, rde, e);
}

// x / 3 for any x: 1/3 is the correctly rounded reciprocal.
__device__ __forceinline__ double third(double x) {
  if (within<-900, 1000>(x)) return quot_raw(x, 3.0, 1.0 / 3.0);
  return is_zero(x) ? x : ieee_div(x, 3.0);
}

// The closed roots (eos_solve).
template <int EOS>
__device__ __forceinline__ void closed_root(double E, double M, double B, double ec, double& e, double& p) {
  const double m3 = (3.0 * M) * M;
  const double s = sqrt_raw((scale<2>(E) * E) - m3);
  const double EM = (E - M) * (E + M);
  const double se = s + E;
  const double pa = quot_raw(EM, se, recip_raw(se));
  const double ea = 3.0 * pa;
  e = ea;
  p = pa;
  if constexpr (EOS == EOS_BAG) {
    if (ea <= ec) return;
    if (E > ec) {
      const double r = (4.0 * (E - B)) * (E - B) - m3;
      if (r >= 0.0) {
        const double sb = f64::sqrt(r);
        const double eb = div(3.0 * EM - (4.0 * B) * E, sb + (E - 2.0 * B));
        if (eb > ec) {
          e = eb;
          p = third(eb - 4.0 * B);
          return;
        }
      }
    }
    e = ec;
    p = div(M * M, E - ec) - E;
  }
}

}  // namespace f64
}  // namespace shasta
