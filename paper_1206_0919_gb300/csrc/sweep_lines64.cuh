// sweep_lines64.cuh -- FP64 SHASTA sweep, whole lines in shared memory, sm_103a.
//
// The same arithmetic as sweep.cuh's streaming kernel, bit for bit, at 0.37 of
// its double instructions.  GB300 does 2 double operations per SM and clock
// against 128 in FP32, so a double sweep is bound by the number of its double
// instructions and by nothing else: here a block holds B whole lines in shared
// memory and runs the sweep stage by stage over all their cells, so that
//  * every quantity is computed once per cell (the streaming form forms each
//    difference of U and Uhat three times) and no position twice: segments of
//    a line re-run a 12-position halo, 1.75x the work at 16-cell segments;
//  * ghost cells cost nothing on reflecting and periodic lines: their velocity
//    and Uhat are read from the cell they mirror (the arithmetic is ordered
//    symmetrically, so mirrored data give mirrored bits);
//  * limiter, comparisons, signs and powers of two are integer operations;
//  * quotients and roots come from fp64_math.cuh, and the transport factors of
//    neighbouring cells share a reciprocal (Q+_j and Q-_{j+1} have the same
//    denominator 1 + eps_{j+1} - eps_j).
// About 240 double operations per cell are left (the streaming kernel executes
// 641).  Shared-memory traffic and the block barriers between stages hide
// behind the double pipe.
// Measured, streaming -> here (us a sweep): 64^3 507 -> 151, 143 x 129 x 151
// 3588 -> 1497, 200^3 8925 -> 4306; the double pipe is 83% busy (85-87% is the
// most any kernel here reaches, with no barriers in it).
#pragma once

#include "chain.cuh"
#include "eos64.cuh"
#include "lines_plan.h"
#include "sweep.cuh"

namespace shasta {
namespace lines64 {

// Launch geometry: B lines per block; NP = n + 6 positions held per line, of
// pitch js from position to position and ls from line to line; sz doubles per
// array.
// eta_exp: k where eta = 2^-k (the method's 1/8: 3), else 0.
struct LineArgs {
  int B, js, ls, sz, eta_exp;
};


using f64::bits;

// Limiter of Sec. 3, s max(0, min(s dhp, |aph|, s dhm)), by the bit patterns:
// nonnegative doubles order as integers.  Infinities and NaN take the
// floating-point form.
__device__ __forceinline__ double limit(double aph, double dhp, double dhm) {
  if (max(max(f64::mag(aph), f64::mag(dhp)), f64::mag(dhm)) >= 0x7ff00000u) {
    const double sg = (aph > 0.0) ? 1.0 : ((aph < 0.0) ? -1.0 : 0.0);
    return sg * fmax(0.0, fmin(fmin(sg * dhp, fabs(aph)), sg * dhm));
  }
  const long long s = bits(aph) & (1ll << 63);
  const long long a = bits(aph) ^ s;
  const long long m = min(min(bits(dhp) ^ s, a), bits(dhm) ^ s);  // a negative one is below zero
  if (a == 0) return 0.0;
  return __longlong_as_double(max(m, 0ll) | s);
}

// eta x, by the exponent where eta is a power of two.
__device__ __forceinline__ double times_eta(double x, double eta, int k) {
  if (f64::is_zero(x)) return x;  // (eta >= 0)
  if (k == 0 || f64::mag(x) - 0x04000000u >= 0x7ff00000u - 0x04000000u) return eta * x;
  return __hiloint2double(f64::hi(x) - (k << 20), __double2loint(x));
}

// m/h for h in [2^-401, 2^401) and any |m| <= h, m != 0: the momentum in the
// tail of a front runs through all magnitudes down to the smallest, and is
// divided 2^400 higher where its residual would leave the range.
__device__ __forceinline__ double far_quot(double m, double h) {
  const bool low = f64::mag(m) < (unsigned)((-500 + 1023) << 20);
  const double ms = low ? f64::scale<400>(m) : m;
  const double q = f64::quot_raw(ms, h, f64::recip_raw(h));
  if (!low) return q;
  // m normal and the quotient normal after the way back, else IEEE division
  if (f64::mag(m) >= (1u << 20) && f64::mag(q) >= (unsigned)(402 << 20)) return f64::scale<-400>(q);
  return f64::ieee_div(m, h);
}

// (out of line, so that the common cells never pay for it by predication)
template <int EOS, int AXIS>
__device__ __noinline__ unsigned recover_rest(double E, double m1, double m2, double m3, double omd, double B,
                                              double ec, const EosTable& T, double& w, double& p) {
  return recover_wp<double, EOS, AXIS>(E, m1, m2, m3, omd, B, ec, T, w, p);
}

// recover_wp of sweep.cuh; cells outside the range the fast forms hold in
// (and clamped ones, and vacuum) take it as it stands.
template <int EOS, int AXIS>
__device__ __forceinline__ unsigned recover(double E, double m1, double m2, double m3, double omd, double B,
                                            double ec, const EosTable& T, double& w, double& p) {
  const double X = AXIS == 0 ? m1 : m2;
  const double Y = AXIS == 0 ? m2 : (AXIS == 1 ? m1 : m3);
  const double Z = AXIS == 2 ? m1 : m3;
  const double M2 = (X * X + Y * Y) + Z * Z;
  // below 2^-470 M changes no bit of what is formed from it and such an E
  // (E +- M, 4 E^2 - 3 M^2, the clamp), so the far tails of a front count as at rest
  const bool still = f64::mag(M2) < (unsigned)((-940 + 1023) << 20);
  if (f64::hi(E) > 0 && f64::within<-400, 400>(E) && (still || f64::within<-940, 810>(M2))) {
    const double M = still ? 0.0 : f64::sqrt_raw(M2);
    if (bits(M) <= bits(omd * E)) {
      double e;
      if constexpr (EOS == EOS_TABLE)
        f64::table_solve(E, M, T, e, p);
      else
        f64::closed_root<EOS>(E, M, B, ec, e, p);
      const double h = E + p;
      if (f64::is_zero(m1))
        w = m1;  // (h > 0)
      else
        w = far_quot(m1, h);
      return 0;
    }
  }
  return recover_rest<EOS, AXIS>(E, m1, m2, m3, omd, B, ec, T, w, p);
}

template <int EOS, int AXIS>
__global__ void __launch_bounds__(kLinesMaxThreads) sweep_lines_kernel(SweepParams P, LineArgs A) {
  extern __shared__ __align__(16) double sm[];
  const int n = P.n, bc = P.bc;
  const bool frozen = bc == BC_FROZEN;
  const long long t0 = (long long)blockIdx.x * A.B;
  const int nl = (int)min((long long)A.B, P.plane - t0);  // lines of this block
  // line l of the block at position j sits at at(j, l) of each array
  auto at = [&](int j, int l) { return (j + NG) * A.js + l * A.ls; };
  auto arr = [&](int k) { return sm + (size_t)k * A.sz; };
  double* const U = arr(0);    // 5 fields in sweep order: E, M along the line, the other two, R
  double* const D = arr(5);    // Delta_j = U_{j+1} - U_j
  double* const D2 = arr(10);  // (Delta_{j+1} + Delta_{j-1}) - 2 Delta_j
  double* const EV = arr(15);  // eps = tau v
  double* const Pv = arr(16);
  double* const PW = arr(17);
  double* const UH = arr(18);
  double* const DH = arr(23);
  double* const AF = arr(28);
  double* const QP = AF;         // transport factors: read before the fluxes are written
  double* const QM = AF + A.sz;
  const int sz = A.sz;

  // one item per (position in [lo, hi), line)
  auto each = [&](int lo, int hi, auto f) {
    const int m = hi - lo, items = m * nl;
    for (int i = threadIdx.x; i < items; i += blockDim.x) {
      int j, l;
      if (AXIS == 0) {
        l = i / m;
        j = lo + (i - l * m);
      } else {
        j = i / nl;
        l = i - j * nl;
        j += lo;
      }
      f(j, l);
    }
  };
  // the cell whose value a ghost position holds, and whether it is a mirror
  auto src = [&](int j, bool& mir) {
    mir = false;
    if (frozen || (j >= 0 && j < n)) return j;
    if (bc == BC_PERIODIC) return j < 0 ? j + n : j - n;
    mir = true;
    return j < 0 ? -1 - j : 2 * n - 1 - j;
  };
  auto flip = [](double x, bool f) {  // by the sign bit: a double negation would be a double addition
    return __hiloint2double(f64::hi(x) ^ (f ? 0x80000000 : 0), __double2loint(x));
  };

  chain_begin();
  // ---- the old state, ghosts included
  each(-NG, n + NG, [&](int j, int l) {
    const long long t = t0 + l;
    const long long base = (t % P.nb) * P.sb + (t / P.nb) * P.sc;
    double v[NF];
    load_ext<double, AXIS>(P, base, t, j, v);
    const int o = at(j, l);
#pragma unroll
    for (int k = 0; k < NF; ++k) U[k * sz + o] = v[k];
  });
  __syncthreads();
  // ---- recovery at level n, Delta
  unsigned nclamp = 0;
  each(frozen ? -NG : 0, frozen ? n + NG : n, [&](int j, int l) {
    const int o = at(j, l);
    double w, p;
    const unsigned c = recover<EOS, AXIS>(U[o], U[sz + o], U[2 * sz + o], U[3 * sz + o], P.omd, P.bag_B, P.bag_ec,
                                          P.tab, w, p);
    if (j >= 0 && j < n) nclamp += c;
    EV[o] = P.tau_h * w;
    Pv[o] = p;
    PW[o] = p * w;
  });
  each(frozen ? -NG : -2, frozen ? n + 2 : n + 1, [&](int j, int l) {
    const int o = at(j, l);
#pragma unroll
    for (int k = 0; k < NF; ++k) D[k * sz + o] = U[k * sz + o + A.js] - U[k * sz + o];
  });
  __syncthreads();
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int nf = h == 0 ? 4 : NF;  // the half step leaves R out
    const double ht = h == 0 ? P.htau_h : P.htau_f;
    // eps of position j; a frozen ghost keeps the eps of the half step, half of it
    auto eps = [&](int j, int l) {
      bool m;
      const double e = flip(EV[at(src(j, m), l)], m);
      return frozen && h && (j < 0 || j >= n) ? e + e : e;
    };
    // ---- transport factors from the denominator at j + 1/2, second differences
    each(frozen ? -NG : -1, frozen ? n + NG - 1 : n, [&](int j, int l) {
      const double e0 = eps(j, l), e1 = eps(j + 1, l);
      const double den = 1.0 + (e1 - e0);
      const double np = 0.5 - e0, nm = 0.5 + e1;
      const int o = at(j, l);
      if (f64::hi(den) > 0 && f64::within<-200, 200>(den) && f64::mag(np) < 0x5f000000u &&
          f64::mag(nm) < 0x5f000000u && f64::mag(np) - 1u >= 0x20000000u - 1u &&
          f64::mag(nm) - 1u >= 0x20000000u - 1u) {
        const double r = f64::recip_raw(den);
        QP[o] = f64::quot_raw(np, den, r);
        QM[o + A.js] = f64::quot_raw(nm, den, r);
      } else {
        QP[o] = f64::ieee_div(np, den);
        QM[o + A.js] = f64::ieee_div(nm, den);
      }
    });
    if (h == 0)
      each(-1, n, [&](int j, int l) {
        const int o = at(j, l);
#pragma unroll
        for (int k = 0; k < NF; ++k) {
          const double* d = D + k * sz + o;
          D2[k * sz + o] = fma(-2.0, d[0], d[A.js] + d[-A.js]);
        }
      });
    __syncthreads();
    // ---- transported values
    each(frozen ? -2 : 0, frozen ? n + 2 : n, [&](int j, int l) {
      const int o = at(j, l);
      const double qp = QP[o], qm = QM[o];
      // twice the coefficients of Eq. shasta-geo; the half goes into the last sum, exactly
      const double a = qp * qp, b = qm * qm, c = qp + qm;
      bool ml, mr;
      const int ol = at(src(j - 1, ml), l), orr = at(src(j + 1, mr), l);
      const double sE = ht * (flip(PW[ol], ml) - flip(PW[orr], mr));
      const double sM = ht * (Pv[ol] - Pv[orr]);
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        if (k < nf) {
          const double* d = D + k * sz + o;
          double u = fma(0.5, a * d[0] - b * d[-A.js], c * U[k * sz + o]);
          if (k == 0) u = u + sE;
          if (k == 1) u = u + sM;
          UH[k * sz + o] = u;
        }
      }
    });
    __syncthreads();
    // ---- their differences
    each(-2, n + 1, [&](int j, int l) {
      bool m0, m1;
      const int o0 = at(src(j, m0), l), o1 = at(src(j + 1, m1), l), o = at(j, l);
#pragma unroll
      for (int k = 0; k < NF; ++k)
        if (k < nf)
          DH[k * sz + o] = flip(UH[k * sz + o1], k == 1 && m1) - flip(UH[k * sz + o0], k == 1 && m0);
    });
    __syncthreads();
    // ---- limited antidiffusive fluxes through the face j + 1/2
    each(-1, n, [&](int j, int l) {
      const int o = at(j, l);
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        if (k < nf) {
          const double* dh = DH + k * sz + o;
          const double aph = times_eta(fma(-0.125, D2[k * sz + o], dh[0]), P.eta, A.eta_exp);
          AF[k * sz + o] = limit(aph, dh[A.js], dh[-A.js]);
        }
      }
    });
    __syncthreads();
    // ---- the new values: recovered (half step) or stored (full step)
    each(0, n, [&](int j, int l) {
      const int o = at(j, l);
      double v[NF];
#pragma unroll
      for (int k = 0; k < NF; ++k)
        v[k] = k < nf ? UH[k * sz + o] - (AF[k * sz + o] - AF[k * sz + o - A.js]) : 0.0;
      if (h == 0) {
        double w, p;
        recover<EOS, AXIS>(v[0], v[1], v[2], v[3], P.omd, P.bag_B, P.bag_ec, P.tab, w, p);
        EV[o] = P.tau_f * w;
        Pv[o] = p;
        PW[o] = p * w;
        return;
      }
      constexpr int FPAR = 1 + AXIS, FT1 = AXIS == 0 ? 2 : 1, FT2 = AXIS == 2 ? 2 : 3;
      const long long t = t0 + l;
      const long long i = (t % P.nb) * P.sb + (t / P.nb) * P.sc + (long long)j * P.stride;
      if (!SH_OK(P, i >= 0 && i < P.ncap, 3, i)) return;
      static_cast<double*>(P.out[0])[i] = v[0];
      static_cast<double*>(P.out[FPAR])[i] = v[1];
      static_cast<double*>(P.out[FT1])[i] = v[2];
      static_cast<double*>(P.out[FT2])[i] = v[3];
      static_cast<double*>(P.out[4])[i] = v[4];
    });
    if (h == 0) __syncthreads();
  }
  add_clamps(P.clamp_count, nclamp);
}

}  // namespace lines64
}  // namespace shasta
