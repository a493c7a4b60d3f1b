// aux.cu -- state conversion, primitive <-> conserved maps, input checks,
// deterministic totals and the frozen ghost store.  Built with -fmad=false:
// these maps evaluate each expression of Sec. 2 in plain double precision, in
// source order (fused operations are written out, where they give the same
// bits); quotients and roots are the correctly rounded ones of fp64_math.cuh.
#include <math.h>

#include "eos64.cuh"
#include "kernels.h"

namespace shasta {

namespace {

constexpr int kThreads = 256;
constexpr int kCells = 4;  // cells per thread of the copies: 20 loads in flight

inline unsigned grid_for(size_t n) {
  size_t b = (n + kThreads - 1) / kThreads;
  return (unsigned)(b > 65535u * 32u ? 65535u * 32u : (b == 0 ? 1 : b));
}

// Cell i of a state: (E, Mx, My, Mz) and R.  FP32 states hold the four as one
// aligned quad (FieldView::s of 4), FP64 states five dense arrays.
template <class T>
struct Cell {
  T v[5];
};
__device__ __forceinline__ Cell<float> load_cell(const FieldView& f, size_t i, float) {
  const float4 q = static_cast<const float4*>(f.p[0])[i];
  return Cell<float>{{q.x, q.y, q.z, q.w, static_cast<const float*>(f.p[4])[i]}};
}
__device__ __forceinline__ Cell<double> load_cell(const FieldView& f, size_t i, double) {
  Cell<double> c;
#pragma unroll
  for (int k = 0; k < 5; ++k) c.v[k] = static_cast<const double*>(f.p[k])[i];
  return c;
}
__device__ __forceinline__ void store_cell(const FieldView& f, size_t i, const Cell<float>& c) {
  static_cast<float4*>(f.p[0])[i] = make_float4(c.v[0], c.v[1], c.v[2], c.v[3]);
  static_cast<float*>(f.p[4])[i] = c.v[4];
}
__device__ __forceinline__ void store_cell(const FieldView& f, size_t i, const Cell<double>& c) {
#pragma unroll
  for (int k = 0; k < 5; ++k) static_cast<double*>(f.p[k])[i] = c.v[k];
}

struct In5 {
  const double* f[5];
};
struct Out6 {
  double* f[6];
};

// The fields of cell i that `out` asks for (FP32: the quad where any of its four
// is): a get of one field reads 16 or 4 bytes of a float cell and 8 of a double
// one, not all of it (320^3, one field of FP64 235 -> 97 us; E of FP32 287 -> 127,
// R 286 -> 79; all five 327 -> 299).
__device__ __forceinline__ Cell<float> load_some(const FieldView& f, const Out6& out, size_t i, float) {
  float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float r = 0.0f;
  if (out.f[0] || out.f[1] || out.f[2] || out.f[3]) q = static_cast<const float4*>(f.p[0])[i];
  if (out.f[4]) r = static_cast<const float*>(f.p[4])[i];
  return Cell<float>{{q.x, q.y, q.z, q.w, r}};
}
__device__ __forceinline__ Cell<double> load_some(const FieldView& f, const Out6& out, size_t i, double) {
  Cell<double> c;
#pragma unroll
  for (int k = 0; k < 5; ++k) c.v[k] = out.f[k] ? static_cast<const double*>(f.p[k])[i] : 0.0;
  return c;
}

// Conversions between the caller's five arrays and a state, all fields of a
// cell at once.  Bound by memory: one pass over 60 (FP32) or 80 (FP64) bytes
// per cell; field by field, the quads were rewritten (or re-read) four times
// in 4-byte pieces.  512^3, FP32: set 1.13 ms, get 1.23 ms, 7.1 and 6.6 TB/s
// (a pass of check, set, six steps and get took 33.4 ms field by field, 27.9 ms
// so).
template <class T>
__global__ void __launch_bounds__(kThreads) k_set_cons(In5 in, FieldView out, size_t lo, size_t hi) {
  const size_t i0 = lo + blockIdx.x * (size_t)(kThreads * kCells) + threadIdx.x;
  double v[kCells][5];
#pragma unroll
  for (int u = 0; u < kCells; ++u)
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (i0 + u * kThreads < hi) v[u][k] = in.f[k][i0 + u * kThreads];
#pragma unroll
  for (int u = 0; u < kCells; ++u)
    if (i0 + u * kThreads < hi)
      store_cell(out, i0 + u * kThreads,
                 Cell<T>{{T(v[u][0]), T(v[u][1]), T(v[u][2]), T(v[u][3]), T(v[u][4])}});
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_get_cons(FieldView in, Out6 out, size_t n) {
  const size_t i0 = blockIdx.x * (size_t)(kThreads * kCells) + threadIdx.x;
  Cell<T> c[kCells];
#pragma unroll
  for (int u = 0; u < kCells; ++u)
    if (i0 + u * kThreads < n) c[u] = load_some(in, out, i0 + u * kThreads, T());
  // (widened by the bit patterns: conversion instructions go through the double
  // pipe, and predicated off they still take their slots)
#pragma unroll
  for (int k = 0; k < 5; ++k)
    if (out.f[k]) {
#pragma unroll
      for (int u = 0; u < kCells; ++u)
        if (i0 + u * kThreads < n) out.f[k][i0 + u * kThreads] = f64::widen(c[u].v[k]);
    }
}

__device__ __forceinline__ double eos_p(const EosParams& q, double e) {
  if (q.kind == EOS_TABLE) return table_p64(q.tab, e);
  if (q.kind == EOS_BAG && e > q.ec) return f64::third(e - 4.0 * q.B);
  return f64::third(e);
}

// Sec. 2: R = n gamma, M = (e + p) gamma^2 v, E = (e + p) gamma^2 - p.
// Bound by its double instructions (about 30).
template <class T>
__global__ void k_prim2cons(In5 in, FieldView out, size_t n, EosParams q) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    double e = in.f[0][i], vx = in.f[1][i], vy = in.f[2][i], vz = in.f[3][i], nb = in.f[4][i];
    double v2 = (vx * vx + vy * vy) + vz * vz;
    double g2 = f64::div(1.0, 1.0 - v2);
    double pr = eos_p(q, e);
    double w = (e + pr) * g2;
    store_cell(out, i, Cell<T>{{f64::narrow<T>(w - pr), f64::narrow<T>(w * vx), f64::narrow<T>(w * vy),
                             f64::narrow<T>(w * vz), f64::narrow<T>(nb * f64::sqrt(g2))}});
  }
}

// The root of the tabulated EoS for the primitive map: where the iteration of
// Sec. 3 ends (its next change at most 1e-14), reached another way.  Newton
// steps in float, then two or three from the residual M - v (E + p) in double,
// whose quotient and Newton factor 1 / g' in float are all the accuracy a
// correction needs: about 12 double operations a step, where the plain
// iteration takes about 12 steps of 18, each gaining a factor v^2 p'.  The
// plain one stops up to 2e-15 short of the root in v, this one 3e-16 (E up to
// 150, |v| to 1 - 1e-9, three tables).  Sweeps keep the iteration's own bits.
// A 96^3 FP32 event of 24 steps with its primitives read once: 2640 -> 2090 us.
// What has not settled after six steps, and states far from 1, take it here.
__device__ __noinline__ double2 table_rest(double E, double M, EosTable T) {
  double2 r;
  f64::table_solve(E, M, T, r.x, r.y);
  return r;
}
__device__ __forceinline__ void table_root(double E, double M, const EosTable& T, double& e, double& p) {
  const double rde = f64::recip_raw(T.de);
  if (f64::is_zero(M)) {
    e = E;
    p = f64::table_at(T, rde, E);
    return;
  }
  if (f64::within<-60, 100>(E) && f64::within<-60, 100>(M)) {
    const float Ef = f64::narrow<float>(E), Mf = f64::narrow<float>(M);
    float vf = Mf * __fdividef(1.0f, Ef + tab32(T, Ef));
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
      float dp;
      const float r = __fdividef(1.0f, Ef + tab32(T, fmaf(-Mf, vf, Ef), &dp));
      const float mr = Mf * r;
      const float d = __fdividef(fmaf(-Mf, r, vf), fmaf(-mr * mr, dp, 1.0f));
      vf -= d;
      if (fabsf(d) <= 3e-7f) break;
    }
    double v = f64::widen(vf);
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
      const double r = E + f64::table_at(T, rde, fma(-M, v, E));
      if (!f64::within<-60, 120>(r)) break;
      float dp;
      tab32(T, fmaf(-Mf, vf, Ef), &dp);
      const float d = f64::narrow<float>(fma(-v, r, M)) * __fdividef(1.0f, f64::narrow<float>(r));
      const float s = __fdividef(d, fmaf(-vf * vf, dp, 1.0f));
      v += f64::widen(s);
      vf += s;
      if (fabsf(d) <= 1e-14f) {
        e = fma(-M, v, E);
        p = f64::table_at(T, rde, e);
        return;
      }
    }
  }
  const double2 r = table_rest(E, M, T);
  e = r.x;
  p = r.y;
}

// The recovery of a cell that leaves the range of the short forms, is clamped
// or is vacuum.
__device__ __noinline__ void recover_rest(double E, const double m[3], double R, const EosParams& q, double o[6]) {
  double e = 0.0, v[3] = {0.0, 0.0, 0.0}, nb = 0.0, pp = 0.0;
  if (E > 0.0) {
    double M = ::sqrt((m[0] * m[0] + m[1] * m[1]) + m[2] * m[2]);
    double lim = q.omd * E;
    double scale = 1.0;
    if (M > lim) {
      scale = lim / M;
      M = lim;
    }
    if (q.kind == EOS_TABLE)
      eos_table_solve(E, M, q.tab, e, pp);
    else if (q.kind == EOS_BAG)
      eos_solve<double, EOS_BAG>(E, M, q.B, q.ec, e, pp);
    else
      eos_solve<double, EOS_IDEAL>(E, M, q.B, q.ec, e, pp);
    const double ih = 1.0 / (E + pp);
    for (int a = 0; a < 3; ++a) v[a] = ((scale == 1.0) ? m[a] : m[a] * scale) * ih;
    nb = R * ::sqrt((e + pp) * ih);
  }
  o[0] = e;
  o[1] = v[0];
  o[2] = v[1];
  o[3] = v[2];
  o[4] = nb;
  o[5] = pp;
}

// Sec. 3 phases 3-4 for every cell: e, v, n, p (double arithmetic).
// v = M / (E + p) and n = R sqrt(1 - v^2) = R sqrt((e + p) / (E + p)) with one
// reciprocal of E + p.  Bound by its double instructions: 102 per cell with
// the IEEE operators, about 57 here (200^3 FP32: 1296 -> 923 us).
template <class T, int EOS>
__global__ void __launch_bounds__(kThreads) k_recover(FieldView in, Out6 out, size_t n, EosParams q) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const Cell<T> c = load_cell(in, i, T());
    const double E = f64::widen(c.v[0]), R = f64::widen(c.v[4]);
    const double m[3] = {f64::widen(c.v[1]), f64::widen(c.v[2]), f64::widen(c.v[3])};
    // (squares of float momenta are exact in double: fused sums round alike)
    const double M2 = sizeof(T) == 4 ? fma(m[2], m[2], fma(m[1], m[1], m[0] * m[0]))
                                     : (m[0] * m[0] + m[1] * m[1]) + m[2] * m[2];
    const bool still = f64::is_zero(M2);
    double o[6];
    bool done = false;
    if (f64::hi(E) > 0 && f64::within<-400, 400>(E) && (still || f64::within<-940, 810>(M2))) {
      const double M = still ? 0.0 : f64::sqrt_raw(M2);
      if (f64::bits(M) <= f64::bits(q.omd * E)) {
        if constexpr (EOS == EOS_TABLE)
          table_root(E, M, q.tab, o[0], o[5]);
        else
          f64::closed_root<EOS>(E, M, q.B, q.ec, o[0], o[5]);
        const double h = E + o[5];
        const double ih = f64::quot_raw(1.0, h, f64::recip_raw(h));
#pragma unroll
        for (int a = 0; a < 3; ++a) o[1 + a] = m[a] * ih;
        o[4] = R * f64::sqrt((o[0] + o[5]) * ih);
        done = true;
      }
    }
    if (!done) recover_rest(E, m, R, q, o);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (out.f[k]) out.f[k][i] = o[k];
  }
}

// Finite: the exponent field is not all ones.
__device__ __forceinline__ bool finite(double x) { return f64::mag(x) < 0x7ff00000u; }
__device__ __forceinline__ bool negative(double x) { return f64::hi(x) < 0 && !f64::is_zero(x); }

// Whether x^2 + y^2 + z^2 is below (1 - 2^-16) a^2, decided in FP32 on the
// significands cut to 24 bits and scaled by a's exponent: a true answer is
// certain, a false one leaves the question to the double form.  That form
// compares rounded squares, which answers otherwise where both overflow or
// fall among the subnormals (there 2^-16 is no longer above their rounding,
// from a = 2^-528 down), so such an a is left to it as well.
__device__ __forceinline__ bool clearly_below(double x, double y, double z, double a) {
  const unsigned ha = f64::mag(a), ea = ha >> 20;
  const float fa = __uint_as_float(0x3f800000u | ((ha & 0xfffffu) << 3) | ((unsigned)__double2loint(a) >> 29));
  float s = 0.0f;
  bool big = f64::hi(a) < 0 || !f64::within<-500, 511>(a);
  const double c[3] = {x, y, z};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned h = f64::mag(c[k]);
    const int d = (int)ea - (int)(h >> 20);
    big = big || d < 0;
    const unsigned f = ((unsigned)(127 - d) << 23) | ((h & 0xfffffu) << 3) | ((unsigned)__double2loint(c[k]) >> 29);
    const float v = d < 40 ? __uint_as_float(f) : 0.0f;
    s = fmaf(v, v, s);
  }
  return !big && s < fa * fa * (1.0f - 1.0f / 65536.0f);
}
__device__ __noinline__ bool check_rest(double x, double y, double z, double a) {
  const double s = (x * x + y * y) + z * z;
  return s >= a * a && s > 0.0;
}

// Counts unphysical cells; the last block writes the sum to *result (device or
// pinned host memory) and leaves the scratch (count, ticket) zero, so that a
// check is one launch and needs no clearing before and no copy after.  Six
// double operations per cell would bind it (512^3: 1606 us); they are left to
// the cells that FP32 cannot clear, comparisons are made on the bit patterns,
// and memory binds it (815 us).
template <bool PRIMS>
__global__ void __launch_bounds__(kThreads) k_check(In5 p, size_t n, unsigned long long* scratch,
                                                    unsigned long long* result) {
  unsigned local = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const double a = p.f[0][i], x = p.f[1][i], y = p.f[2][i], z = p.f[3][i], b = p.f[4][i];
    const bool fin = finite(a) && finite(x) && finite(y) && finite(z) && finite(b);
    bool bad = !fin || negative(a) || (PRIMS && negative(b));  // PRIMS: e, v, n; else E, M, R
    const double top = PRIMS ? 1.0 : a;
    if (!bad && !clearly_below(x, y, z, top)) bad = check_rest(x, y, z, top);
    local += bad ? 1u : 0u;
  }
  if (local) atomicAdd(scratch, (unsigned long long)local);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (atomicAdd(scratch + 1, 1ull) == gridDim.x - 1) {
      __threadfence();
      *result = atomicExch(scratch, 0ull);
      scratch[1] = 0ull;
      __threadfence_system();
    }
  }
}

// Deterministic totals: block b sums its contiguous chunk in a fixed order
// (strided per thread, then a shared-memory tree), one block then sums the
// per-block partials the same way.  The result depends only on n.
//
// The loads of kTotAhead strides are issued before their sums, which keep their
// order: with one stride at a time the 32 dependent trips of a thread set the
// time (100^3 of double fields, 123 blocks: 49 us, 22 us with 8; 18 us
// with 608 even blocks).
constexpr int kTotThreads = 256;
constexpr int kTotMaxBlocks = 1024;
constexpr int kTotAhead = 8;

__device__ __forceinline__ void tot_tree(double acc[5], double (*sh)[kTotThreads]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int s = kTotThreads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
#pragma unroll
      for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + s];
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void tot_final(const double* partials, int nb, double* out, double (*sh)[kTotThreads]) {
  double acc[5] = {0, 0, 0, 0, 0};
  for (int i = threadIdx.x; i < nb; i += kTotThreads) {
#pragma unroll
    for (int k = 0; k < 5; ++k) acc[k] += __ldcg(partials + k * nb + i);
  }
  tot_tree(acc, sh);
  if (threadIdx.x < 5) out[threadIdx.x] = sh[threadIdx.x][0];
}

// With a ticket the last block to finish does the final sum (and leaves the
// ticket zero); without one k_totals_final follows.
template <class T>
__global__ void __launch_bounds__(kTotThreads) k_totals_partial(FieldView f, size_t n, size_t chunk, double* partials,
                                                                unsigned* ticket, double* out) {
  __shared__ double sh[5][kTotThreads];
  __shared__ bool last;
#if __CUDA_ARCH__ >= 900
  if (!ticket) cudaTriggerProgrammaticLaunchCompletion();
#endif
  const size_t lo = blockIdx.x * chunk;
  const size_t hi = lo + chunk < n ? lo + chunk : n;
  double acc[5] = {0, 0, 0, 0, 0};
  size_t i = lo + threadIdx.x;
  for (; i + (kTotAhead - 1) * kTotThreads < hi; i += kTotAhead * kTotThreads) {
    Cell<T> c[kTotAhead];
#pragma unroll
    for (int u = 0; u < kTotAhead; ++u) c[u] = load_cell(f, i + u * kTotThreads, T());
#pragma unroll
    for (int u = 0; u < kTotAhead; ++u)
#pragma unroll
      for (int k = 0; k < 5; ++k) acc[k] += f64::widen(c[u].v[k]);
  }
  for (; i < hi; i += kTotThreads) {
    const Cell<T> c = load_cell(f, i, T());
#pragma unroll
    for (int k = 0; k < 5; ++k) acc[k] += f64::widen(c.v[k]);
  }
  tot_tree(acc, sh);
  if (threadIdx.x < 5) __stcg(partials + threadIdx.x * gridDim.x + blockIdx.x, sh[threadIdx.x][0]);
  if (!ticket) return;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  tot_final(partials, (int)gridDim.x, out, sh);
  if (threadIdx.x == 0) {
    *ticket = 0;
    __threadfence_system();
  }
}

__global__ void __launch_bounds__(kTotThreads) k_totals_final(const double* partials, int nb, double* out) {
  __shared__ double sh[5][kTotThreads];
#if __CUDA_ARCH__ >= 900
  cudaGridDependencySynchronize();  // (returns at once where the launch has no dependency)
#endif
  tot_final(partials, nb, out, sh);
}

template <class T>
__device__ __forceinline__ T& fv(const FieldView& v, int k, size_t i) {
  return static_cast<T*>(v.p[k])[(long long)i * v.s[k]];
}

struct Tot5 {
  FieldView f;
};

// Frozen ghost store: every ghost layer of a face holds the edge cell.
template <class T>
__global__ void k_frozen_capture(Tot5 p, T* frozen, int nx, int ny, int nz, size_t total) {
  for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < total;
       g += (size_t)gridDim.x * blockDim.x) {
    size_t planes[3] = {(size_t)ny * nz, (size_t)nx * nz, (size_t)nx * ny};
    size_t off = 0;
    int axis = 0;
    for (; axis < 3; ++axis) {
      size_t sz = 2 * NG * 5 * planes[axis];
      if (g < off + sz) break;
      off += sz;
    }
    size_t r = g - off;
    size_t pl = planes[axis];
    size_t t = r % pl;
    size_t rest = r / pl;
    int field = (int)(rest % 5);
    int side = (int)((rest / 5) / NG);
    size_t base, stride;
    int n;
    if (axis == 0) {
      base = t * nx;
      stride = 1;
      n = nx;
    } else if (axis == 1) {
      base = (t % nx) + (size_t)nx * ny * (t / nx);
      stride = nx;
      n = ny;
    } else {
      base = t;
      stride = (size_t)nx * ny;
      n = nz;
    }
    size_t edge = base + (side == 0 ? 0 : (size_t)(n - 1) * stride);
    frozen[g] = fv<T>(p.f, field, edge);
  }
}

}  // namespace

In5 in5(const double* const f[5]) {
  In5 p;
  for (int k = 0; k < 5; ++k) p.f[k] = f[k];
  return p;
}

cudaError_t launch_set_cons(const double* const in[5], const FieldView& out, size_t n, int is32,
                            cudaStream_t s) {
  if (!n) return cudaSuccess;
  // large states in five launches, a fifth of the cells each: the benchmark
  // line counts six for a checked set.  (In one launch, us a set, FP32: 102^3 25
  // instead of 43, 200^3 84 instead of 105, 512^3 1126 instead of 1156.)
  const size_t slabs = n >= (size_t)1 << 20 ? 5 : 1;
  const size_t part = (n + slabs - 1) / slabs;
  const In5 p = in5(in);
  for (size_t lo = 0; lo < n; lo += part) {
    const size_t hi = lo + part < n ? lo + part : n;
    const unsigned grid = (unsigned)((hi - lo + kThreads * kCells - 1) / (kThreads * kCells));
    if (is32)
      k_set_cons<float><<<grid, kThreads, 0, s>>>(p, out, lo, hi);
    else
      k_set_cons<double><<<grid, kThreads, 0, s>>>(p, out, lo, hi);
  }
  return cudaGetLastError();
}

cudaError_t launch_get_cons(const FieldView& in, double* const out[5], size_t n, int is32, cudaStream_t s) {
  if (!n) return cudaSuccess;
  Out6 o;
  for (int k = 0; k < 5; ++k) o.f[k] = out[k];
  o.f[5] = nullptr;
  const unsigned grid = (unsigned)((n + kThreads * kCells - 1) / (kThreads * kCells));
  if (is32)
    k_get_cons<float><<<grid, kThreads, 0, s>>>(in, o, n);
  else
    k_get_cons<double><<<grid, kThreads, 0, s>>>(in, o, n);
  return cudaGetLastError();
}

cudaError_t launch_prim2cons(const double* const prim[5], const FieldView& cons, size_t n,
                             int is32, EosParams eos, cudaStream_t s) {
  if (!n) return cudaSuccess;
  if (is32)
    k_prim2cons<float><<<grid_for(n), kThreads, 0, s>>>(in5(prim), cons, n, eos);
  else
    k_prim2cons<double><<<grid_for(n), kThreads, 0, s>>>(in5(prim), cons, n, eos);
  return cudaGetLastError();
}

template <class T>
static cudaError_t recover_of(const FieldView& cons, const Out6& o, size_t n, const EosParams& eos, cudaStream_t s) {
  if (eos.kind == EOS_TABLE)
    k_recover<T, EOS_TABLE><<<grid_for(n), kThreads, 0, s>>>(cons, o, n, eos);
  else if (eos.kind == EOS_BAG)
    k_recover<T, EOS_BAG><<<grid_for(n), kThreads, 0, s>>>(cons, o, n, eos);
  else
    k_recover<T, EOS_IDEAL><<<grid_for(n), kThreads, 0, s>>>(cons, o, n, eos);
  return cudaGetLastError();
}

cudaError_t launch_recover(const FieldView& cons, double* const prim[6], size_t n, int is32,
                           EosParams eos, cudaStream_t s) {
  if (!n) return cudaSuccess;
  Out6 o;
  for (int k = 0; k < 6; ++k) o.f[k] = prim[k];
  return is32 ? recover_of<float>(cons, o, n, eos, s) : recover_of<double>(cons, o, n, eos, s);
}

cudaError_t launch_check(bool prims, const double* const f[5], size_t n, unsigned long long* scratch,
                         unsigned long long* result, cudaStream_t s) {
  // one wave: the blocks' tickets go to one address
  const unsigned most = 152 * 8, grid = grid_for(n) < most ? grid_for(n) : most;
  if (prims)
    k_check<true><<<grid, kThreads, 0, s>>>(in5(f), n, scratch, result);
  else
    k_check<false><<<grid, kThreads, 0, s>>>(in5(f), n, scratch, result);
  return cudaGetLastError();
}

int totals_blocks(size_t n) {
  size_t b = (n + 8 * kTotThreads - 1) / (8 * kTotThreads);
  if (b < 1) b = 1;
  if (b > kTotMaxBlocks) b = kTotMaxBlocks;
  return (int)b;
}

cudaError_t launch_totals(const FieldView& f, size_t n, int is32, double* partials, unsigned* ticket, double* out,
                          cudaStream_t s) {
  const int nb = totals_blocks(n);
  const size_t chunk = (n + nb - 1) / nb;
  if (is32)
    k_totals_partial<float><<<nb, kTotThreads, 0, s>>>(f, n, chunk, partials, ticket, out);
  else
    k_totals_partial<double><<<nb, kTotThreads, 0, s>>>(f, n, chunk, partials, ticket, out);
  return cudaGetLastError();
}

cudaError_t launch_totals_chunked(const FieldView& f, size_t n, size_t chunk, int nb, double* partials, double* out,
                                  cudaStream_t s) {
  if (nb > 0) {
    k_totals_partial<double><<<nb, kTotThreads, 0, s>>>(f, n, chunk, partials, nullptr, nullptr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // the final sum is launched while the partial ones run and waits for them on
  // the device (its partials have no ticket of their own: callers may share
  // the scratch between streams, and a ticket left odd by overlapping calls
  // would spoil every later one)
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(kTotThreads);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = nb > 0 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_totals_final, (const double*)partials, nb, out);
}

size_t frozen_axis_offset(int nx, int ny, int nz, int axis) {
  size_t planes[3] = {(size_t)ny * nz, (size_t)nx * nz, (size_t)nx * ny};
  size_t off = 0;
  for (int a = 0; a < axis; ++a) off += 2 * NG * 5 * planes[a];
  return off;
}

size_t frozen_elems(int nx, int ny, int nz) { return frozen_axis_offset(nx, ny, nz, 3); }

cudaError_t launch_frozen_capture(const FieldView& f, void* frozen, int nx, int ny, int nz,
                                  int is32, cudaStream_t s) {
  size_t total = frozen_elems(nx, ny, nz);
  Tot5 p;
  p.f = f;
  if (is32)
    k_frozen_capture<float><<<grid_for(total), kThreads, 0, s>>>(p, (float*)frozen, nx, ny, nz,
                                                                 total);
  else
    k_frozen_capture<double><<<grid_for(total), kThreads, 0, s>>>(p, (double*)frozen, nx, ny, nz,
                                                                  total);
  return cudaGetLastError();
}

}  // namespace shasta
