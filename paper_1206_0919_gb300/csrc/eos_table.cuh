// eos_table.cuh -- tabulated equation of state: lookups and recovery.
#pragma once

#include <cuda_runtime.h>

namespace shasta {

// Tabulated EoS (EOS_TABLE): p at e = k de, k = 0 .. n-1, linear in
// between, the last interval continued above the table (device copies in
// double, and in float as the pairs p_k, p_{k+1} - p_k).
struct EosTable {
  const double* p64;
  const float2* p32;
  int n;
  double de;
  float inv_de32;  // 1 / de in float (FP32 lookups)
};

// p(e) of a tabulated EoS in float: linear between the nodes k de, the
// last interval continued above the table (the index stays inside the table
// for any e, NaN included); *slope receives dp/de of the interval.
__device__ __forceinline__ float tab32(const EosTable& T, float e, float* slope = nullptr) {
  const float x = e * T.inv_de32;
  int k = (int)x;
  k = k < 0 ? 0 : (k > T.n - 2 ? T.n - 2 : k);
  const float f = x - (float)k;
  const float2 a = __ldg(T.p32 + k);
  if (slope) *slope = a.y * T.inv_de32;
  return fmaf(f, a.y, a.x);
}

// Tabulated EoS: p from E and |M|^2 of N cells.  The root is the fixed point
// of Sec. 3, |v| = |M| / (E + p(E - |M| |v|)), started as there from
// |M| / (E + p(E)).  In float the root is found by Newton steps on
// g(v) = v - |M| / (E + p), g'(v) = 1 - |M|^2 p'(e) / (E + p)^2
// >= 1 - v^2 p' > 0 (exact within one interval of the piecewise-linear
// table), until the change is at most 1e-7 (12 steps at most), then
// p = p(E - |M| |v|).
// A step is one chain of a lookup and two reciprocals, and the 4 warps a
// scheduler holds leave it half idle at them.  So a lane takes kTogether cells
// through their steps side by side, a finished one keeping its root: 96^3, 24
// steps, 2930 us one by one, 2666 by two, 2606 by three, 2655 by four or all
// seven (the group runs as long as its slowest cell).  The streaming sweeps
// take their two cells together: 200^3, 830 -> 531 us a step with the tiled x.
constexpr int kTogether = 3;
template <int N>
__device__ __forceinline__ void table_p32(const EosTable& T, const float (&E)[N], const float (&M2)[N],
                                          float (&p)[N]) {
  constexpr int K = N < kTogether ? N : kTogether;
  float M[N], v[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    M[i] = sqrtf(M2[i]);
    v[i] = M[i] * __fdividef(1.0f, E[i] + tab32(T, E[i]));
  }
#pragma unroll
  for (int i0 = 0; i0 < N; i0 += K) {
    bool done[K];
#pragma unroll
    for (int k = 0; k < K; ++k) done[k] = false;
#pragma unroll 1
    for (int it = 0; it < 12; ++it) {
      bool all = true;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int i = i0 + k;
        if (i >= N) continue;
        float dp;
        const float pe = tab32(T, fmaf(-M[i], v[i], E[i]), &dp);
        const float r = __fdividef(1.0f, E[i] + pe);
        const float g = fmaf(-M[i], r, v[i]);         // v - M / (E + p)
        const float mr = M[i] * r;
        const float gp = fmaf(-mr * mr, dp, 1.0f);    // 1 - M^2 p' / (E + p)^2
        const float d = __fdividef(g, gp);
        v[i] = done[k] ? v[i] : v[i] - d;
        done[k] = done[k] || fabsf(d) <= 1e-7f;
        all = all && done[k];
      }
      if (all) break;
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) p[i] = tab32(T, fmaf(-M[i], v[i], E[i]));
}

}  // namespace shasta
