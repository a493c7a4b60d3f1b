// sweep_tile.cuh -- FP32 / MIXED SHASTA sweep on tiles in shared memory, sm_103a.
//
// The same sweep as sweep_fast.cuh, bit for bit, with the parallelism turned
// round: there one lane streams along a line and the positions of a piece are
// a serial chain; here the 32 lanes of a warp share 1 or 2 lines, each lane
// holds C consecutive cells of a line in registers, and whatever a cell needs
// from beyond its lane's cells (velocity and pressure, Uhat, the limited flux)
// comes from the neighbouring lanes by shuffle.  A tile is T = 32 C / XL
// positions of XL lines (its own ones and HALO on each side, ghosts mapped on
// load), so a sweep is many short independent pieces instead of few long ones.
//
// What bounds it: the streaming sweep needs at least one range per resident
// warp of a length that hides its 13-position lead-in, about 100 positions;
// below that (200^3 holds 137) it is bound by the serial chain, about 0.45 us
// per position.  A tile's chain is C cells that are independent within each
// stage.  Measured, x / y / z sweep, streaming -> tile (us):
//   48^3   20.8 / 18.7 / 18.7 ->  6.4 /  6.4 /  6.4
//   64^3   28.9 / 26.8 / 26.8 ->  8.4 /  8.4 /  8.4
//   128^3  51.4 / 45.3 / 43.4 -> 28.9 / 33.0 / 33.0
//   131 x 97 x 110  45.3 / 37.1 / 41.2 -> 22.6 / 24.8 / 26.8
//   200^3  116 / 100 / 100 -> 90.3 / 103 / 111
// On large grids both are bound by instruction issue (66% / 57% of the slots
// at 200^3 along x / y here; 249 warp-instructions per 32 computed positions
// along x, 241 along y, 279 and 270 per 32 of the lines' own cells: a tile's
// halo wastes 11-25%); the y/z tiles lose their lead to the block barrier
// between tiles, so large y/z sweeps keep streaming.  A line much shorter than
// a tile wastes the rest of it; tile_plan.h holds the estimates that leave such
// lines to the streaming sweep.
//
//  * The half-step and the full-step pass are two trips through one loop
//    body (recovery, transport factors, the passes of the field pairs), which
//    keeps the unrolled code within the instruction cache (unrolled twice it
//    measured 60% of the time lost to fetch stalls more).
//  * The cells of a lane are recovered without branches, with the clamp and
//    the vacuum rule in warps that hold such a cell only.
//  * (E, Mx) and (My, Mz) go through packed f32x2 arithmetic: 241 instead of
//    278 instructions per 32 positions, 103 instead of 109 us (200^3, y).
//  * y/z: the four warps of a block copy a tile of 8 adjacent lines, so that
//    global accesses are whole 128-byte rows; x: each warp copies its own rows.
//    Two buffers: the next tile is copied while one is computed.
#pragma once

#include "chain.cuh"
#include "sweep_fast.cuh"

namespace shasta {
namespace tile {

using fast::cp_async16;
using fast::cp_async4;
using fast::cp_commit;
using fast::cp_wait;

constexpr int HALO = 2 * NG;  // positions a tile holds beyond its own, per side
constexpr int YL = 8;         // y/z: lines per block (a 128-byte row of quads per position)

// Geometry of a tile: C cells per lane, XL lines per warp, G = 32 / XL lanes
// along each line, T positions.
template <int AXIS, int C, int XL>
struct Lay {
  static constexpr bool XP = AXIS == 0;
  static constexpr int G = 32 / XL;
  static constexpr int T = G * C;
  static constexpr int WARPS = XP ? 4 : YL / XL;  // warps per block
  // y/z, one buffer per block: cell (lane group g, cell c, line l) in slot
  // g * GS + c * YL + l.  x, one buffer per warp: slot l * ROW + g * GS + c.
  // The group stride GS puts the eight lanes of a 128-bit access phase in
  // eight different 16-byte bank groups.
  static constexpr int GS = XP ? (C % 2 ? C : C + 1) : YL * C + XL;
  static constexpr int CS = XP ? 1 : YL;  // slots from cell to cell
  static constexpr int M0 = XP ? 3 : GS;  // slots before the first cell (cell -1 of group 0)
  static constexpr int ROWN = G * GS + 3;
  static constexpr int ROW = XL == 1 ? ROWN : ROWN + ((4 - ROWN % 8 + 8) % 8);
  static constexpr int SLOTS = M0 + (XP ? XL * ROW : G * GS + 2 * GS);
  static constexpr int FLOATS = ((SLOTS * 5 + 3) / 4) * 4;  // quads, then R
  // the reads of cells -1 .. C + 1 by the first and the last lane group stay inside
  static_assert(M0 - CS - (GS - C * CS) >= 0, "cell -1 of group 0");
  static_assert(M0 + (XP ? (XL - 1) * ROW : YL - 1) + (G - 1) * GS + (C + 1) * CS + (GS - C * CS) < SLOTS,
                "cell C + 1 of the last group");
  static constexpr int BUFS = XP ? WARPS : 1;
  static constexpr int SMEM = 2 * BUFS * FLOATS * 4;
  // slot of cell c (-1 .. C+1) relative to the lane's first cell
  __host__ __device__ static constexpr int rel(int c) {
    return c < 0 ? c * CS - (GS - C * CS) : (c >= C ? c * CS + (GS - C * CS) : c * CS);
  }
  __device__ static __forceinline__ int slot(int pos, int l) {
    const int g = pos / C, c = pos - g * C;
    return M0 + g * GS + c * CS + (XP ? l * ROW : l);
  }
};

// Launch geometry: ntile tiles of len positions per line (the last may be
// shorter), and the divisor P.nb as multiplier and shift (exact below 2^31).
struct TileArgs {
  int ntile, len;
  unsigned nb_mul, nb_shift;
};

inline void set_divisor(TileArgs& A, unsigned d) {
  unsigned s = 0;
  while ((1ull << s) < d) ++s;
  A.nb_mul = (unsigned)((((1ull << s) - d) << 32) / d + 1);
  A.nb_shift = s;
}

template <int XL>
__device__ __forceinline__ float from_left(float v) { return __shfl_up_sync(0xffffffffu, v, XL); }
template <int XL>
__device__ __forceinline__ float from_right(float v) { return __shfl_down_sync(0xffffffffu, v, XL); }

// One SHASTA pass of R (no source) over the C cells of a lane, u from cell -1
// to cell C + 1: Delta, Uhat, their differences and the limited flux as in
// fast::step1, every cell's operations in the same order.  The neighbouring
// lanes supply Uhat of cells -1, C, C + 1 and the flux of cell -1.
template <int C, int XL>
__device__ __forceinline__ void pass1(const float (&u)[C + 3], const float (&a)[C], const float (&nb)[C],
                                      const float (&cc)[C], float eta, float (&out)[C]) {
  float d[C + 2];  // Delta of cells -1 .. C
#pragma unroll
  for (int c = 0; c < C + 2; ++c) d[c] = u[c + 1] - u[c];
  float uh[C + 3];  // Uhat of cells -1 .. C + 1
#pragma unroll
  for (int c = 0; c < C; ++c) uh[c + 1] = fmaf(cc[c], u[c + 1], fmaf(a[c], d[c + 1], nb[c] * d[c]));
  uh[0] = from_left<XL>(uh[C]);
  uh[C + 1] = from_right<XL>(uh[1]);
  uh[C + 2] = from_right<XL>(uh[2]);
  float dd[C + 1];  // first differences of Delta, cells 0 .. C
#pragma unroll
  for (int c = 0; c < C + 1; ++c) dd[c] = d[c + 1] - d[c];
  float dh[C + 2];  // Delta-hat of cells -1 .. C
#pragma unroll
  for (int c = 0; c < C + 2; ++c) dh[c] = uh[c + 1] - uh[c];
  float A[C + 1];  // limited flux of cells -1 .. C - 1
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const float d2 = dd[c + 1] - dd[c];
    const float aph = eta * fmaf(-0.125f, d2, dh[c + 1]);
    A[c + 1] = fast::limit(aph, dh[c + 2], dh[c]);
  }
  A[0] = from_left<XL>(A[C]);
#pragma unroll
  for (int c = 0; c < C; ++c) out[c] = (uh[c + 1] + A[c]) - A[c + 1];
}

// Two fields of a cell as one packed pair: (E, Mx) and (My, Mz) arrive as
// aligned register pairs of the 128-bit loads, so one f32x2 instruction does
// both fields without moves.
typedef unsigned long long p2;
__device__ __forceinline__ p2 mk2(float x, float y) {
  p2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void un2(p2 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ p2 add2p(p2 a, p2 b) {
  p2 r;
  asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 sub2p(p2 a, p2 b) {
  p2 r;
  asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 mul2p(p2 a, p2 b) {
  p2 r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ p2 fma2p(p2 a, p2 b, p2 c) {
  p2 r;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <int XL>
__device__ __forceinline__ p2 left2(p2 v) {
  float x, y;
  un2(v, x, y);
  return mk2(from_left<XL>(x), from_left<XL>(y));
}
template <int XL>
__device__ __forceinline__ p2 right2(p2 v) {
  float x, y;
  un2(v, x, y);
  return mk2(from_right<XL>(x), from_right<XL>(y));
}

// The pass of a pair of fields (pass1 with a source src(c) where SRC).
template <int C, int XL, bool SRC, class Src>
__device__ __forceinline__ void pass2(const p2 (&u)[C + 3], const p2 (&a)[C], const p2 (&nb)[C], const p2 (&cc)[C],
                                      Src src, float eta, float (&o0)[C], float (&o1)[C]) {
  const p2 eta2 = mk2(eta, eta), m8 = mk2(-0.125f, -0.125f);
  p2 d[C + 2];
#pragma unroll
  for (int c = 0; c < C + 2; ++c) d[c] = sub2p(u[c + 1], u[c]);
  p2 uh[C + 3];
#pragma unroll
  for (int c = 0; c < C; ++c)
    uh[c + 1] = fma2p(cc[c], u[c + 1], fma2p(a[c], d[c + 1], SRC ? fma2p(nb[c], d[c], src(c)) : mul2p(nb[c], d[c])));
  uh[0] = left2<XL>(uh[C]);
  uh[C + 1] = right2<XL>(uh[1]);
  uh[C + 2] = right2<XL>(uh[2]);
  p2 dd[C + 1];
#pragma unroll
  for (int c = 0; c < C + 1; ++c) dd[c] = sub2p(d[c + 1], d[c]);
  p2 dh[C + 2];
#pragma unroll
  for (int c = 0; c < C + 2; ++c) dh[c] = sub2p(uh[c + 1], uh[c]);
  p2 A[C + 1];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const p2 d2 = sub2p(dd[c + 1], dd[c]);
    const p2 aph = mul2p(eta2, fma2p(m8, d2, dh[c + 1]));
    float p0, p1, q0, q1, r0, r1;
    un2(aph, p0, p1);
    un2(dh[c + 2], q0, q1);
    un2(dh[c], r0, r1);
    A[c + 1] = mk2(fast::limit(p0, q0, r0), fast::limit(p1, q1, r1));
  }
  A[0] = left2<XL>(A[C]);
#pragma unroll
  for (int c = 0; c < C; ++c) un2(sub2p(add2p(uh[c + 1], A[c]), A[c + 1]), o0[c], o1[c]);
}

// Transport coefficients of the C cells from w of cells -1 .. C.
template <int C, int XL>
__device__ __forceinline__ void coeffs(float tau, const float (&w)[C + 2], float (&a)[C], float (&nb)[C],
                                       float (&cc)[C]) {
  float qp[C + 1];  // cells -1 .. C-1
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const float num = fmaf(-tau, w[c + 1], 0.5f);
    const float den = fmaf(tau, w[c + 2] - w[c + 1], 1.0f);
    qp[c + 1] = num * __fdividef(1.0f, den);
  }
  qp[0] = from_left<XL>(qp[C]);
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const float qm = 1.0f - qp[c];
    a[c] = 0.5f * (qp[c + 1] * qp[c + 1]);
    nb[c] = -0.5f * (qm * qm);
    cc[c] = qp[c + 1] + qm;
  }
}

// rec32 (REC_F32, REC_DF) in two parts, so that the cells of a lane are
// recovered without branches: |M|^2 of all of them, then the roots, with the
// clamp and the vacuum rule as selections (CLAMP) only where a lane of the warp
// holds such a cell.  Evolved states hold many (hot spots, 200^3, step 120:
// 1.5% of the recoveries); recovering such a lane's cells again by rec32 took
// 106 us along x there, this 101; 92 before the first clamp.
template <int REC>
__device__ __forceinline__ float norm2(float mx, float my, float mz, float& lo) {
  lo = 0.0f;
  if constexpr (REC == fast::REC_DF) {
    const float a = mx * mx, a_l = fmaf(mx, mx, -a);
    const float b = my * my, b_l = fmaf(my, my, -b);
    const float c = mz * mz, c_l = fmaf(mz, mz, -c);
    const float s1 = a + b;
    float bb = s1 - a;
    const float r1 = (a - (s1 - bb)) + (b - bb);
    const float M2 = s1 + c;
    bb = M2 - s1;
    const float r2 = (s1 - (M2 - bb)) + (c - bb);
    lo = ((a_l + b_l) + c_l) + (r1 + r2);
    return M2;
  } else {
    return fmaf(mx, mx, fmaf(my, my, mz * mz));
  }
}
// The velocity w along the sweep and the pressure p; true if clamped or vacuum.
template <int EOS, int REC, bool CLAMP>
__device__ __forceinline__ bool root(float E, float M2, float M2lo, float m, float omd, float B, float ec, float& w,
                                     float& p) {
  const float E2 = E * E;
  float D = REC == fast::REC_DF ? fmaf(E, E, -M2) - M2lo : E2 - M2;
  bool cl = false;
  if (CLAMP) {
    const float lim = omd * E;
    const float L2 = lim * lim;
    cl = M2 > L2;
    m = cl ? m * (lim * rsqrtf(M2)) : m;
    D = cl ? E2 - L2 : D;
    M2 = cl ? L2 : M2;
  }
  D = fmaxf(D, 0.0f);
  float pp;
  if constexpr (EOS == EOS_BAG) {
    const float R0 = fmaf(3.0f, D, E2);
    const float te = E + ec;
    const bool bag = R0 > te * te;
    const float b = bag ? B : 0.0f;
    const float r = fmaf(-4.0f * b, fmaf(2.0f, E, -b), R0);
    const float s = sqrtf(fmaxf(r, 0.0f));
    const float b43 = (4.0f / 3.0f) * b;
    pp = fmaf(fmaf(-b43, E, D), __fdividef(1.0f, fmaf(-2.0f, b, E + s)), -b43);
    if (bag && !(E > ec && r >= 0.0f && fmaf(3.0f, pp, 4.0f * B) > ec)) pp = __fdividef(M2, E - ec) - E;
  } else {
    const float s = sqrtf(fmaf(3.0f, D, E2));
    pp = D * __fdividef(1.0f, E + s);
  }
  w = m * __fdividef(1.0f, E + pp);
  p = pp;
  if (CLAMP) {
    const bool vac = !(E > 0.0f);
    w = vac ? 0.0f : w;
    p = vac ? 0.0f : p;
    cl = cl || vac;
  }
  return cl;
}

template <int EOS, int AXIS, int REC, int C, int XL, int MINB>
__global__ void __launch_bounds__(Lay<AXIS, C, XL>::WARPS * 32, MINB)
    sweep_tile_kernel(SweepParams P, TileArgs A) {
  using L = Lay<AXIS, C, XL>;
  constexpr bool XP = AXIS == 0;
  constexpr int T = L::T, G = L::G, W = L::WARPS;
  extern __shared__ __align__(16) float smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int xl = lane % XL, g = lane / XL;
  const int n = P.n;
  const unsigned plane = (unsigned)P.plane;
  const int len = A.len;
  const unsigned stride = (unsigned)P.stride;
  // work units: x, XL lines of a warp; y/z, YL lines of a block
  constexpr unsigned UL = XP ? XL : YL;
  float* const buf0 = smem + (XP ? (size_t)warp * 2 * L::FLOATS : 0);
  const unsigned nunit = (plane + UL - 1) / UL;
  const int ntile = A.ntile;
  const unsigned step = XP ? gridDim.x * W : gridDim.x;
  // this warp's (block's) tile: unit k at segment seg of the line
  int seg = 0;
  unsigned k = XP ? blockIdx.x * W + warp : blockIdx.x;
  auto wrap = [&](int& sg, unsigned& kk) {
    while (kk >= nunit && sg < ntile) {
      kk -= nunit;
      ++sg;
    }
  };
  wrap(seg, k);
  unsigned nclamp = 0;
  const int bc = P.bc;

  // first cell of line t
  auto line_base = [&](unsigned t) -> unsigned {
    if (AXIS == 0) return t * (unsigned)P.sb;
    if (AXIS == 2) return t;
    const unsigned c = (__umulhi(t, A.nb_mul) + t) >> A.nb_shift;  // t / nb
    return t + c * ((unsigned)P.sc - (unsigned)P.nb);
  };
  // one cell from the state into slot s of a buffer (quads at b, R at r)
  auto copy = [&](float* b, float* r, int s, unsigned i) {
    if (!SH_OK(P, i < (unsigned long long)P.ncap, 1, i) || !SH_OK(P, s >= 0 && s < L::SLOTS, 4, s)) return;
    cp_async16(b + 4 * s, P.qin + 4 * (size_t)i);
    cp_async4(r + s, P.rin + i);
  };
  auto store = [&](unsigned i, const float4& q, float R) {
    if (!SH_OK(P, i < (unsigned long long)P.ncap, 3, i)) return;
    *reinterpret_cast<float4*>(P.qout + 4 * (size_t)i) = q;
    P.rout[i] = R;
  };
  auto sync = [&] {
    if (XP)
      __syncwarp();
    else
      __syncthreads();
  };
  // copies the tile of unit k, segment seg into buffer b
  auto issue = [&](int seg, unsigned k, float* b) {
    const int p0 = seg * len - HALO;                // position of the tile's first cell
    const int pe = min(seg * len + len, n) + HALO;  // one past the last position needed
    float* r = b + L::SLOTS * 4;
    const bool edge = p0 < 0 || pe > n;
    const bool rare = edge && (bc == BC_FROZEN || n < HALO);
    auto mapped = [&](int q) {
      q = min(q, pe - 1);
      if (edge) {
        if (bc == BC_REFLECT) {
          q = max(q, -1 - q);
          q = min(q, 2 * n - 1 - q);
        } else {
          q += q < 0 ? n : 0;
          q -= q >= n ? n : 0;
        }
      }
      return q;
    };
    if (rare) {
      const fast::GeoP Gp{P};
#pragma unroll 1
      for (int e = XP ? lane : threadIdx.x; e < T * (int)UL; e += XP ? 32 : W * 32) {
        const int pos = XP ? e % T : e / (int)UL, x = XP ? e / T : e % (int)UL;
        unsigned t = k * UL + x;
        t = t < plane ? t : plane - 1;
        const int s = L::slot(pos, x);
        fast::copy_cell(P, Gp, b + 4 * s, r + s, line_base(t), stride, t, min(p0 + pos, pe - 1), n);
      }
    } else if (XP) {
#pragma unroll
      for (int x = 0; x < XL; ++x) {
        unsigned t = k * XL + x;
        t = t < plane ? t : plane - 1;
        const unsigned rb = line_base(t);
#pragma unroll
        for (int j = 0; j < (T + 31) / 32; ++j) {
          const int pos = j * 32 + lane;
          if (T % 32 == 0 || pos < T) {
            copy(b, r, L::slot(pos, x), rb + (unsigned)mapped(p0 + pos));
          }
        }
      }
    } else {
      const int l = threadIdx.x % YL, gg = threadIdx.x / YL;  // 32 W / YL = G lane groups
      unsigned t = k * YL + l;
      t = t < plane ? t : plane - 1;
      const unsigned rb = line_base(t);
      const int sl = L::M0 + gg * L::GS + l;
      const int q0 = p0 + gg * C;
      if (q0 >= 0 && q0 + C <= min(n, pe)) {
        unsigned i = rb + (unsigned)q0 * stride;
#pragma unroll
        for (int c = 0; c < C; ++c, i += stride) copy(b, r, sl + YL * c, i);
      } else {
        // ghosts, or past the tile's end
#pragma unroll 1
        for (int c = 0; c < C; ++c) copy(b, r, sl + YL * c, rb + (unsigned)mapped(q0 + c) * stride);
      }
    }
  };

  chain_begin();
  if (seg < ntile) issue(seg, k, buf0);
  cp_commit();
  int cur = 0;
  const float eta = P.f_eta;
#pragma unroll 1
  for (; seg < ntile; cur ^= 1) {
    float* const b = buf0 + cur * L::FLOATS;
    int segn = seg;
    unsigned kn = k + step;
    wrap(segn, kn);
    cp_wait<0>();
    sync();  // the tile is in place, and every lane is done with the other buffer
    if (segn < ntile) issue(segn, kn, buf0 + (cur ^ 1) * L::FLOATS);
    cp_commit();
    const int s0 = seg * len, s1 = min(s0 + len, n);
    const int p0 = s0 - HALO;
    const bool edge = p0 < 0 || s1 + HALO > n;
    if (edge && bc == BC_REFLECT) {
      // mirror images have the momentum along the line negated
      const int nlo = max(-p0, 0), nhi = max(s1 + HALO - n, 0);
#pragma unroll 1
      for (int e = XP ? lane : threadIdx.x; e < (nlo + nhi) * (int)UL; e += XP ? 32 : W * 32) {
        const int o = e / (int)UL, x = e % (int)UL;
        const int pos = o < nlo ? o : n - p0 + (o - nlo);
        if (fast::flips(p0 + pos, n, BC_REFLECT)) {
          const int s = L::slot(pos, x);
          if (!SH_OK(P, s >= 0 && s < L::SLOTS, 4, s)) continue;
          float* m = b + 4 * s + 1 + AXIS;
          *m = -*m;
        }
      }
      sync();
    }
    const unsigned tl = k * UL + (XP ? 0 : warp * XL) + xl;
    const bool valid = tl < plane;
    const int pos0 = p0 + g * C;  // position of this lane's first cell
    const int sb = L::M0 + g * L::GS + (XP ? xl * L::ROW : warp * XL + xl);
    const float4* const q4 = reinterpret_cast<const float4*>(b) + sb;
    const float* const r1 = b + L::SLOTS * 4 + sb;
    float H[4][C];  // the state recovered next: U^n, then U^(n+1/2)
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float4 v = q4[L::rel(c)];
      H[0][c] = v.x;
      H[1][c] = v.y;
      H[2][c] = v.z;
      H[3][c] = v.w;
    }
    float a[C], nb[C], cc[C];
    float tau = P.f_tau_h, ht = P.f_htau_h;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      float w[C + 2], p[C + 2];
      if constexpr (EOS == EOS_TABLE) {
        float wc[C], pc[C];
        bool cl[C];
        fast::rec32_table<C>(H[0], H[1], H[2], H[3], H[1 + AXIS], P.f_omd, P.tab, wc, pc, cl);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          w[c + 1] = wc[c];
          p[c + 1] = pc[c];
          if (cl[c] && h == 0) nclamp += valid && (unsigned)(pos0 + c - s0) < (unsigned)(s1 - s0) ? 1u : 0u;
        }
      } else if constexpr (REC == fast::REC_F64) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const unsigned cl = fast::rec32<EOS, REC>(H[0][c], H[1][c], H[2][c], H[3][c], H[1 + AXIS][c], P.f_omd,
                                                    P.omd, P.f_bag_B, P.f_bag_ec, P.tab, w[c + 1], p[c + 1]);
          if (cl && h == 0) nclamp += valid && (unsigned)(pos0 + c - s0) < (unsigned)(s1 - s0) ? 1u : 0u;
        }
      } else {
        float M2[C], Ml[C];
        bool okl = true, okm = true, okr = true;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          M2[c] = norm2<REC>(H[1][c], H[2][c], H[3][c], Ml[c]);
          const float lim = P.f_omd * H[0][c];
          bool& ok = c < NG ? okl : (c >= C - NG ? okr : okm);
          ok = ok & (M2[c] <= lim * lim) & (H[0][c] > 0.0f);
        }
        // the half-step values of the tile's outer three cells per side are not used
        const bool rare = !okm || (!okl && (h == 0 || g > 0)) || (!okr && (h == 0 || g < G - 1));
        if (!__any_sync(0xffffffffu, rare)) {
#pragma unroll
          for (int c = 0; c < C; ++c)
            root<EOS, REC, false>(H[0][c], M2[c], Ml[c], H[1 + AXIS][c], P.f_omd, P.f_bag_B, P.f_bag_ec, w[c + 1],
                                  p[c + 1]);
        } else {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const bool cl = root<EOS, REC, true>(H[0][c], M2[c], Ml[c], H[1 + AXIS][c], P.f_omd, P.f_bag_B,
                                                 P.f_bag_ec, w[c + 1], p[c + 1]);
            if (cl && h == 0) nclamp += valid && (unsigned)(pos0 + c - s0) < (unsigned)(s1 - s0) ? 1u : 0u;
          }
        }
      }
      w[0] = from_left<XL>(w[C]);
      w[C + 1] = from_right<XL>(w[1]);
      p[0] = from_left<XL>(p[C]);
      p[C + 1] = from_right<XL>(p[1]);
      coeffs<C, XL>(tau, w, a, nb, cc);
      float pw[C + 2];
#pragma unroll
      for (int c = 0; c < C + 2; ++c) pw[c] = p[c] * w[c];
      auto sp = [&](int c) { return ht * (p[c] - p[c + 2]); };
      auto se = [&](int c) { return ht * (pw[c] - pw[c + 2]); };
      auto srcA = [&](int c) { return AXIS == 0 ? mk2(se(c), sp(c)) : mk2(se(c), 0.0f); };
      auto srcB = [&](int c) { return AXIS == 1 ? mk2(sp(c), 0.0f) : mk2(0.0f, sp(c)); };
      p2 a2[C], nb2[C], cc2[C], u[C + 3];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        a2[c] = mk2(a[c], a[c]);
        nb2[c] = mk2(nb[c], nb[c]);
        cc2[c] = mk2(cc[c], cc[c]);
      }
#pragma unroll
      for (int c = 0; c < C + 3; ++c) {
        const float4 q = q4[L::rel(c - 1)];
        u[c] = mk2(q.x, q.y);
      }
      pass2<C, XL, true>(u, a2, nb2, cc2, srcA, eta, H[0], H[1]);
#pragma unroll
      for (int c = 0; c < C + 3; ++c) {
        const float4 q = q4[L::rel(c - 1)];
        u[c] = mk2(q.z, q.w);
      }
      pass2<C, XL, AXIS != 0>(u, a2, nb2, cc2, srcB, eta, H[2], H[3]);
      if (h == 0 && edge && bc == BC_FROZEN) {
#pragma unroll
        for (int c = 0; c < C; ++c)
          if (pos0 + c < 0 || pos0 + c >= n) {
            const float4 z = q4[L::rel(c)];
            H[0][c] = z.x;
            H[1][c] = z.y;
            H[2][c] = z.z;
            H[3][c] = z.w;
          }
      }
      tau = P.f_tau_f;
      ht = P.f_htau_f;
    }
    float R[C];
    {
      float v[C + 3];
#pragma unroll
      for (int c = 0; c < C + 3; ++c) v[c] = r1[L::rel(c - 1)];
      pass1<C, XL>(v, a, nb, cc, eta, R);
    }
    if (XP) {
      // through the tile's own buffer, so that rows are written whole
      __syncwarp();
      float4* o4 = const_cast<float4*>(q4);
      float* o1 = const_cast<float*>(r1);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        o4[L::rel(c)] = make_float4(H[0][c], H[1][c], H[2][c], H[3][c]);
        o1[L::rel(c)] = R[c];
      }
      __syncwarp();
#pragma unroll
      for (int x = 0; x < XL; ++x) {
        const unsigned t = k * XL + x;
        if (t < plane) {
          const unsigned rb = line_base(t) + (unsigned)s0;
#pragma unroll
          for (int j = 0; j < (T - 2 * HALO + 31) / 32; ++j) {
            const int o = j * 32 + lane;
            if (o < s1 - s0) {
              const int s = L::slot(o + HALO, x);
              if (!SH_OK(P, s >= 0 && s < L::SLOTS, 4, s)) continue;
              store(rb + o, reinterpret_cast<float4*>(b)[s], (b + L::SLOTS * 4)[s]);
            }
          }
        }
      }
    } else if (valid) {
      const unsigned lo = (unsigned)max(0, s0 - pos0), hi = (unsigned)max(0, min(C, s1 - pos0));
      const unsigned own = ((1u << hi) - 1u) & ~((1u << min(lo, 31u)) - 1u);
      unsigned i = line_base(tl) + (unsigned)pos0 * stride;
#pragma unroll
      for (int c = 0; c < C; ++c, i += stride) {
        if (own & (1u << c)) store(i, make_float4(H[0][c], H[1][c], H[2][c], H[3][c]), R[c]);
      }
    }
    seg = segn;
    k = kn;
  }
  cp_wait<0>();
  add_clamps(P.clamp_count, nclamp);
}

}  // namespace tile
}  // namespace shasta
