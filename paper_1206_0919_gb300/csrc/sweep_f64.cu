// sweep_f64.cu -- FP64 instances of the fused sweep: whole lines in shared
// memory (sweep_lines64.cuh), or one thread per line segment (sweep.cuh).
// Built with -fmad=false and IEEE division / square root so that the
// arithmetic is the plain double-precision evaluation of each expression in
// source order.
#include "kernels.h"
#include "chain.cuh"
#include "sweep_lines64.cuh"

#include <math.h>

namespace shasta {

template <int EOS, int AXIS>
static cudaError_t go(const SweepParams& P, cudaStream_t s) {
  const int threads = 128;
  const int L = P.range_len > 0 && P.range_len < P.n ? (int)P.range_len : P.n;
  const long long work = P.plane * ((P.n + L - 1) / L);
  long long blocks = (work + threads - 1) / threads;
  sweep_kernel<double, double, EOS, AXIS, false><<<(unsigned)blocks, threads, 0, s>>>(P);
  return cudaGetLastError();
}

template <int EOS>
static const void* lines_kernel(int axis) {
  return axis == 0   ? (const void*)lines64::sweep_lines_kernel<EOS, 0>
         : axis == 1 ? (const void*)lines64::sweep_lines_kernel<EOS, 1>
                     : (const void*)lines64::sweep_lines_kernel<EOS, 2>;
}

static const void* lines_kernel_of(int eos, int axis) {
  return eos == EOS_IDEAL ? lines_kernel<EOS_IDEAL>(axis)
                          : (eos == EOS_BAG ? lines_kernel<EOS_BAG>(axis) : lines_kernel<EOS_TABLE>(axis));
}

cudaError_t prepare_lines_f64(int axis, int eos, const LinesPlan& t) {
  return cudaFuncSetAttribute(lines_kernel_of(eos, axis), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kLinesSmem);
}

cudaError_t launch_lines_f64(const SweepParams& P, const LinesPlan& t, int axis, int eos, bool chain,
                             cudaStream_t s) {
  if (P.plane <= 0) return cudaSuccess;
  if (t.B < 1 || P.n < NG) return cudaErrorInvalidValue;
  const int np = P.n + 2 * NG;
  lines64::LineArgs A;
  A.B = t.B;
  A.js = axis == 0 ? 1 : t.B;
  A.ls = axis == 0 ? np : 1;
  A.sz = t.B * np;
  A.eta_exp = 0;
  int ex;
  if (frexp(P.eta, &ex) == 0.5 && ex <= 0 && ex > -60) A.eta_exp = 1 - ex;
  void* args[] = {const_cast<SweepParams*>(&P), &A};
  return launch_sweep_kernel(lines_kernel_of(eos, axis), dim3((unsigned)((P.plane + t.B - 1) / t.B)),
                          dim3(t.threads), args, t.smem, chain, s);
}

cudaError_t launch_sweep_f64(const SweepParams& P, int axis, int eos, cudaStream_t s) {
  if (P.plane <= 0) return cudaSuccess;
  switch (eos * 3 + axis) {
    case 0: return go<EOS_IDEAL, 0>(P, s);
    case 1: return go<EOS_IDEAL, 1>(P, s);
    case 2: return go<EOS_IDEAL, 2>(P, s);
    case 3: return go<EOS_BAG, 0>(P, s);
    case 4: return go<EOS_BAG, 1>(P, s);
    case 5: return go<EOS_BAG, 2>(P, s);
    case 6: return go<EOS_TABLE, 0>(P, s);
    case 7: return go<EOS_TABLE, 1>(P, s);
    case 8: return go<EOS_TABLE, 2>(P, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace shasta
