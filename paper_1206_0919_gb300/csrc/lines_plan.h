// lines_plan.h -- lines per block of the FP64 line sweep (host code, no CUDA).
#pragma once

namespace shasta {

// Arrays of doubles a block holds per position: U, Delta and its second
// difference (5 each), eps, p and p v, Uhat, Delta-hat and the limited flux (5
// each; the transport factors share the fluxes' room).
constexpr int kLinesArrays = 33;
constexpr int kLinesMaxThreads = 512;
constexpr long long kLinesSmem = 227 * 1024;  // shared memory a block may take
constexpr long long kLinesSmemSM = 228 * 1024;  // an SM has, 1 KB of it per block reserved

// One axis: B lines per block (0: the streaming sweep), threads per block,
// bytes of shared memory.
struct LinesPlan {
  int B, threads, smem;
};

inline long long lines_smem(int n, int B) { return (long long)B * (n + 6) * kLinesArrays * 8; }

inline LinesPlan lines_plan_for(int n, int B) {
  // one item per thread and stage where 512 threads reach (a stage has up to
  // n + 3 per line), else even shares
  const long long items = (long long)B * (n + 3);
  const long long rounds = (items + kLinesMaxThreads - 1) / kLinesMaxThreads;
  const int th = (int)((items + rounds - 1) / rounds + 31) / 32 * 32;
  return LinesPlan{B, th, (int)lines_smem(n, B)};
}

// The sweep is bound by double warp-instructions, so by the warps its cells
// fill on the busiest SM: rounds of blocks x warps per block.  Few warps per
// block leave its stages to the barriers' and loads' latency, one or two
// blocks per SM leave the pipe idle at them; measured (64^3, 96 x 48 x 120,
// 143 x 129 x 151, 200^3, B = 1 .. 8) against three blocks of five warps: two
// blocks 0.97, one 0.93; four warps 0.955, three 0.94, two 0.92.  Longer lines,
// one block of 9 to 16 warps per SM, stay at about a third of the streaming
// kernel's time (us a sweep along x, ideal gas: 256 x 64 x 48 1331 -> 398, 512
// 2548 -> 911, 874 3654 -> 1429; 512^3, a step 339 -> 231 ms).
inline int lines_per_block(long long plane, int n, int sm_count) {
  int best = 0;
  double cost = 0.0;
  for (int B = 1; B <= 16; ++B) {
    const long long smem = lines_smem(n, B);
    if (smem > kLinesSmem) break;
    const LinesPlan t = lines_plan_for(n, B);
    long long resident = kLinesSmemSM / (smem + 1024);
    if (resident > 2048 / t.threads) resident = 2048 / t.threads;
    const long long warps = ((long long)B * n + 31) / 32;
    const double fb = resident >= 3 ? 1.0 : (resident == 2 ? 0.97 : 0.93);
    const double fw = warps >= 5 ? 1.0 : (warps == 4 ? 0.955 : (warps == 3 ? 0.94 : 0.92));
    const long long blocks = (plane + B - 1) / B;
    const double c = (double)((blocks + sm_count - 1) / sm_count * warps) / (fb * fw);
    if (best == 0 || c < cost) {
      best = B;
      cost = c;
    }
  }
  return best;
}

}  // namespace shasta
