// Fused joiner + softmax + Eq. 3-7 for TW_MODE_BF16.  The [rows, V] logits live
// only in tensor memory: a thread-block cluster of CL = V / NC CTAs (NC = 256, 128 or 64 columns each) owns a tile of 128
// rows, CTA c holding columns [NC c, NC c + NC) of it in TMEM (two accumulator buffers, so the contraction of
// the next row tile overlaps this tile's epilogue).
//
// Per row tile, in every CTA of the cluster:
//   contraction   TMA ring -> tcgen05.mma (as in gemm_bf16.cu), z = tanh(E + Pp) W_out^T
//   epilogue A    per row: running max / sum-exp over the CTA's columns, the blank logit
//   exchange      (max, sum-exp[, blank logit]) of every row to every CTA of the cluster through
//                 distributed shared memory, completion by remote mbarrier arrivals
//   scan          lse, blank log-probability, the occupancy recursion la over the S frames of a
//                 hypothesis (frames of a hypothesis are adjacent lanes of one warp): Eq. 3-5, 7
//   epilogue B    delta_nb(k) = sum_t exp(la[t] - lse[t] + z[t, k]) (Eq. 6) by a segmented warp
//                 reduction, written to device memory ([rows / S, V]: S times smaller than the logits);
//                 with, for some segment sizes, the maximum of every 16 or 32 columns; hyp_step_kernel picks the N best
// Row layout: a tile holds 4 * (32 / S) hypotheses; hypothesis j of warp quarter q sits in TMEM lanes
// 32 q + j S .. + S - 1 (one lane per frame); lanes past (32 / S) S are idle.
//
// No TMA multicast is used: every CTA fetches the A tile it shares with its cluster mates itself.
// Waits on mbarriers are bounded; the two cluster-wide hardware barriers (start, end) are reached by
// every thread of every CTA on every path.
#include <array>
#include <map>
#include <mutex>

#include "operand.cuh"
#include "sm100.cuh"

namespace tw {

namespace {

using namespace sm100;

constexpr int BM = 128, BK = 64;             // rows per tile, K per stage
constexpr int kMaxCL = 16;
constexpr int kColGroups = 4;                // epilogue warps per TMEM lane quarter, a quarter of the CTA's columns each
constexpr int kEpiWarps = 4 * kColGroups, kEpiThreads = 32 * kEpiWarps;
constexpr int kThreadsFused = 64 + kEpiThreads;
constexpr uint32_t kABytes = BM * BK * 2, kAQuarter = kABytes / 4;
// longer segments (S >= 5): the sum over a hypothesis's frames goes through a per-warp staging tile in shared
// memory, 16 columns at a time (row = TMEM lane, odd pitch: conflict-free row-per-lane writes)
constexpr int kStagePitch = 17;

// NC: columns of the vocabulary per CTA
template <int NC>
struct FusedSmem {
  static constexpr int kStages = NC == 256 ? 3 : (NC == 128 ? 4 : 6);
  static constexpr uint32_t kBBytes = NC * BK * 2;
  // offsets from the 1024-aligned base
  static constexpr size_t kA = 0;
  static constexpr size_t kB = kA + (size_t)kStages * kABytes;
  static constexpr size_t kXch = kB + (size_t)kStages * kBBytes;                  // float2 [2][kMaxCL][BM]
  static constexpr size_t kXchBlank = kXch + (size_t)2 * kMaxCL * BM * 8;         // float  [2][BM]
  static constexpr size_t kPart = kXchBlank + (size_t)2 * BM * 4;                 // float2 [kColGroups][BM]
  static constexpr size_t kZb = kPart + (size_t)kColGroups * BM * 8;                       // float  [BM]
  static constexpr size_t kBias = kZb + (size_t)BM * 4;                           // float  [NC]
  static constexpr size_t kBars = kBias + (size_t)NC * 4;                         // uint64 [2 kStages + 6], uint32, int
  static constexpr size_t kStage = kBars + (2 * kStages + 8) * 8;                 // float  [kEpiWarps][32][kStagePitch]
  static constexpr size_t kTotal = kStage + (size_t)kEpiWarps * 32 * kStagePitch * 4;
  static constexpr size_t kBytes = kTotal + 1024;
};

constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
__device__ __forceinline__ float ex2f(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float lg2f(float x) { float y; asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// log2(2^a + 2^b), branch-free; log 0 = -inf on either side or both
__device__ __forceinline__ float logaddexp2_fast(float a, float b) {
  const float mx = fmaxf(a, b), mn = fminf(a, b);
  const float d = (mn == -INFINITY) ? -INFINITY : mn - mx;    // (-inf) - (-inf) would be NaN
  return mx + lg2f(1.f + ex2f(d));
}

// sum over the S lanes [lane, lane + S) of x, valid in lanes whose window stays inside the warp
template <int S>
__device__ __forceinline__ float window_sum(float x) {
  float total = x;
#pragma unroll
  for (int d = 1; d < S; ++d) total += __shfl_down_sync(0xffffffffu, x, d);
  return total;
}

#include "joiner_tile.inc"
#include "fused_joiner_kernel.inc"

}  // namespace

#include "fused_joiner_host.inc"

}  // namespace tw
