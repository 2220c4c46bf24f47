// The predictor's output projection and the joiner's operand in one kernel, for a decode step with an LSTM predictor and
// segments below 8 frames:  Pp = W_p h of every new hypothesis (tcgen05, bf16, fp32 accumulation), and from the accumulators
// the operand rows act(E[t] + Pp) of the segment's frames, straight into the fused joiner kernel's tile layout.
// What this saves is a kernel in the step's chain of dependent ones (the operand kernel: 4 us on a small step, 7 us with
// 128 utterances at J = 1024, plus 2 to 4 us until it starts) and the round trip of Pp through L2.  Every frame is read
// once per hypothesis: with longer segments that is L2-bound, and the per-utterance operand kernel stays.
// The rows of hypotheses carried over a segment turn-over, which have no new Pp, are written by carry_rows (hyp.cu).  A live
// hypothesis's rows of padding frames are written as zeros: the joiner multiplies their exponentials by 0, and an older pass
// may have left a NaN there (an utterance with such frames must not reach its neighbours' sums).
#include "operand.cuh"
#include "sm100.cuh"

namespace tw {

namespace {

using namespace sm100;

constexpr int BM = 128, BK = 64, kCols = 16;       // kCols: accumulator columns a thread of the epilogue takes
// frames of a segment that it fetches ahead of the accumulators; with two, S = 3 paid a round trip to L2 behind them (128 utterances
// at V = 4096 75.9 -> 75.2 ms, 32 at V = 1024 9.94 -> 9.82 ms; 92 and 96 registers a thread, four frames would leave no second CTA)
constexpr int kEarlyFrames = 3;

template <int BN>
struct WpCfg {
  // the ring: stages of 128 rows; BN = 32: half an SM, to be resident beside a gate GEMM's CTA
  static constexpr int kFullStages = BN == 64 ? 8 : 5;
  static constexpr int kEpiWarps = 4 * (BN / kCols), kThreads = 64 + 32 * kEpiWarps;
  static constexpr uint32_t kABytes = BM * BK * 2, kBBytes = BN * BK * 2;
  static constexpr uint32_t kRing = kFullStages * (kABytes + kBBytes);
  static constexpr size_t kSmem = (size_t)kRing + 1024 + 256;
};

template <int BN>
__global__ void __launch_bounds__(WpCfg<BN>::kThreads, BN == 64 ? 1 : 2)
wp_operand_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmA32, const __grid_constant__ CUtensorMap tmB,
                  WpOperandParams p) {
  using C = WpCfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // (A and B apart: an MMA that reads 128 rows of a smaller stage stays inside the ring)
  const uint32_t a_stage = (uint32_t)ring_quarters(p.M) * (C::kABytes / 4);
  const int nst = min((int)(C::kRing / (a_stage + C::kBBytes)), kMaxRingStages);
  uint8_t* sA = smem;
  uint8_t* sB = smem + nst * a_stage;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kRing);
  uint64_t* empty = full + kMaxRingStages;
  uint64_t* acc_full = empty + kMaxRingStages; // [2]
  uint64_t* acc_empty = acc_full + 2;          // [2]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(acc_empty + 2);

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int num_kb = (p.K + BK - 1) / BK;
  // The work list is hyp_step_kernel's, which had finished before the last gate GEMM (the kernel ahead) began: the list and
  // the utterances' positions are read ahead of the wait.
  const int M = warp_uniform(__ldcg(p.M_dev));
  // the joiner kernel that follows streams W_out, which a large step's other traffic has pushed out of L2: every CTA asks for
  // its share (a constant weight: nothing to wait for)
  if (p.pf_base != nullptr && threadIdx.x == 64) {
    const long long per = ((p.pf_bytes + gridDim.x - 1) / gridDim.x + 127) & ~127ll, off = per * blockIdx.x;
    if (off < p.pf_bytes) prefetch_l2_bulk(p.pf_base + off, (uint32_t)((off + per <= p.pf_bytes ? per : p.pf_bytes - off) & ~15ll));
  }
  if (threadIdx.x == 0) {
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmA32);
    prefetch_tensormap(&tmB);
    for (int s = 0; s < nst; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], C::kEpiWarps); }
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) { tmem_alloc(tmem_holder, 2 * BN); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  const int m_tiles = (M + BM - 1) / BM, n_tiles = (p.N + BN - 1) / BN;
  const int num_tiles = m_tiles * n_tiles;     // a CTA past the last tile runs no loop iteration below
  bool ok = true;                              // every wait of this thread so far has ended in time

  if (warp == 0) {
    int npre = 0;                              // W_p is a constant: the first tile's first stages ahead of the wait
    const uint64_t keep = l2_policy_evict_last();
    const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB), full0 = smem_u32(full), empty0 = smem_u32(empty);
    if ((int)blockIdx.x < num_tiles) {
      npre = num_kb < nst ? num_kb : nst;
      for (int kb = 0; kb < npre; ++kb) {
        if (elect_one()) {
          mbar_expect_only_a(full0 + 8 * kb, C::kBBytes);         // the arrival comes with A
          tma_load_2d_hint_a(b0 + kb * C::kBBytes, &tmB, full0 + 8 * kb, kb * BK, ((int)blockIdx.x % n_tiles) * BN, keep);
        }
      }
    }
    pdl_wait();
    pdl_trigger();
    {
      int s = 0;
      uint32_t ph = 0;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        const int m0 = (tile / n_tiles) * BM, n0 = (tile % n_tiles) * BN;
        const int nq = M - m0 <= 64 ? (M - m0 + 31) >> 5 : 4;          // lane quarters with rows in them, three as four
        const uint32_t a_bytes = (uint32_t)nq * (C::kABytes / 4);
        for (int kb = 0; kb < num_kb; ++kb) {
          const bool first = npre > 0;                       // B is on its way
          if (!first) {
            ok = mbar_wait_warp(empty0 + 8 * s, ph ^ 1, p.err);
            if (!ok) break;
          } else {
            --npre;
          }
          if (elect_one()) {
            const uint32_t adst = a0 + s * a_stage;
            mbar_arrive_expect_a(full0 + 8 * s, first ? a_bytes : a_bytes + C::kBBytes);
            if (nq == 4) tma_load_2d_a(adst, &tmA, full0 + 8 * s, kb * BK, m0);
            else for (int q = 0; q < nq; ++q) tma_load_2d_a(adst + q * (C::kABytes / 4), &tmA32, full0 + 8 * s, kb * BK, m0 + 32 * q);
            if (!first) tma_load_2d_hint_a(b0 + s * C::kBBytes, &tmB, full0 + 8 * s, kb * BK, n0, keep);
          }
          if (++s == nst) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    pdl_wait();
    pdl_trigger();
    {
      constexpr uint32_t idesc = make_idesc_bf16(BM, BN);
      int s = 0;
      uint32_t ph = 0, lt = 0;
      const uint32_t a_lo = desc_lo(smem_u32(sA)), b_lo = desc_lo(smem_u32(sB)), full0 = smem_u32(full), empty0 = smem_u32(empty);
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++lt) {
        const uint32_t buf = lt & 1, aph = (lt >> 1) & 1;
        ok = mbar_wait_warp(smem_u32(acc_empty) + 8 * buf, aph ^ 1, p.err);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + buf * BN;
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = mbar_wait_warp(full0 + 8 * s, ph, p.err);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t al = a_lo + s * (a_stage >> 4), bl = b_lo + s * (C::kBBytes >> 4);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) umma_bf16(tmem_d, desc_of(al + 2 * k), desc_of(bl + 2 * k), idesc, (kb | k) != 0);
            umma_commit_a(empty0 + 8 * s);
          }
          if (++s == nst) { s = 0; ph ^= 1; }
        }
        if (ok && elect_one()) umma_commit_a(smem_u32(acc_full) + 8 * buf);
      }
    }
  } else {
    const int q = warp & 3, grp = (warp - 2) >> 2;           // TMEM lane quarter, group of kCols columns
    uint32_t lt = 0;
    bool waited = false;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++lt) {
      const int m = (tile / n_tiles) * BM + q * 32 + lane, n = (tile % n_tiles) * BN + grp * kCols;
      const uint32_t buf = lt & 1, aph = (lt >> 1) & 1;
      const bool live = m < M && n < p.N, two = n + 8 < p.N;                   // N is a multiple of 8
      // list entry m: its slot, and the utterance and list position behind the slot
      int sl = 0;
      const float* e = nullptr;
      float* pp = nullptr;
      __nv_bfloat16* dst = nullptr;
      float ev[kEarlyFrames][kCols];                          // the first frames, fetched under the contraction
      if (live) {
        const int bi = p.pw_bi[m], b = bi / kMaxBeam, i = bi - b * kMaxBeam;
        pp = p.Pp + (long long)p.pw_new[m] * p.N + n;
        sl = p.slen[b];
        e = p.E + ((long long)b * p.T + p.t0[b]) * p.N + n;
        dst = p.A + operand_row(p.row_off[b] + i, 0, p.S) * p.N + n;
#pragma unroll
        for (int t = 0; t < kEarlyFrames; ++t) {
          if (t < sl) {
            ld_global_v8(e + (long long)t * p.N, ev[t]);
            if (two) ld_global_v8(e + (long long)t * p.N + 8, ev[t] + 8);
          }
        }
      }
      if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }
      ok = mbar_wait(&acc_full[buf], aph, p.err);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      uint32_t raw[kCols];
      tmem_ld16_issue(tmem_base + ((uint32_t)(q * 32) << 16) + buf * BN + (uint32_t)(grp * kCols), raw);
      tmem_ld_wait16(raw);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
      if (!live) continue;
      float v[kCols];
#pragma unroll
      for (int u = 0; u < kCols; ++u) v[u] = __uint_as_float(raw[u]);
      st_global_v8(pp, v);                                    // read again when the hypothesis is carried into the next segment
      if (two) st_global_v8(pp + 8, v + 8);
      auto frame = [&](int t, const float* x) {
        *reinterpret_cast<uint4*>(dst + (long long)t * p.N) = act8(x, v, p.act);
        if (two) *reinterpret_cast<uint4*>(dst + (long long)t * p.N + 8) = act8(x + 8, v + 8, p.act);
      };
#pragma unroll
      for (int t = 0; t < kEarlyFrames; ++t) if (t < sl) frame(t, ev[t]);
      for (int t = kEarlyFrames; t < sl; ++t) {
        float x[kCols];
        ld_global_v8(e + (long long)t * p.N, x);
        if (two) ld_global_v8(e + (long long)t * p.N + 8, x + 8);
        frame(t, x);
      }
      if (__builtin_expect(sl < p.S, 0)) {                    // padding frames (a last, short segment)
#pragma unroll 1
        for (int t = sl; t < p.S; ++t) {
          *reinterpret_cast<uint4*>(dst + (long long)t * p.N) = make_uint4(0, 0, 0, 0);
          if (two) *reinterpret_cast<uint4*>(dst + (long long)t * p.N + 8) = make_uint4(0, 0, 0, 0);
        }
      }
    }
    if (!waited) { pdl_wait(); pdl_trigger(); }
  }
  tc_fence_before();
  settle_copies(ok);
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, 2 * BN);
}

template <int BN>
void launch_wp(const Bf16Mat& A, const CUtensorMap& tmB, const WpOperandParams& p, int mt, cudaStream_t st) {
  const int tiles = mt * ((p.N + BN - 1) / BN);
  launch_pdl(wp_operand_kernel<BN>, dim3(tiles < sm_count() ? tiles : sm_count()), dim3(WpCfg<BN>::kThreads), WpCfg<BN>::kSmem, st, A.as_A, A.as_B32, tmB, p);
}

}  // namespace

int wp_operand_setup() {
  const cudaError_t e1 = cudaFuncSetAttribute(wp_operand_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WpCfg<64>::kSmem);
  const cudaError_t e2 = cudaFuncSetAttribute(wp_operand_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WpCfg<32>::kSmem);
  return (e1 == cudaSuccess && e2 == cudaSuccess) ? TW_OK : TW_ERR_CUDA;
}

// 32-column tiles where 64-column tiles would leave half of the SMs idle: a CTA's time is its operands' way through the SM's
// L2 port and its share of the epilogue
void launch_wp_operand(const Bf16Mat& A, const Bf16Mat& W, const WpOperandParams& p, cudaStream_t st) {
  if (p.M <= 0) return;
  const int mt = (p.M + BM - 1) / BM;
  if (2 * mt * ((p.N + 63) / 64) <= sm_count()) launch_wp<32>(A, W.as_B32, p, mt, st);
  else launch_wp<64>(A, W.as_B64, p, mt, st);
}

}  // namespace tw
