// Hypothesis management of Algorithm 1 on the device: lists A and B, AddAndMerge, the N-th score
// threshold, N-best expansions with the strict '>' filter, segment turn-over, N-best read-out.
// One CTA owns one utterance; utterances advance independently of each other (an utterance whose
// list A runs empty moves to its next segment at once, it does not wait for the batch).
//
// Scores are carried in float64: a hypothesis' log-probability reaches thousands of nats, where
// float32 spacing (1.2e-4 at 2048) is coarser than the accuracy the stage kernels deliver.  The
// stage kernels work on values relative to the row's score, which stay small.
#include <cuda_bf16.h>

#include "operand.cuh"
#include "rank_order.h"
#include "sm100.cuh"

namespace tw {

namespace {

constexpr int kThreads = 256;
constexpr unsigned long long kHashSeed = 0x9E3779B97F4A7C15ull;

__device__ __forceinline__ unsigned long long hash_push(unsigned long long h, int tok) {
  unsigned long long x = h * 0x100000001B3ull + (unsigned long long)(tok + 1);
  x ^= x >> 33; x *= 0xFF51AFD7ED558CCDull;
  x ^= x >> 33; x *= 0xC4CEB9FE1A85EC53ull;
  x ^= x >> 33;
  return x;
}

// The list a segment starts with, ChooseNBest(B) of the one before, in shared memory: slots and scores, best first
struct CarryList { int n; int slot[kMaxBeam]; double ls[kMaxBeam]; };

// Starts the next segment of utterance b, at frame t0 with slen frames: A = ChooseNBest(B) (cl), B = [], d = (s, 0, ..., 0).
// Called by the whole CTA, with cl visible to it.
__device__ void turn_over(const HypState& hs, int b, const CarryList& cl, int t0, int slen) {
  if (threadIdx.x < kMaxBeam) {              // one thread per carried hypothesis
    const int i = threadIdx.x;
    if (i < cl.n) {
      hs.A_slot[b * kMaxBeam + i] = cl.slot[i];
      hs.A_ls[b * kMaxBeam + i] = cl.ls[i];
      hs.A_done[b * kMaxBeam + i] = -INFINITY;
      hs.carry[b * kMaxBeam + i] = cl.slot[i];
    } else {
      hs.carry[b * kMaxBeam + i] = -1;
    }
  }
  if (threadIdx.x == 32) {
    hs.t0[b] = t0;
    hs.slen[b] = slen;
    hs.nA[b] = cl.n;
    hs.nB[b] = 0;
    hs.nTop[b] = 0;
    hs.iters[b] = 0;
    // only the carried hypotheses' slots are held now: the ring starts over, so that the few dozen slots of a segment are the
    // same ones (in L2) again and not, one segment after the other, all N (I_max + 1) of them
    hs.cursor[b] = hs.capSlot - 1;
  }
  for (int i = threadIdx.x; i < cl.n * hs.S; i += blockDim.x) {
    const int a = i / hs.S, t = i - a * hs.S;
    hs.A_ld[((long long)b * kMaxBeam + a) * hs.S + t] = (t == 0) ? cl.ls[a] : -INFINITY;
  }
}

// Row of a hypothesis in the projected predictor outputs: its slot, or (stateless predictor) its last token's row of the table
__device__ __forceinline__ int pp_row(const HypState& hs, long long gs) {
  if (!hs.stateless) return (int)gs;
  const int ln = hs.slot_len[gs];
  return ln > 0 ? hs.slot_tok[gs * hs.U_cap + ln - 1] : hs.empty_row;
}

// Eight operand values of row e_row of E and the hypothesis in slot `slot` of utterance b, from column x on
__device__ __forceinline__ uint4 carry_operand(const HypState& hs, int b, long long e_row, int slot, int x) {
  const float* e = hs.E + e_row * hs.J + x;
  const float* pp = hs.slot_Pp + ((long long)b * hs.capSlot + slot) * hs.J + x;
  return act8(*reinterpret_cast<const float4*>(e), *reinterpret_cast<const float4*>(e + 4), *reinterpret_cast<const float4*>(pp),
              *reinterpret_cast<const float4*>(pp + 4), hs.act);
}

// own_rows, beside a turn_over: the tables and operand rows of the carried hypotheses' joiner rows r0 .. r0 + n - 1.  Called by
// the whole CTA.  (own_rows == 1) of the first `done` operand rows, one per (hypothesis, frame), the first kEarlyCols columns
// have been written.
constexpr int kEarlyCols = 1024;             // four 16-byte pieces a lane, a warp per row
__device__ void carry_rows(const HypState& hs, int b, const CarryList& cl, int t0, int sl, int r0, int done) {
  const int n = cl.n, S = hs.S, J = hs.J, per = J >> 3, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) hs.row_off[b] = r0;
  if (threadIdx.x < n) hs.row_slen[r0 + threadIdx.x] = sl;
  if (hs.own_rows == 2 && threadIdx.x < n) {
    hs.row_e0[r0 + threadIdx.x] = b * hs.E_T + t0;
    hs.row_p[r0 + threadIdx.x] = pp_row(hs, (long long)b * hs.capSlot + cl.slot[threadIdx.x]);
  }
  for (int i = threadIdx.x; i < n * S; i += blockDim.x) hs.row_ld[(long long)r0 * S + i] = (i % S) == 0 ? 0.f : -INFINITY;   // all mass on the first frame
  if (hs.own_rows == 2) return;
#pragma unroll 1
  for (int pair = threadIdx.x >> 5; pair < n * S; pair += blockDim.x >> 5) {
    const int hh = pair / S, t = pair - hh * S, first = pair < done ? kEarlyCols / 8 : 0;
    __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(hs.A_next) + operand_row(r0 + hh, t, S) * J;
    // (padding frames of a short segment: zeros, whatever an older pass left there, see pred_out.cu)
#pragma unroll 1
    for (int c = first + lane; c < per; c += 32)
      *reinterpret_cast<uint4*>(dst + c * 8) = t < sl ? carry_operand(hs, b, (long long)b * hs.E_T + t0 + t, cl.slot[hh], c * 8) : make_uint4(0, 0, 0, 0);
  }
}

// turn_over of an utterance whose list A is empty and that has frames left, from the lists in memory.  Called by the whole CTA.
__device__ void next_segment(const HypState& hs, int b) {
  __shared__ CarryList s_cl;
  __shared__ int s_r0;
  __syncthreads();
  const int n = hs.nTop[b], t0 = hs.t0[b] + hs.slen[b], slen = min(hs.S, hs.len[b] - t0);
  if (threadIdx.x < n) {
    const int e = hs.B_top[b * kMaxBeam + threadIdx.x];
    s_cl.slot[threadIdx.x] = hs.B_slot[(long long)b * hs.capB + e];
    s_cl.ls[threadIdx.x] = hs.B_ls[(long long)b * hs.capB + e];
  }
  if (threadIdx.x == 0) {
    s_cl.n = n;
    if (hs.own_rows) s_r0 = atomicAdd(hs.rows_next, n);
  }
  __syncthreads();
  turn_over(hs, b, s_cl, t0, slen);
  if (hs.own_rows) carry_rows(hs, b, s_cl, t0, slen, s_r0, 0);
}

__global__ void __launch_bounds__(kThreads) hyp_init_kernel(HypState hs, const int* lengths, int T) {
  const int b = blockIdx.x;
  const long long gs = (long long)b * hs.capSlot;   // slot 0 holds the empty hypothesis
  if (threadIdx.x == 0) {
    int len = lengths[b], st = TW_OK;
    if (len < 0) { len = 0; st = TW_ERR_ARG; }
    if (len > T) { len = T; st = TW_ERR_ARG; }
    hs.len[b] = len; hs.status[b] = st; hs.avail[b] = len;
    hs.calls[b] = 0; hs.joins[b] = 0; hs.iters[b] = 0; hs.cursor[b] = 0; hs.n_new[b] = 0;
    hs.t0[b] = 0; hs.slen[b] = 0; hs.nA[b] = 0;
    hs.slot_len[gs] = 0; hs.slot_hash[gs] = kHashSeed;
    // B = [([], 1, InitPredictor(), Null)]
    hs.B_slot[(long long)b * hs.capB] = 0;
    hs.B_ls[(long long)b * hs.capB] = 0.0;
    hs.B_hash[(long long)b * hs.capB] = kHashSeed;
    hs.B_len[(long long)b * hs.capB] = 0;
    hs.nB[b] = 1; hs.nTop[b] = 1; hs.B_top[b * kMaxBeam] = 0;
  }
  if (!hs.stateless) {
    const int nhc = hs.L * 2 * hs.Hd;
    for (int i = threadIdx.x; i < nhc; i += blockDim.x) hs.slot_hc[gs * nhc + i] = hs.init_hc[i];
    for (int i = threadIdx.x; i < hs.J; i += blockDim.x) hs.slot_Pp[gs * hs.J + i] = hs.init_Pp[i];
  }
  __syncthreads();
  if (hs.len[b] > 0) next_segment(hs, b);
}

constexpr int kStepThreads = 512;   // 16 warps: one per hypothesis of list A
constexpr int kSelCap = 64;         // survivors of a row's bound that are ranked directly

__device__ __forceinline__ bool tok_better(float v1, int k1, float v2, int k2) { return v1 > v2 || (v1 == v2 && k1 < k2); }
// (value desc, token asc) of a positive value as one integer, larger first
__device__ __forceinline__ unsigned long long tok_key(float v, int k) { return ((unsigned long long)__float_as_uint(v) << 32) | (0xffffffffu - (unsigned)k); }

// The kernel is a chain of short phases, each as long as its slowest dependent accesses; it is organised to have few of them
// behind the wait for the joiner kernel:
//   ahead of the wait   lists A and B's best entries into shared memory, the search of list B, which of B's best entries are
//                       merged into, the free slots of the ring
//   1                   warp 0: the blank expansions into list B and the threshold (ChooseNthScore); warp 16 + h: the N best
//                       tokens of row h
//   2                   the expansions above the threshold listed, the N best of them
//   3                   work-list entries and rows claimed (atomics); beside that the new hypotheses' tokens, log J of the kept
//                       expansions and the parents' h - or, with nothing kept, the next segment's list and operand rows
//   4                   what goes to the claimed places
// tok_cap: capacity (tokens) of the dynamic shared memory's [N] token sequences of list A's hypotheses, 0: they stay in
// global memory.  Every new hypothesis is a child of one of these, whose tokens the search below reads anyway.
constexpr int kTokStageMax = 24 * 1024;
__global__ void __launch_bounds__(2 * kStepThreads) hyp_step_kernel(HypState hs, int tok_cap) {
  extern __shared__ int s_tok[];
  __shared__ int s_found[kMaxBeam], s_fslot[kMaxBeam];   // the entry of list B that a hypothesis merges with (-1: none), its slot
  __shared__ double s_Bls[kMaxBeam];                     // and score
  __shared__ double s_Als[kMaxBeam];
  __shared__ int s_Aslot[kMaxBeam], s_Alen[kMaxBeam];
  __shared__ unsigned long long s_Ahash[kMaxBeam];
  __shared__ long long s_orow[kMaxBeam];                 // operand row of a hypothesis's first frame (own_rows == 1)
  __shared__ int s_iters, s_nT0, s_Btop[kMaxBeam], s_Btopslot[kMaxBeam];   // list B's best entries as the previous pass left them
  __shared__ double s_Btopls[kMaxBeam];
  __shared__ int s_free[32];                             // the next free slots of the ring
  __shared__ __align__(16) ulonglong2 s_ent[32];         // (key, index) of the entries that B's new best ones are chosen from,
  __shared__ double s_els[32];                           // their scores
  __shared__ int s_eslot[32];                            // and slots
  __shared__ CarryList s_cl;                             // B's new best entries
  __shared__ int s_nB, s_hasthr, s_bad, s_np, s_nkeep, s_wbase, s_rbase;
  __shared__ double s_thr;
  __shared__ int s_ck[kMaxBeam * kMaxBeam];
  __shared__ double s_abs[kMaxBeam * kMaxBeam];
  __shared__ __align__(16) ulonglong2 s_pass[kMaxBeam * kMaxBeam];   // (key, place) of the candidates above the threshold
  __shared__ __align__(16) unsigned s_lm[kMaxBeam][32];  // in-kernel selection: lane maxima, survivors of a row, its chunks to look at
  __shared__ unsigned long long s_sv[kMaxBeam][kSelCap];
  __shared__ unsigned char s_chunk[kMaxBeam][128];
  __shared__ int s_cnt[kMaxBeam];
  __shared__ int s_keep_h[kMaxBeam], s_keep_k[kMaxBeam];
  __shared__ double s_keep_ls[kMaxBeam];
  __shared__ float s_rel[kMaxBeam * 8];                  // own_rows == 1 (S < 8): frame distributions relative to the scores

  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  // The lists and counters read below were written by the previous pass's kernels, all of which had finished before
  // the joiner kernel that runs ahead of this one began (and that kernel writes none of them): they are fetched
  // before the wait for it, under its tail.  Every first-round load is issued before the early exit, so that none
  // of them waits for H.
  const int H = hs.nA[b];
  const int r0 = hs.row_off[b];
  const int slen = hs.slen[b];
  const int nB0 = hs.nB[b];
  const int t0 = hs.t0[b], len = hs.len[b];
  const long long bB = (long long)b * hs.capB;
  const long long bS = (long long)b * hs.capSlot;
  // the search of list B (warp h looks for hypothesis h's tokens): its own slot and the first 32 entries of the list are
  // asked for now as well; the slot's hash and length follow as soon as the slot is there, still before the barriers
  int my_slot = 0, pre_len = -1, pre_slot = 0;
  unsigned long long pre_hash = 0;
  double my_ls = 0.0;
  if (warp < kMaxBeam) {                    // all kMaxBeam entries of the lists; those past H are never used
    my_slot = hs.A_slot[b * kMaxBeam + warp];
    my_ls = hs.A_ls[b * kMaxBeam + warp];
    if (lane < hs.capB) { pre_hash = hs.B_hash[bB + lane]; pre_len = hs.B_len[bB + lane]; pre_slot = hs.B_slot[bB + lane]; }
  }
  const int N = hs.N, S = hs.S, V = hs.V;
  const bool two_halves = hs.dnb_sel != nullptr;     // with in-kernel selection: 32 warps, the upper half selects
  if (H == 0) {                              // idle (finished) utterance
    pdl_wait();
    pdl_trigger();
    return;
  }
  if (warp == 15) {
    // ring cursor, pass counter and the best-N set of list B as the previous pass left it, by a warp that mostly has
    // nothing to do in the search
    const int nT = hs.nTop[b], cursor = hs.cursor[b], iters = hs.iters[b];
    const int carry = lane < kMaxBeam ? hs.carry[b * kMaxBeam + lane] : -1;
    if (lane < nT) {
      const int bt = hs.B_top[b * kMaxBeam + lane];
      s_Btop[lane] = bt;
      s_Btopls[lane] = hs.B_ls[bB + bt];                      // before this pass's merges
      s_Btopslot[lane] = hs.B_slot[bB + bt];
    }
    // The ring's slots after the cursor; those still held by hypotheses carried into this segment are skipped.  At most
    // N of them are, and at most N are wanted: 32 slots hold enough (a ring that is shorter starts over).
    const int slot = (cursor + 1 + lane) % hs.capSlot;
    bool busy = false;
#pragma unroll 4
    for (int q = 0; q < kMaxBeam; ++q) busy |= __shfl_sync(0xffffffffu, carry, q) == slot;
    const unsigned free_mask = __ballot_sync(0xffffffffu, !busy);
    if (!busy) s_free[__popc(free_mask & ((1u << lane) - 1u))] = slot;
    if (lane == 0) { s_iters = iters; s_nT0 = nT; s_bad = 0; s_np = 0; }
  }
  if (tid < kMaxBeam && hs.own_rows == 1) s_orow[tid] = operand_row(r0 + tid, 0, S);
  // ---- AddAndMerge, search: warp h looks for the tokens of A_h among the entries already in B.  It needs the lists only,
  // so it runs ahead of the wait.  (Entries of A are distinct sequences, so two of them never merge with each other.)
  if (warp < H) {                            // (H <= kMaxBeam)
    const unsigned long long my_hash = hs.slot_hash[bS + my_slot];
    const int my_len = hs.slot_len[bS + my_slot];
    const int* ta = hs.slot_tok + (bS + my_slot) * hs.U_cap;
    if (tok_cap > 0) for (int i = lane; i < my_len; i += 32) s_tok[warp * tok_cap + i] = ta[i];
    int found = -1, fslot = my_slot;
    for (int base = 0; base < nB0 && found < 0; base += 32) {
      const int e = base + lane;
      const bool match = e < nB0 && (base == 0 ? (pre_hash == my_hash && pre_len == my_len)
                                               : (hs.B_hash[bB + e] == my_hash && hs.B_len[bB + e] == my_len));
      unsigned mask = __ballot_sync(0xffffffffu, match);
      while (mask != 0 && found < 0) {
        const int c = base + __ffs(mask) - 1;
        mask &= mask - 1;
        const int oslot = base == 0 ? __shfl_sync(0xffffffffu, pre_slot, c) : hs.B_slot[bB + c];
        int diff = 0;                       // a 64-bit hash match is not proof: compare the tokens
        if (oslot != my_slot) {
          const int* tb = hs.slot_tok + (bS + oslot) * hs.U_cap;
          for (int i = lane; i < my_len; i += 32) diff |= (ta[i] != tb[i]);
        }
        if (!__any_sync(0xffffffffu, diff)) { found = c; fslot = oslot; }
      }
    }
    if (lane == 0) {
      s_found[warp] = found; s_fslot[warp] = fslot; s_Alen[warp] = my_len; s_Ahash[warp] = my_hash;
      s_Bls[warp] = found >= 0 ? hs.B_ls[bB + found] : 0.0;
    }
  }
  if (warp < kMaxBeam && lane == 0) { s_Als[warp] = my_ls; s_Aslot[warp] = my_slot; }
  __syncthreads();

  // ---- warp 0, still ahead of the wait: lanes 0 .. 15 hold B's old best entries, lane 16 + h the entry that hypothesis h
  // goes to.  m_src: the lane of the hypothesis that is merged into this old best entry.
  int idx = -1, m_src = -1, m_slot = 0;
  bool m_old = false, m_dup = false;
  double score = -INFINITY, done = -INFINITY;
  if (warp == 0) {
    const int nT = s_nT0, h = lane - 16;
    const int f = h >= 0 && h < H ? s_found[h] : 0;
    const unsigned appended = __ballot_sync(0xffffffffu, f < 0);
    if (lane == 0) s_nB = nB0 + __popc(appended);      // capB = N * I_max bounds this by construction
    if (h < 0) {
      if (lane < nT) {
        idx = s_Btop[lane]; score = s_Btopls[lane]; m_slot = s_Btopslot[lane];
#pragma unroll 4
        for (int q = 0; q < H; ++q) if (s_found[q] == idx) m_src = 16 + q;
      }
    } else if (h < H) {
      m_old = f >= 0;
      idx = m_old ? f : nB0 + __popc(appended & ((1u << lane) - 1u));
      m_slot = s_fslot[h];
      if (hs.mono) done = hs.A_done[b * kMaxBeam + h];
#pragma unroll 4
      for (int i = 0; i < nT; ++i) m_dup |= s_Btop[i] == f;
    }
  }
  pdl_wait();                               // from here on: what the joiner kernel wrote (delta_phi, delta_nb, occupancies)
  pdl_trigger();

  if (warp == 0) {
    // ---- AddAndMerge, apply: sum into the matching entry or append (appends keep the order of A)
    const int h = lane - 16;
    if (h >= 0 && h < H) {
      const double dphi = hs.ldphi_d ? hs.ldphi_d[r0 + h] : (double)hs.ldphi[r0 + h];
      double val = s_Als[h] + dphi;
      if (hs.mono) val = logaddexp_d(val, done);       // plus what had already left the segment (else log 0)
      if (m_old) {
        val = logaddexp_d(s_Bls[h], val);              // (two hypotheses never merge with the same entry)
      } else {
        hs.B_slot[bB + idx] = s_Aslot[h];
        hs.B_hash[bB + idx] = s_Ahash[h]; hs.B_len[bB + idx] = s_Alen[h];
      }
      hs.B_ls[bB + idx] = val;
      score = val;
    }
    // ---- ChooseNthScore: the best N of B are among the previous best N and the entries touched now
    const double merged = __shfl_sync(0xffffffffu, score, m_src & 31);
    if (m_src >= 0) score = merged;
    if (m_dup) idx = -1;                     // it stands among the old best entries
    s_ent[lane] = make_ulonglong2(order_key(score), (unsigned long long)(long long)idx);
    s_els[lane] = score; s_eslot[lane] = m_slot;
    const int count = __popc(__ballot_sync(0xffffffffu, idx >= 0));
    if (lane == 0) { s_cl.n = min(N, count); s_hasthr = count >= N; }
  } else if (warp == 1 && lane == 0) {
    atomicAdd(&hs.calls[b], 1);              // (nobody else writes these: additions without a round trip)
    atomicAdd(&hs.joins[b], slen);
    if (hs.own_rows) {                      // totals of the pass
      atomicAdd(reinterpret_cast<unsigned long long*>(hs.rows_total), (unsigned long long)H);
      atomicAdd(reinterpret_cast<unsigned long long*>(hs.rows_total) + 1, (unsigned long long)(H * slen));
    }
  }
  if (warp < 16) {
    if (!two_halves && warp >= 8) {                     // the rows' candidate lists, by the warps that merge nothing
      const int c = tid - kMaxBeam * kMaxBeam, h = c / kMaxBeam, j = c % kMaxBeam;
      int n = 0, k = -1;
      float v = 0.f;
      if (h < H) {
        const long long at = (long long)(r0 + h) * kMaxBeam + j;
        n = hs.cand_n[r0 + h]; v = hs.cand_v[at]; k = hs.cand_k[at];
      }
      s_abs[c] = j < n ? s_Als[h] + (double)v : -INFINITY;
      s_ck[c] = j < n ? k : -1;
    }
    // the entries' ranks, two a warp: every lane compares with one of the others
    asm volatile("bar.sync 1, 512;" ::: "memory");
    const ulonglong2 o = s_ent[lane];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = 2 * warp + u;
      const ulonglong2 me = s_ent[e];
      const int oi = (int)o.y, mi = (int)me.y;
      const int rank = __popc(__ballot_sync(0xffffffffu, oi >= 0 && (o.x > me.x || (o.x == me.x && oi < mi))));
      if (lane == 0 && mi >= 0 && rank < N) {
        hs.B_top[b * kMaxBeam + rank] = mi;
        s_cl.slot[rank] = s_eslot[e]; s_cl.ls[rank] = s_els[e];
        if (rank == N - 1) s_thr = s_els[e];
      }
    }
  }
  if (two_halves && warp >= 16) {
    // ---- ChooseNBestExpansions, first stage, for the row of hypothesis warp - 16: its N best tokens by delta_nb,
    // order (value desc, token asc), straight into the candidate table of the second stage.
    const int h = warp - 16;
    if (lane < kMaxBeam) {
      s_abs[h * kMaxBeam + lane] = -INFINITY; s_ck[h * kMaxBeam + lane] = -1;
    }
    if (h < H) {
      const float* src = hs.dnb_sel + (long long)(r0 + h) * V;
      const double base = s_Als[h];
      // a lower bound of the N-th best value: the N-th largest of the 32 lane maxima (distinct elements), whose last five bits
      // make room for the lane
      const int nchunk = V >> 5;
      const bool pairs = hs.dnb_chunk == 16;     // maxima of 16 columns: two make a chunk's
      const float* cmax = (hs.dnb_max != nullptr && (V & 31) == 0 && nchunk <= 128) ? hs.dnb_max + (long long)(r0 + h) * (pairs ? 2 * nchunk : nchunk) : nullptr;
      float lmax = 0.f;
      float m4[4] = {0.f, 0.f, 0.f, 0.f};        // with chunk maxima: those of chunks lane, lane + 32, lane + 64, lane + 96
      if (cmax != nullptr) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = lane + 32 * u;
          if (c < nchunk) {
            if (pairs) { const float2 m2 = __ldg(reinterpret_cast<const float2*>(cmax) + c); m4[u] = fmaxf(m2.x, m2.y); }
            else m4[u] = __ldg(cmax + c);
          }
          lmax = fmaxf(lmax, m4[u]);
        }
      } else {
#pragma unroll 8
        for (int k = lane * 4; k < V; k += 128) {             // eight independent loads in flight per lane
          const float4 v = __ldg(reinterpret_cast<const float4*>(src + k));
          lmax = fmaxf(fmaxf(lmax, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
        }
      }
      const unsigned lkey = (__float_as_uint(lmax) & ~31u) | (31u - lane);
      s_lm[h][lane] = lkey;
      if (lane == 0) s_cnt[h] = 0;
      __syncwarp();
      int lrank = 0;
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(&s_lm[h][j]);
        lrank += (o.x > lkey) + (o.y > lkey) + (o.z > lkey) + (o.w > lkey);
      }
      const unsigned who = __ballot_sync(0xffffffffu, lrank == N - 1);        // exactly one lane: the ranks are 0..31
      const float bound = __uint_as_float(__shfl_sync(0xffffffffu, lkey, __ffs(who) - 1) & ~31u);
      auto push4 = [&](const float4& v4, int k) {
        const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (vv[c] >= bound && vv[c] > 0.f) {
            const int i = atomicAdd(&s_cnt[h], 1);
            if (i < kSelCap) s_sv[h][i] = tok_key(vv[c], k + c);
          }
        }
      };
      if (cmax != nullptr) {
        // Only the chunks whose maximum reaches the bound can hold a survivor: a few 128-byte pieces of the row, N or some
        // more of them.  They are listed, and the warp takes sixteen at a time, eight lanes to a piece, so that their loads
        // (mostly from DRAM: a large step moves more than L2 holds) are in flight at the same time.
        int total = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool in = m4[u] >= bound && m4[u] > 0.f;
          const unsigned m = __ballot_sync(0xffffffffu, in);
          if (in) s_chunk[h][total + __popc(m & ((1u << lane) - 1u))] = (unsigned char)(lane + 32 * u);
          total += __popc(m);
        }
        __syncwarp();
        const int k0 = (lane & 7) * 4;
#pragma unroll 1
        for (int c0 = lane >> 3; c0 - (lane >> 3) < total; c0 += 16) {
          float4 v[4];
          int id[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const bool in = c0 + 4 * x < total;
            id[x] = in ? (int)s_chunk[h][c0 + 4 * x] * 32 + k0 : 0;
            v[x] = in ? __ldg(reinterpret_cast<const float4*>(src + id[x])) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const float g = fmaxf(fmaxf(v[x].x, v[x].y), fmaxf(v[x].z, v[x].w));
            if (g >= bound && g > 0.f) push4(v[x], id[x]);
          }
        }
      } else {
        // second sweep (the row is in L2): eight loads at a time, and only a group of four that holds a survivor
        // enters the branch with the shared-memory counter
        for (int k0 = lane * 4; k0 < V; k0 += 8 * 128) {
          float4 v8[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int k = k0 + u * 128;
            v8[u] = k < V ? __ldg(reinterpret_cast<const float4*>(src + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const float g = fmaxf(fmaxf(v8[u].x, v8[u].y), fmaxf(v8[u].z, v8[u].w));
            if (g >= bound && g > 0.f) push4(v8[u], k0 + u * 128);
          }
        }
      }
      __syncwarp();
      const int ns = s_cnt[h];
      if (ns <= kSelCap) {
        for (int i = lane; i < ns; i += 32) {
          const unsigned long long me = s_sv[h][i];
          int rank = 0;
#pragma unroll 4
          for (int j = 0; j < ns; ++j) rank += s_sv[h][j] > me ? 1 : 0;
          if (rank < N) {
            s_abs[h * kMaxBeam + rank] = base + (double)__logf(__uint_as_float((unsigned)(me >> 32)));
            s_ck[h * kMaxBeam + rank] = (int)(0xffffffffu - (unsigned)me);
          }
        }
      } else {
        // many ties at the bound: N rounds, each taking the best element after the previous pick in that order
        float pv = INFINITY; int pk = -1;
        for (int j = 0; j < N; ++j) {
          float bv = 0.f; int bk = 0x7fffffff;
          for (int k = lane * 4; k < V; k += 128) {
            const float4 v4 = __ldg(reinterpret_cast<const float4*>(src + k));
            const float vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const bool after = vv[c] < pv || (vv[c] == pv && k + c > pk);
              if (vv[c] > 0.f && after && tok_better(vv[c], k + c, bv, bk)) { bv = vv[c]; bk = k + c; }
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
            if (tok_better(ov, ok, bv, bk)) { bv = ov; bk = ok; }
          }
          if (!(bv > 0.f)) break;
          if (lane == 0) { s_abs[h * kMaxBeam + j] = base + (double)__logf(bv); s_ck[h * kMaxBeam + j] = bk; }
          pv = bv; pk = bk;
        }
      }
      // (hardly ever: neighbours whose logarithms are in the other order)
      __syncwarp();
      double* row = s_abs + h * kMaxBeam;
      if (__any_sync(0xffffffffu, lane > 0 && lane < N && row[lane] > row[lane - 1]) && lane == 0) settle_row(row, N);
    }
  }
  __syncthreads();

  // ---- ChooseNBestExpansions, second stage: the N best (h, k) over the rows' candidate lists, in float64; order (score desc, h
  // asc, k asc), which within a row is the order of its list.  Only those above the threshold are ever kept (Length(B) < N or
  // delta_nb > threshold), and all that rank before such a one are above it too: they are listed, mostly a handful, and
  // ranked among themselves, a warp per candidate with a lane for each of the others.
  if (tid < kMaxBeam * kMaxBeam) {
    // (a row with N candidates bounds the N-th best score from below by its last one, log 0 where there is none: the first row,
    // the best hypothesis's, leaves few to rank (one utterance, N = 10: 28.3 -> 27.6 ms); the largest of all rows' bounds leaves
    // fewer and takes longer than it saves at N = 5).  No score rises along its row.
    const double sc = s_abs[tid], low = s_abs[N - 1];
    const bool pass = s_ck[tid] >= 0 && !(sc < low) && (s_hasthr == 0 || sc > s_thr);
    const unsigned m = __ballot_sync(0xffffffffu, pass);
    if (m != 0) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&s_np, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (pass) s_pass[at] = make_ulonglong2(order_key(sc), (unsigned long long)tid);
    }
  }
  __syncthreads();
  const int np = s_np;
  for (int i = warp; i < np; i += nwarps) {
    const ulonglong2 me = s_pass[i];
    int rank = 0;
    for (int j = 0; j < np; j += 32) {
      const ulonglong2 o = j + lane < np ? s_pass[j + lane] : make_ulonglong2(0, ~0ull);     // ahead of nobody
      rank += __popc(__ballot_sync(0xffffffffu, ranks_before(o.x, o.y, me.x, me.y)));
    }
    if (lane == 0 && rank < N) {
      const int c = (int)me.y, h = c / kMaxBeam;
      s_keep_h[rank] = h; s_keep_k[rank] = s_ck[c]; s_keep_ls[rank] = s_abs[c];
      if (s_Alen[h] + 1 > hs.U_cap) s_bad = 1;
    }
  }
  __syncthreads();
  int nk = min(np, N);
  if (nk > 0 && (s_iters + 1 >= hs.I_max || s_bad != 0)) {   // pass cap or token capacity: what does not fit is dropped
    if (warp == 0) {
      const int h = lane < nk ? s_keep_h[lane] : 0, k = lane < nk ? s_keep_k[lane] : 0;
      const double ls = lane < nk ? s_keep_ls[lane] : 0.0;
      const bool keep = lane < nk && s_iters + 1 < hs.I_max && s_Alen[h] + 1 <= hs.U_cap;
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      if (keep) { const int i = __popc(m & ((1u << lane) - 1u)); s_keep_h[i] = h; s_keep_k[i] = k; s_keep_ls[i] = ls; }
      if (lane == 0) { s_nkeep = __popc(m); hs.status[b] = TW_ERR_LIMIT; }
    }
    __syncthreads();
    nk = s_nkeep;
  }
  // list A empty and frames left: this segment is done, the next one starts with ChooseNBest(B)
  const bool turn = nk == 0 && t0 + slen < len;
  const int t0n = t0 + slen, slen_n = min(S, len - t0n);

  // ---- the places in the work list and among the joiner rows; everybody else goes on until the barrier below
  int claimed = 0;
  if (warp == 0) {
    const bool listed = (hs.inline_gather || hs.own_rows == 2) && nk > 0;
    const int rows = turn ? s_cl.n : nk;
    if (lane == 0 && listed) claimed = atomicAdd(&hs.scalars[kScNPred], nk);
    if (lane == 1 && hs.own_rows && rows > 0) claimed = atomicAdd(hs.rows_next, rows);
  }
  // the first pieces of the parents' h (or of the carried hypotheses' operand rows), a warp per row of up to kEarlyCols values:
  // fetched here, written below
  uint4 pk[4];
  const int L = hs.L, Hd = hs.Hd;
  const long long stride = (long long)L * 2 * Hd;
  const bool vec = (Hd & 7) == 0 && (reinterpret_cast<uintptr_t>(hs.slot_hc) & 15) == 0;
  const bool gather = hs.inline_gather && nk > 0;
  auto h_src = [&](int i, int l) { return hs.slot_hc + (bS + s_Aslot[s_keep_h[i]]) * stride + (long long)l * 2 * Hd; };
  auto h_piece = [&](const float* src) {
    const float4 a = *reinterpret_cast<const float4*>(src), e = *reinterpret_cast<const float4*>(src + 4);
    const __nv_bfloat162 p0 = __floats2bfloat162_rn(a.x, a.y), p1 = __floats2bfloat162_rn(a.z, a.w);
    const __nv_bfloat162 p2 = __floats2bfloat162_rn(e.x, e.y), p3 = __floats2bfloat162_rn(e.z, e.w);
    return make_uint4(*reinterpret_cast<const uint32_t*>(&p0), *reinterpret_cast<const uint32_t*>(&p1),
                      *reinterpret_cast<const uint32_t*>(&p2), *reinterpret_cast<const uint32_t*>(&p3));
  };
  const bool early_op = turn && hs.own_rows == 1 && warp < s_cl.n * S;
  const int o_h = early_op ? warp / S : 0, o_t = warp - o_h * S;
  // (the first nk warps write the new lists: the rows go to those behind them, the dot products to the last ones)
  const int g_at = warp - nk;
  const bool early_h = gather && vec && g_at >= 0 && g_at < nk * L;
  __nv_bfloat16* g_dst = nullptr;            // this warp's destination, for work-list entry 0
  int g_ld = 0;
  if (early_h) {
    const int i = g_at / L, l = g_at - i * L;
    const float* src = h_src(i, l);
#pragma unroll
    for (int u = 0; u < 4; ++u) { const int x = (lane + 32 * u) * 8; if (x < Hd) pk[u] = h_piece(src + x); }
    g_ld = hs.xg_ld[l];
    g_dst = reinterpret_cast<__nv_bfloat16*>(hs.xg_dst[l]) + (long long)i * g_ld + hs.xg_off[l];
  } else if (early_op) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int x = (lane + 32 * u) * 8;
      if (x < hs.J) pk[u] = o_t < slen_n ? carry_operand(hs, b, (long long)b * hs.E_T + t0n + o_t, s_cl.slot[o_h], x) : make_uint4(0, 0, 0, 0);
    }
  }

  if (turn) {
    turn_over(hs, b, s_cl, t0n, slen_n);
    if (tid == 32) hs.n_new[b] = 0;
  } else if (tid == 32) {
    hs.nB[b] = s_nB;
    hs.nTop[b] = s_cl.n;
    hs.iters[b] = s_iters + 1;
    hs.nA[b] = nk; hs.n_new[b] = nk;
    if (nk > 0) hs.cursor[b] = s_free[nk - 1];
  }

  // ---- own_rows: log J(t, k) of the kept expansions, a warp per (expansion, frame), the last warps first (the first ones
  // write the new lists below); their joiner rows' frame distributions relative to their scores
  if (hs.own_rows == 1) {
    const int J = hs.J;
    for (int pair = nwarps - 1 - warp; pair < nk * slen; pair += nwarps) {
      const int i = pair / slen, t = pair - i * slen;
      const int h = s_keep_h[i], k = s_keep_k[i];
      const long long rt = (long long)(r0 + h) * S + t;
      const __nv_bfloat16* arow = static_cast<const __nv_bfloat16*>(hs.A_cur) + (s_orow[h] + t) * J;
      const __nv_bfloat16* wrow = static_cast<const __nv_bfloat16*>(hs.W_out) + (long long)k * J;
      const float la = hs.la[rt], lse = hs.lse_j[rt], bias = hs.b_out[k];
      float acc = 0.f;
#pragma unroll 4
      for (int x = lane * 8; x < J; x += 256) {
        const uint4 av = *reinterpret_cast<const uint4*>(arow + x), wv = __ldg(reinterpret_cast<const uint4*>(wrow + x));
        const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&av);
        const __nv_bfloat162* w2 = reinterpret_cast<const __nv_bfloat162*>(&wv);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 af = __bfloat1622float2(a2[u]), wf = __bfloat1622float2(w2[u]);
          acc = fmaf(af.x, wf.x, fmaf(af.y, wf.y, acc));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) {
        const double d = s_Als[h] + (double)la + ((double)(acc + bias) - (double)lse), ls = s_keep_ls[i];
        const float rel = d == -INFINITY ? -INFINITY : (float)(d - ls);
        float* out = s_rel + i * 8;
        if (!hs.mono) {
          out[t] = rel;
        } else {                            // emitted at frame t: continues at t + 1, or has left the segment
          if (t == 0) out[0] = -INFINITY;
          if (t + 1 < slen) out[t + 1] = rel;
          else hs.A_done[b * kMaxBeam + i] = d;
        }
      }
    }
  }

  // ---- new list A (one warp per kept expansion): tokens, hash, frame distribution d_h(k) (Eq. 5)
  long long gp = 0, gn = 0;
  double d_t[2] = {-INFINITY, -INFINITY};             // the distribution at frames lane and lane + 32 (S <= 64)
  if (warp < nk) {
    const int i = warp;
    const int h = s_keep_h[i], k = s_keep_k[i], slot = s_free[i];
    gp = bS + s_Aslot[h]; gn = bS + slot;
    const int plen = s_Alen[h];
    const int* src = tok_cap > 0 ? s_tok + h * tok_cap : hs.slot_tok + gp * hs.U_cap;
    int* dst = hs.slot_tok + gn * hs.U_cap;
    for (int q = lane; q < plen; q += 32) dst[q] = src[q];
    if (lane == 0) {
      dst[plen] = k;
      hs.slot_len[gn] = plen + 1;
      hs.slot_hash[gn] = hash_push(s_Ahash[h], k);
      hs.new_slot[b * kMaxBeam + i] = (int)gn;
      hs.new_par[b * kMaxBeam + i] = (int)gp;
      hs.new_tok[b * kMaxBeam + i] = k;
      hs.new_row[b * kMaxBeam + i] = r0 + h;
      hs.A_slot[b * kMaxBeam + i] = slot;
      hs.A_ls[b * kMaxBeam + i] = s_keep_ls[i];
    }
    if (hs.inline_gather && lane == 0) {           // what the predictor will read of this hypothesis's token and parent
      if (hs.pf_table != nullptr) sm100::prefetch_l2_bulk(hs.pf_table + (long long)k * hs.pf_row_bytes, (uint32_t)hs.pf_row_bytes);
      if ((Hd & 3) == 0) {
        const float* pc = hs.slot_hc + gp * stride + Hd;      // the parent's c, layer by layer
        for (int l = 0; l < L; ++l) sm100::prefetch_l2_bulk(pc + (long long)l * 2 * Hd, (uint32_t)Hd * 4u);
      }
    }
    const long long r = r0 + h;
    // d_h(k) at frame t of the segment: occupancy times J(t, k)
    auto d_at = [&](int t) -> double {
      if (t < 0 || t >= slen) return -INFINITY;
      const double a = hs.la_d ? hs.la_d[r * S + t] : (double)hs.la[r * S + t];
      double v = s_Als[h] + a;
      if (hs.logp != nullptr) {      // otherwise log J(t, k) is added by a follow-up kernel
        double lj = (double)hs.logp[(r * S + t) * V + k];
        if (hs.lse) lj -= (double)hs.lse[r * S + t];
        v += lj;
      }
      return v;
    };
    if (hs.own_rows != 1) {
      // (monotonic: emitted at frame t, the hypothesis continues at frame t + 1, or has left the segment)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = lane + 32 * u;
        if (t < S) d_t[u] = !hs.mono ? d_at(t) : (t < slen ? d_at(t - 1) : -INFINITY);
      }
      if (hs.mono && lane == 0) hs.A_done[b * kMaxBeam + i] = d_at(slen - 1);
    }
  }
  if (warp == 0) {
    if (lane == 0) s_wbase = claimed;
    if (lane == 1) s_rbase = claimed;
  }
  __syncthreads();

  // ---- what goes to the claimed places
  const int wbase = s_wbase, rbase = s_rbase;
  if (turn) {
    if (early_op) {
      __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(hs.A_next) + operand_row(rbase + o_h, o_t, S) * hs.J;
#pragma unroll
      for (int u = 0; u < 4; ++u) { const int x = (lane + 32 * u) * 8; if (x < hs.J) *reinterpret_cast<uint4*>(dst + x) = pk[u]; }
    }
    if (hs.own_rows) carry_rows(hs, b, s_cl, t0n, slen_n, rbase, nwarps);
    return;
  }
  if (nk == 0) return;
  if (hs.own_rows) {
    if (tid == 32) hs.row_off[b] = rbase;
    if (tid < nk) hs.row_slen[rbase + tid] = slen;
  }
  if (hs.own_rows == 1) {
    if (tid < nk * 8 && (tid & 7) < slen) hs.row_ld[(long long)(rbase + (tid >> 3)) * S + (tid & 7)] = s_rel[tid];
  } else if (warp < nk) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int t = lane + 32 * u;
      const double d = d_t[u];
      if (t >= S) continue;
      if (hs.own_rows == 2) hs.row_ld[(long long)(rbase + warp) * S + t] = d == -INFINITY ? -INFINITY : (float)(d - s_keep_ls[warp]);
      else hs.A_ld[((long long)b * kMaxBeam + warp) * S + t] = d;
    }
  }
  if (warp < nk && lane == 0 && (hs.inline_gather || hs.own_rows == 2)) {      // the predictor's work-list entry, the joiner row's tables
    const int wrow = wbase + warp, k = s_keep_k[warp];
    if (wrow < hs.B * hs.N) {
      hs.pw_new[wrow] = (int)gn; hs.pw_par[wrow] = (int)gp; hs.pw_tok[wrow] = k;
      if (hs.inline_gather) hs.pw_bi[wrow] = b * kMaxBeam + warp;
    } else {
      hs.status[b] = TW_ERR_LIMIT;                   // cannot happen: the list holds at most N entries per utterance
    }
    if (hs.own_rows == 2) {
      hs.row_e0[rbase + warp] = b * hs.E_T + t0;
      hs.row_p[rbase + warp] = hs.stateless ? k : (int)gn;
    }
  }
  // the parents' h of every layer as bf16 in the recurrent halves of the gate GEMMs' operand rows
  if (!gather || wbase + nk > hs.B * hs.N) return;
  bool done_early = false;
  if (early_h) {
    __nv_bfloat16* d = g_dst + (long long)wbase * g_ld;
    done_early = (reinterpret_cast<uintptr_t>(d) & 15) == 0 && Hd <= kEarlyCols;
    if (done_early) {
#pragma unroll
      for (int u = 0; u < 4; ++u) { const int x = (lane + 32 * u) * 8; if (x < Hd) *reinterpret_cast<uint4*>(d + x) = pk[u]; }
    }
  }
  // (rows that have not been fetched early, or not whole)
#pragma unroll 1
  for (int pair = g_at; pair < nk * L; pair += nwarps) {
    if (pair < 0 || (pair == g_at && done_early)) continue;
    const int i = pair / L, l = pair - i * L;
    const float* src = h_src(i, l);
    __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(hs.xg_dst[l]) + (long long)(wbase + i) * hs.xg_ld[l] + hs.xg_off[l];
    if (vec && (reinterpret_cast<uintptr_t>(d) & 15) == 0) {
      for (int x = lane * 8; x < Hd; x += 256) *reinterpret_cast<uint4*>(d + x) = h_piece(src + x);
    } else {
      for (int x = lane; x < Hd; x += 32) d[x] = __float2bfloat16_rn(src[x]);
    }
  }
}

// One CTA: packs the live hypotheses of all utterances into joiner rows and the new hypotheses
// into the predictor's work list.
__global__ void __launch_bounds__(1024) compact_kernel(HypState hs, int B, int T) {
  __shared__ int s_wa[32], s_wn[32];       // per-warp totals of the two scans
  __shared__ int s_cnt[1024], s_off[1024]; // batches of up to 1024 utterances: nA | n_new << 8, row_off | new_off << 16 kept on chip
  __shared__ int s_base_a, s_base_n, s_frames;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_wait();
  pdl_trigger();
  if (tid == 0) { s_base_a = 0; s_base_n = 0; s_frames = 0; }
  __syncthreads();
  // exclusive scans of the list sizes -> row_off, new_off (shuffle scan per warp, then over the warp totals)
  for (int b0 = 0; b0 < B; b0 += 1024) {
    const int b = b0 + tid;
    const int a = b < B ? hs.nA[b] : 0;
    const int nn = b < B ? hs.n_new[b] : 0;
    const int fr = (b < B && a > 0) ? a * hs.slen[b] : 0;
    int ia = a, in = nn;                   // inclusive scans inside the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int va = __shfl_up_sync(0xffffffffu, ia, o), vn = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) { ia += va; in += vn; }
    }
    if (lane == 31) { s_wa[warp] = ia; s_wn[warp] = in; }
    if (fr > 0) atomicAdd(&s_frames, fr);
    __syncthreads();
    int pa = 0, pn = 0;                    // totals of the warps before this one
    for (int w = 0; w < warp; ++w) { pa += s_wa[w]; pn += s_wn[w]; }
    if (b < B) {
      hs.row_off[b] = s_base_a + pa + ia - a;
      hs.new_off[b] = s_base_n + pn + in - nn;
      if (B <= 1024) { s_cnt[tid] = a | (nn << 8); s_off[tid] = (pa + ia - a) | ((pn + in - nn) << 16); }
    }
    __syncthreads();
    if (tid == 1023) { s_base_a += pa + ia; s_base_n += pn + in; }
    __syncthreads();
  }
  // fill: one thread per (utterance, list position)
  for (int idx = tid; idx < B * kMaxBeam; idx += 1024) {
    const int b = idx / kMaxBeam, h = idx % kMaxBeam;
    const bool chip = B <= 1024;           // offsets fit 16 bits: at most 1024 * kMaxBeam rows
    const int nA_b = chip ? (s_cnt[b] & 255) : hs.nA[b], nnew_b = chip ? (s_cnt[b] >> 8) : hs.n_new[b];
    if (h < nA_b && !hs.defer_rows) {
      const int r = (chip ? (s_off[b] & 0xffff) : hs.row_off[b]) + h;
      const int slot = hs.A_slot[b * kMaxBeam + h];
      const long long gs = (long long)b * hs.capSlot + slot;
      hs.row_e0[r] = b * T + hs.t0[b];
      hs.row_slen[r] = hs.slen[b];
      if (hs.stateless) {
        const int ln = hs.slot_len[gs];
        hs.row_p[r] = ln > 0 ? hs.slot_tok[gs * hs.U_cap + ln - 1] : hs.empty_row;
      } else {
        hs.row_p[r] = (int)gs;
      }
      const double ls = hs.A_ls[b * kMaxBeam + h];
      for (int t = 0; t < hs.S; ++t) {
        const double d = hs.A_ld[((long long)b * kMaxBeam + h) * hs.S + t];
        hs.row_ld[(long long)r * hs.S + t] = (d == -INFINITY) ? -INFINITY : (float)(d - ls);
      }
    }
    if (h < nnew_b) {
      const int o = (chip ? (s_off[b] >> 16) : hs.new_off[b]) + h;
      hs.pw_new[o] = hs.new_slot[b * kMaxBeam + h];
      hs.pw_par[o] = hs.new_par[b * kMaxBeam + h];
      hs.pw_tok[o] = hs.new_tok[b * kMaxBeam + h];
    }
  }
  __syncthreads();
  if (!hs.defer_rows) for (int b = tid; b < B; b += 1024) hs.n_new[b] = 0;
  if (tid == 0) {
    const int R = s_base_a;
    hs.scalars[kScR] = R;
    hs.scalars[kScM] = R * hs.S;
    hs.scalars[kScNPred] = s_base_n;
    hs.scalars[kScActive] = R > 0;
    if (R > 0) { hs.scalars[kScSteps] += 1; hs.rows_total[0] += R; hs.rows_total[1] += s_frames; }
  }
}

__global__ void stream_rows_kernel(HypState hs, const int* chunk_lens, int B, int Tc, int max_T, int dump_row, int* oidx) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= B * Tc) return;
  const int b = m / Tc, i = m - b * Tc;
  const int have = hs.avail[b];
  const bool ok = i < chunk_lens[b] && have + i < max_T;
  oidx[m] = ok ? b * max_T + have + i : dump_row;
}

__global__ void __launch_bounds__(kThreads) stream_advance_kernel(HypState hs, const int* chunk_lens, int max_T, int closing) {
  const int b = blockIdx.x;
  __shared__ int s_go;
  if (threadIdx.x == 0) {
    int add = chunk_lens ? max(chunk_lens[b], 0) : 0;
    int have = hs.avail[b];
    if (have + add > max_T) { add = max_T - have; hs.status[b] = TW_ERR_LIMIT; }
    have += add;
    hs.avail[b] = have;
    const int len = closing ? have : (have / hs.S) * hs.S;    // only whole segments while the stream is open
    hs.len[b] = len;
    s_go = (hs.nA[b] == 0 && hs.t0[b] + hs.slen[b] < len);
  }
  __syncthreads();
  if (s_go) next_segment(hs, b);
}

// ChooseNBest(B) at the end of the utterance, best first.
__global__ void __launch_bounds__(kThreads) finish_kernel(HypState hs, int* out_tokens, int* out_lens,
                                                          double* out_scores, int* out_status) {
  const int b = blockIdx.x;
  const int nT = hs.nTop[b];
  for (int i = 0; i < hs.N; ++i) {
    int* dst = out_tokens + ((long long)b * hs.N + i) * hs.U_cap;
    int ln = -1;
    double sc = -INFINITY;
    const int* src = nullptr;
    if (i < nT) {
      const int e = hs.B_top[b * kMaxBeam + i];
      const long long gs = (long long)b * hs.capSlot + hs.B_slot[(long long)b * hs.capB + e];
      ln = hs.slot_len[gs];
      sc = hs.B_ls[(long long)b * hs.capB + e];
      src = hs.slot_tok + gs * hs.U_cap;
    }
    for (int q = threadIdx.x; q < hs.U_cap; q += blockDim.x) dst[q] = (q < ln) ? src[q] : -1;
    if (threadIdx.x == 0) { out_lens[b * hs.N + i] = ln; out_scores[b * hs.N + i] = sc; }
  }
  if (threadIdx.x == 0) out_status[b] = hs.status[b];
}

}  // namespace

void launch_hyp_init(const HypState& hs, const int* lengths, int B, int T, cudaStream_t st) {
  if (B > 0) hyp_init_kernel<<<B, kThreads, 0, st>>>(hs, lengths, T);
}
void launch_hyp_step(const HypState& hs, int B, cudaStream_t st) {
  if (B <= 0) return;
  const int tok_cap = hs.N * hs.U_cap * 4 <= kTokStageMax ? hs.U_cap : 0;
  launch_pdl(hyp_step_kernel, dim3(B), dim3(hs.dnb_sel ? 2 * kStepThreads : kStepThreads), (size_t)hs.N * tok_cap * 4, st, hs, tok_cap);
}
void launch_compact(const HypState& hs, int B, int T, cudaStream_t st) {
  launch_pdl(compact_kernel, dim3(1), dim3(1024), 0, st, hs, B, T);
}
void launch_stream_rows(const HypState& hs, const int* chunk_lens, int B, int Tc, int max_T, int dump_row,
                        int* oidx, cudaStream_t st) {
  const int n = B * Tc;
  if (n > 0) stream_rows_kernel<<<(n + 255) / 256, 256, 0, st>>>(hs, chunk_lens, B, Tc, max_T, dump_row, oidx);
}
void launch_stream_advance(const HypState& hs, const int* chunk_lens, int B, int max_T, int closing,
                           cudaStream_t st) {
  if (B > 0) stream_advance_kernel<<<B, kThreads, 0, st>>>(hs, chunk_lens, max_T, closing);
}
void launch_finish(const HypState& hs, int B, int* out_tokens, int* out_lens, double* out_scores,
                   int* out_status, cudaStream_t st) {
  if (B > 0) finish_kernel<<<B, kThreads, 0, st>>>(hs, out_tokens, out_lens, out_scores, out_status);
}
}  // namespace tw
