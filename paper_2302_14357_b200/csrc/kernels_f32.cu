// fp32 (TW_MODE_F32) stage kernels: SIMT GEMM, joiner contraction, log-softmax, Eq. 3-7.
// This is the accuracy path: plain FFMA accumulation and libm tanhf/expf/logf, no fast-math.
#include <atomic>

#include "topn.cuh"
#include "bf16_path.cuh"
#include "sm100.cuh"
#include "tw_internal.cuh"

namespace tw {

namespace {

// ---------------------------------------------------------------------------------------------
// SIMT fp32 GEMM.  The rows of a decode step are few (tens to hundreds) and K is long, so a CTA owns a short, wide tile
// (16 rows x 256 columns) and its eight warps split every K block between them: each accumulates the whole tile over its
// eighth of K, and the partial tiles are summed in a fixed order at the end.  Where such tiles leave SMs idle, a cluster
// of two or four CTAs splits K once more and sums over distributed shared memory.  A lane holds 16 x NJ outputs: shared
// memory delivers one register per lane and cycle to the whole SM, so the 16 + 8 operand registers of a k take 96 of
// the 128 cycles in which the four schedulers issue its FMAs (with 8 x 8 outputs it would be 64 of 64).  The 64-column
// tiles (NJ = 2) are for narrow matrices.
// Only eight warps fit beside that many accumulators, so nothing but FMAs and operand reads may take issue slots: the
// weights arrive by TMA (128-byte swizzle: the 16-byte reads along K of eight neighbouring rows hit distinct banks), the
// rows of A by bulk copies, four blocks of 32 ahead, each block sent for by another warp, and the warps meet on the
// ring's mbarriers only.  The weights of the first blocks are asked for before the wait for the kernel ahead.
// Measured: 27 us for 112 x 2560 x 1280 and 26 us for 435 x 1024 x 640 (77 and 59 us with 64 x 64 tiles, 4 x 4 outputs a
// thread, whole K), 27 and 22 TFLOP/s, where register-only FFMA loops reach 51 of the nominal 74 on a B200.  By FFMA issue
// alone the share of one CTA (16 x 256 x 640) would take 15 us at that rate; the rest is the way of the first blocks
// into shared memory, the sum over warps and CTAs, and the SMs that the 140 and 112 CTAs leave idle.
constexpr int TM = 16, BK = 32, kStagesF = 6, kAhead = kStagesF - 2, kWarpsF = 8, kThreadsF = 32 * kWarpsF;
template <int NJ> struct F32Smem {
  static constexpr size_t kB = (size_t)32 * NJ * BK * 4, kA = (size_t)TM * BK * 4;
  static constexpr size_t kOps = kStagesF * (kB + kA), kRed = (size_t)kWarpsF * TM * 32 * NJ * 4;
  static constexpr size_t kTotal = (kOps > kRed ? kOps : kRed) + 1024 + 2 * kStagesF * 8;
};

struct GemmParams {
  GemmOperand op[2];
  GemmOut out;
  const int* M_dev;
  int M_scale;        // rows = *M_dev * M_scale
  int M_max, N;
  // joiner mode
  JoinerRows jr;
  const float* W_out;
  const float* b_out;
  float* z;
  int* err;           // raised by a wait that gave up
};

__device__ __forceinline__ float4 load4(const float* p, int k, int K) {
  if (k + 3 < K && ((reinterpret_cast<uintptr_t>(p + k) & 15) == 0)) return *reinterpret_cast<const float4*>(p + k);
  float v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = (k + i < K) ? p[k + i] : 0.f;
  return make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ float sigmoidf_acc(float x) { return 1.f / (1.f + expf(-x)); }
__device__ __forceinline__ float act_f32(float x, int act) { return act == TW_ACT_RELU ? fmaxf(x, 0.f) : tanhf(x); }

// MODE 0: plain / gathered rows, one or two operand pairs.  MODE 1: joiner rows, A = act(E + Pp) formed on the way.
// VEC: K is a multiple of 4 and every row starts on a 16-byte boundary (TMA and bulk copies); otherwise the warps copy
// the operands element by element.
template <int MODE, int NJ, bool VEC>
__global__ void __launch_bounds__(kThreadsF, 1)
gemm_f32_kernel(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1, GemmParams p) {
  using namespace sm100;
  using Sm = F32Smem<NJ>;
  extern __shared__ uint8_t smem_raw[];
  constexpr int BN = 32 * NJ;                                // lane: all 16 rows, columns lane + 32 j
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  float* sm_f32 = reinterpret_cast<float*>(smem);            // the partial tiles, once the operands are done with
  uint8_t* sB = smem;                                        // [kStagesF][BN][BK], swizzled
  uint8_t* sA = smem + kStagesF * Sm::kB;                    // [kStagesF][TM][BK]
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (Sm::kOps > Sm::kRed ? Sm::kOps : Sm::kRed));
  uint64_t* empty = full + kStagesF;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int N = (MODE == 1) ? p.jr.V : p.N;
  const int n_tiles = (N + BN - 1) / BN;                     // row tiles by column tiles, all on grid.x (grid.y would end at 65535 row tiles)
  const int m0 = (int)blockIdx.x / n_tiles * TM, n0 = (int)blockIdx.x % n_tiles * BN;
  const int K0 = (MODE == 1) ? p.jr.J : p.op[0].K, K1 = (MODE == 1) ? 0 : p.op[1].K;
  const int nb0 = (K0 + BK - 1) / BK, nb_all = nb0 + (K1 + BK - 1) / BK;
  const int split = gridDim.z, part = blockIdx.z;            // the CTAs of a cluster share K
  const int b_lo = nb_all * part / split, nb = nb_all * (part + 1) / split - b_lo;
  constexpr bool kBulkA = VEC && MODE == 0;

  if (tid == 0) {
    for (int s = 0; s < kStagesF; ++s) { mbar_init(&full[s], VEC ? (MODE == 0 ? 2 : 1 + kWarpsF) : kWarpsF); mbar_init(&empty[s], kWarpsF); }
    fence_barrier_init();
  }
  fence_proxy_async_smem();
  __syncthreads();
  auto send_B = [&](int i) {               // one thread: the weights of block i
    const int blk = b_lo + i, s = i % kStagesF;
    mbar_arrive_expect(&full[s], (uint32_t)Sm::kB);
    tma_load_2d(sB + s * Sm::kB, blk < nb0 ? &tm0 : &tm1, &full[s], (blk < nb0 ? blk : blk - nb0) * BK, n0);
  };
  const int pre = nb < kAhead ? nb : kAhead;
  if (VEC && tid == 0) for (int i = 0; i < pre; ++i) send_B(i);   // constant weights: ahead of the wait
  pdl_wait();
  pdl_trigger();
  int M;
  if (MODE == 1) M = (p.jr.R_dev ? *p.jr.R_dev : p.jr.R_max) * p.jr.S;
  else M = p.M_dev ? *p.M_dev * p.M_scale : p.M_max;
  if (m0 >= M) {                           // no rows here: only the copies already under way have to be waited for
    if (VEC && tid == 0)
      for (int i = 0; i < pre; ++i) {
        for (int c = 1; c < (MODE == 0 ? 2 : 1 + kWarpsF); ++c) mbar_arrive(&full[i]);
        mbar_wait(&full[i], 0, p.err);
      }
    return;
  }

  const int lrow = kBulkA ? (lane & 15) : (tid >> 4);        // the row of A this thread looks after
  const float* arow = nullptr;
  const float* prow = nullptr;             // MODE 0: the row of the second operand; MODE 1: the Pp row
  if (m0 + lrow < M) {
    const int m = m0 + lrow;
    if (MODE == 1) {
      const int r = m / p.jr.S, t = m - r * p.jr.S;
      const int sl = p.jr.row_slen ? p.jr.row_slen[r] : p.jr.S;
      if (t < sl) {
        arow = p.jr.E + (long long)(p.jr.row_e0[r] + t) * K0;
        prow = p.jr.Pp + (long long)(p.jr.row_p ? p.jr.row_p[r] : r) * K0;
      }
    } else {
      arow = p.op[0].A + (long long)(p.op[0].idx ? p.op[0].idx[m] : m) * p.op[0].ldA;
      if (K1 > 0) prow = p.op[1].A + (long long)(p.op[1].idx ? p.op[1].idx[m] : m) * p.op[1].ldA;
    }
  }
  // the rows of A of block i (bulk copies: one warp; else: the whole CTA forms them, and copies B if it has to)
  auto send_A = [&](int i) {
    const int blk = b_lo + i, s = i % kStagesF;
    const bool second = blk >= nb0;
    const int k = (second ? blk - nb0 : blk) * BK, kn = min(BK, (second ? K1 : K0) - k);
    if (kn < BK) {      // short last block: the rest meets zeros of B, and an infinity that an earlier block left there would make them NaN
      if (lane < TM)
        for (int x = kn; x < BK; x += 4) *reinterpret_cast<float4*>(sA + s * Sm::kA + (lane * BK + x) * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
      fence_proxy_async_smem();
      __syncwarp();
    }
    if (lane == 0) mbar_arrive_expect(&full[s], (uint32_t)(min(TM, M - m0) * kn * 4));
    __syncwarp();
    if (lane < TM && arow != nullptr)
      bulk_load(sA + s * Sm::kA + lane * (BK * 4), (second ? prow : arow) + k, (uint32_t)kn * 4u, &full[s]);
  };
  auto form = [&](int i) {
    const int blk = b_lo + i, s = i % kStagesF;
    const bool second = blk >= nb0;
    const int k0 = (second ? blk - nb0 : blk) * BK, K = second ? K1 : K0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {          // two elements of A per thread
      const int k = k0 + (tid & 15) * 2 + u;
      float v = 0.f;
      if (arow != nullptr && k < K) v = MODE == 1 ? act_f32(arow[k] + prow[k], p.jr.act) : (second ? prow : arow)[k];
      reinterpret_cast<float*>(sA + s * Sm::kA)[lrow * BK + (tid & 15) * 2 + u] = v;
    }
    if (!VEC) {
      const float* Bm = (MODE == 1) ? p.W_out : (second ? p.op[1].B : p.op[0].B);
      const long long ld = (MODE == 1) ? p.jr.J : (second ? p.op[1].ldB : p.op[0].ldB);
      for (int e = tid; e < BN * BK; e += kThreadsF) {
        const int r = e / BK, kk = e % BK;
        const float v = (n0 + r < N && k0 + kk < K) ? Bm[(n0 + r) * ld + k0 + kk] : 0.f;
        reinterpret_cast<float*>(sB + s * Sm::kB)[r * BK + (((kk >> 2) ^ (r & 7)) << 2) + (kk & 3)] = v;
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&full[s]);
  };
  for (int i = 0; i < pre; ++i) {
    if (!kBulkA) form(i);
    else if (warp == i % kWarpsF) send_A(i);
  }

  float acc[TM][NJ];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0.f;
  bool ok = true;
  uint32_t st = 0, ph = 0;                 // stage and phase of block blk
#pragma unroll 1
  for (int blk = 0; blk < nb && ok; ++blk) {
    const int nxt = blk + kAhead;
    if (nxt < nb && (!kBulkA || warp == nxt % kWarpsF)) {
      const int use = nxt / kStagesF;
      if (use > 0) ok = mbar_wait(&empty[nxt % kStagesF], (use - 1) & 1, p.err);
      if (!ok) break;
      if (VEC && lane == 0 && (kBulkA || warp == 0)) send_B(nxt);
      if (kBulkA) send_A(nxt); else form(nxt);
    }
    ok = mbar_wait(&full[st], ph, p.err);
    if (!ok) break;
    const float* a = reinterpret_cast<const float*>(sA + st * Sm::kA) + warp * 4;
    const uint8_t* b = sB + st * Sm::kB + lane * (BK * 4) + ((warp ^ (lane & 7)) << 4);
    float4 av[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4*>(a + i * BK);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 bv = *reinterpret_cast<const float4*>(b + j * (32 * BK * 4));
#pragma unroll
      for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(av[i].x, bv.x, acc[i][j]);
#pragma unroll
      for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(av[i].y, bv.y, acc[i][j]);
#pragma unroll
      for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(av[i].z, bv.z, acc[i][j]);
#pragma unroll
      for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(av[i].w, bv.w, acc[i][j]);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[st]);
    if (++st == kStagesF) { st = 0; ph ^= 1; }
  }

  // ---- the warps' partial tiles, summed in the order of K; [kWarpsF][TM][BN] in the operands' place
  settle_copies(ok);
  __syncthreads();                         // every block has been waited for: nothing is on its way into shared memory
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) sm_f32[(warp * TM + i) * BN + lane + 32 * j] = acc[i][j];
  __syncthreads();
  auto part_sum = [&](int at) {
    float4 v = *reinterpret_cast<const float4*>(&sm_f32[at]);
#pragma unroll
    for (int w = 1; w < kWarpsF; ++w) {
      const float4 u = *reinterpret_cast<const float4*>(&sm_f32[w * TM * BN + at]);
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    return v;
  };
  if (split > 1) {                         // this CTA's sums in place; each CTA then finishes its share of the tile
#pragma unroll
    for (int i = 0; i < NJ / 2; ++i) {
      const int at = (tid + i * kThreadsF) * 4;
      *reinterpret_cast<float4*>(&sm_f32[at]) = part_sum(at);
    }
    sm100::cluster_sync_all();
  }
  const int chunks = TM * BN / 4 / split;  // of four columns
  for (int i = tid; i < chunks; i += kThreadsF) {
    const int c = part * chunks + i, rr = c / (BN / 4), cc = (c - rr * (BN / 4)) * 4;
    const int m = m0 + rr, n = n0 + cc;
    if (m >= M || n >= N) continue;
    float4 v;
    if (split == 1) {
      v = part_sum(c * 4);
    } else {
      v = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int q = 0; q < split; ++q) {
        const float4 u = sm100::ld_cluster_f32x4(sm100::map_to_cta(sm100::smem_u32(&sm_f32[c * 4]), (uint32_t)q));
        v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
      }
    }
    if (MODE == 0 && p.out.lstm.hc_out != nullptr) {           // the four gates of hidden unit n / 4
      const LstmF32& q = p.out.lstm;
      const float4 b4 = *reinterpret_cast<const float4*>(p.out.bias + n);
      const long long pin = (q.idx_in ? q.idx_in[m] : m) * q.stride + q.lo + (n >> 2), pout = (q.idx_out ? q.idx_out[m] : m) * q.stride + q.lo + (n >> 2);
      const float cn = sigmoidf_acc(v.y + b4.y) * q.hc_in[pin + q.Hd] + sigmoidf_acc(v.x + b4.x) * tanhf(v.z + b4.z);
      q.hc_out[pout] = sigmoidf_acc(v.w + b4.w) * tanhf(cn);
      q.hc_out[pout + q.Hd] = cn;
      continue;
    }
    float* crow;
    const float* bias;
    if (MODE == 1) {
      const int r = m / p.jr.S, t = m - r * p.jr.S;
      const int sl = p.jr.row_slen ? p.jr.row_slen[r] : p.jr.S;
      if (t >= sl) continue;
      crow = p.z + (long long)m * N;
      bias = p.b_out;
    } else {
      crow = p.out.C + (long long)(p.out.oidx ? p.out.oidx[m] : m) * p.out.ldC;
      bias = p.out.bias;
    }
    if (n + 3 < N && ((reinterpret_cast<uintptr_t>(crow + n) & 15) == 0)) {
      if (bias) { v.x += bias[n]; v.y += bias[n + 1]; v.z += bias[n + 2]; v.w += bias[n + 3]; }
      *reinterpret_cast<float4*>(crow + n) = v;
    } else {
      const float o[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) if (n + j < N) crow[n + j] = o[j] + (bias ? bias[n + j] : 0.f);
    }
  }
  if (split > 1) sm100::cluster_sync_all();          // nobody leaves while a cluster mate still reads its sums
}

// the joiner's operand act(E + Pp) of every (row, frame) as float32 [R S, J]: a joiner with many column tiles forms it
// once instead of once per column tile (rows of padding frames are left as they are: nothing reads their products)
__global__ void __launch_bounds__(256) joiner_A_f32_kernel(JoinerRows jr, float* __restrict__ A) {
  pdl_wait();
  pdl_trigger();
  const int M = (jr.R_dev ? *jr.R_dev : jr.R_max) * jr.S;
  const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;      // a warp per row
  if (m >= M) return;
  const int r = m / jr.S, t = m - r * jr.S;
  if (t >= (jr.row_slen ? jr.row_slen[r] : jr.S)) return;
  const float* e = jr.E + (long long)(jr.row_e0[r] + t) * jr.J;
  const float* q = jr.Pp + (long long)(jr.row_p ? jr.row_p[r] : r) * jr.J;
  float* dst = A + (long long)m * jr.J;
  for (int k = lane * 4; k < jr.J; k += 128) {
    const float4 ev = load4(e, k, jr.J), pv = load4(q, k, jr.J);
    const float v[4] = {act_f32(ev.x + pv.x, jr.act), act_f32(ev.y + pv.y, jr.act), act_f32(ev.z + pv.z, jr.act), act_f32(ev.w + pv.w, jr.act)};
    if (k + 3 < jr.J && ((reinterpret_cast<uintptr_t>(dst + k) & 15) == 0)) {
      *reinterpret_cast<float4*>(dst + k) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
      for (int i = 0; i < 4 && k + i < jr.J; ++i) dst[k + i] = v[i];
    }
  }
}

// C[m, n] = sum_k A[m, k] B[n, k] + bias[n] for the tables that tw_init builds from the weights: every product is
// accumulated over k in ascending order by one thread, so that a table's values do not depend on how a tile is split
// (a table feeds every later step; the decode-time kernel above is free to choose its split).  64 x 64 tiles, 4 x 4 a thread.
__global__ void __launch_bounds__(256) gemm_f32_table_kernel(const float* __restrict__ A, const float* __restrict__ B, const float* __restrict__ bias,
                                                             float* __restrict__ C, int M, int N, int K) {
  __shared__ __align__(16) float As[16][68], Bs[16][68];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 16) {
    for (int i = tid; i < 64 * 16; i += 256) {
      const int r = i >> 4, k = i & 15;
      As[k][r] = (m0 + r < M && k0 + k < K) ? A[(long long)(m0 + r) * K + k0 + k] : 0.f;
      Bs[k][r] = (n0 + r < N && k0 + k < K) ? B[(long long)(n0 + r) * K + k0 + k] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[k][ty * 4]), b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
      const float aa[4] = {a.x, a.y, a.z, a.w}, bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(aa[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty * 4 + i, n = n0 + tx * 4 + j;
      if (m < M && n < N) C[(long long)m * N + n] = acc[i][j] + (bias ? bias[n] : 0.f);
    }
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(256) log_softmax_kernel(JoinerRows jr, int blank, float* z) {
  __shared__ float red[8];
  __shared__ float bcast;
  const int R = jr.R_dev ? *jr.R_dev : jr.R_max;
  const int m = blockIdx.x;
  const int r = m / jr.S, t = m - r * jr.S;
  if (r >= R) return;
  float* row = z + (long long)m * jr.V;
  const int sl = jr.row_slen ? jr.row_slen[r] : jr.S;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (t >= sl) {
    for (int k = tid; k < jr.V; k += 256) row[k] = (k == blank) ? 0.f : -INFINITY;
    return;
  }
  const bool hat = jr.hat != 0;
  float mx = -INFINITY;
  for (int k = tid; k < jr.V; k += 256) if (!hat || k != blank) mx = fmaxf(mx, row[k]);
  mx = warp_max(mx);
  if (lane == 0) red[w] = mx;
  __syncthreads();
  if (tid == 0) { float v = red[0]; for (int i = 1; i < 8; ++i) v = fmaxf(v, red[i]); bcast = v; }
  __syncthreads();
  mx = bcast;
  float s = 0.f;
  for (int k = tid; k < jr.V; k += 256) if (!hat || k != blank) s += expf(row[k] - mx);
  s = warp_sum(s);
  __syncthreads();
  if (lane == 0) red[w] = s;
  __syncthreads();
  if (tid == 0) { float v = 0.f; for (int i = 0; i < 8; ++i) v += red[i]; bcast = mx + logf(v); }
  __syncthreads();
  const float lse = bcast;
  if (!hat) {
    for (int k = tid; k < jr.V; k += 256) row[k] = row[k] - lse;
    return;
  }
  // factorised output: log sigmoid(zb), log(1 - sigmoid(zb)) without cancellation
  const float zb = row[blank];
  __syncthreads();                               // every thread has read the blank logit before it is overwritten
  const float sp = (zb >= 0.f) ? log1pf(expf(-zb)) : -zb + log1pf(expf(zb));     // softplus(-zb)
  const float log_pb = -sp, log_rest = -sp - zb;
  const bool skip = log_pb > jr.log_tau;         // blank thresholding: the label part is left out
  if (skip && tid == 0 && jr.skipped != nullptr) atomicAdd(jr.skipped, 1ull);
  for (int k = tid; k < jr.V; k += 256)
    row[k] = (k == blank) ? log_pb : (skip ? -INFINITY : row[k] - lse + log_rest);
}

// One CTA per hypothesis row.  Eq. 3-7 through the occupancy recursion
//   la[1] = ld_old[1];  la[t+1] = logaddexp(la[t] + lb[t], ld_old[t+1]),  lb[t] = log J(t, blank)
//   log d(k, t) = la[t] + log J(t, k);  delta_nb(k) = sum_t d(k, t);  delta_phi = la[S'] + lb[S'].
__global__ void __launch_bounds__(256) expand_f32_kernel(const float* __restrict__ logp,
                                                         const float* __restrict__ ld_old,
                                                         const int* row_slen, const int* R_dev,
                                                         int R_max, int S, int V, int blank,
                                                         float* ldphi, float* ldnb, float* la_out,
                                                         double* ldphi_d, double* la_d, CandOut cand, StepWords words, const int* err) {
  update_step_words(words);
  __shared__ float la[kMaxSeg];
  __shared__ float s_wv[8][kMaxBeam];
  __shared__ int s_wk[8][kMaxBeam];
  __shared__ int s_wn[8];
  const int R = R_dev ? *R_dev : R_max;
  const int r = blockIdx.x;
  if (r >= R) return;
  const int sl = row_slen ? min(max(row_slen[r], 0), S) : S;   // a caller's value outside [0, S] must not index past the row
  const float* lp = logp + (long long)r * S * V;
  if (threadIdx.x == 0) {
    // the recursion is S steps long and its values grow to hundreds of nats: carry it in float64
    double a = (double)ld_old[(long long)r * S];
    double phi = -INFINITY;
    for (int t = 0; t < sl; ++t) {
      la[t] = (float)a;
      if (la_d) la_d[(long long)r * S + t] = a;
      const double nxt = a + (double)lp[(long long)t * V + blank];   // -inf + finite stays -inf
      if (t + 1 < sl) a = logaddexp_d(nxt, (double)ld_old[(long long)r * S + t + 1]);
      else phi = nxt;
    }
    for (int t = (sl > 0 ? sl : 0); t < S; ++t) {
      la[t] = -INFINITY;
      if (la_d) la_d[(long long)r * S + t] = -INFINITY;
    }
    ldphi[r] = (err != nullptr && *err != 0) ? NAN : (float)phi;
    if (ldphi_d) ldphi_d[r] = phi;
  }
  __syncthreads();
  if (threadIdx.x < S) la_out[(long long)r * S + threadIdx.x] = la[threadIdx.x];
  TopList best;
  best.init();
  float admit = -INFINITY;
  for (int k = threadIdx.x; k < V; k += blockDim.x) {
    float out = -INFINITY;
    if (k != blank) {
      float mx = -INFINITY;
      for (int t = 0; t < sl; ++t) mx = fmaxf(mx, la[t] + lp[(long long)t * V + k]);
      if (mx > -INFINITY) {
        float s = 0.f;
        for (int t = 0; t < sl; ++t) s += expf(la[t] + lp[(long long)t * V + k] - mx);
        out = mx + logf(s);
      }
    }
    if (ldnb) ldnb[(long long)r * V + k] = out;
    if (cand.n && out > admit) {          // the blank column is -inf and never a candidate
      best.insert(out, k);
      admit = best.nth(cand.N);
    }
  }
  if (cand.n == nullptr) return;
  // ChooseNBestExpansions, first stage: this row's N best non-blank tokens
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wn = warp_merge_lists(best, cand.N, s_wv[warp], s_wk[warp]);
  if (lane == 0) s_wn[warp] = wn;
  __syncthreads();
  if (warp == 0) {
    int pos = 0;
    const int mine = lane < 8 ? s_wn[lane] : 0;
    int cnt = 0;
    for (int j = 0; j < cand.N; ++j) {
      float bv = (pos < mine) ? s_wv[lane][pos] : -INFINITY;
      int bk = (pos < mine) ? s_wk[lane][pos] : 0x7fffffff;
      int bl = lane;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
        if (cand_better(ov, ok, bv, bk)) { bv = ov; bk = ok; bl = ol; }
      }
      bv = __shfl_sync(0xffffffffu, bv, 0); bk = __shfl_sync(0xffffffffu, bk, 0); bl = __shfl_sync(0xffffffffu, bl, 0);
      if (bv == -INFINITY) break;
      if (lane == 0) { cand.v[(long long)r * kMaxBeam + j] = bv; cand.k[(long long)r * kMaxBeam + j] = bk; }
      if (lane == bl) ++pos;
      ++cnt;
    }
    if (lane == 0) cand.n[r] = cnt;
  }
}

__global__ void permute_rows_f32_kernel(const float* __restrict__ src, const int* __restrict__ perm, long long rows, int cols, float* __restrict__ dst) {
  const float* s = src + (long long)perm[blockIdx.x] * cols;
  for (int c = threadIdx.x; c < cols; c += blockDim.x) dst[(long long)blockIdx.x * cols + c] = s[c];
}

__global__ void rows_from_groups_kernel(const int* row_group, const int* seg_len, int R, int G, int S,
                                        int* row_e0, int* row_slen, int* clear) {
  pdl_wait();
  pdl_trigger();
  if (clear != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  int g = row_group[r];
  if (g < 0 || g >= G) { row_e0[r] = 0; row_slen[r] = 0; return; }   // no such segment: an empty row, nothing is read for it
  row_e0[r] = g * S;
  int sl = seg_len ? seg_len[g] : S;
  row_slen[r] = sl < 0 ? 0 : (sl > S ? S : sl);
}

}  // namespace

namespace {
bool row_aligned(const float* base, long long ld) { return (reinterpret_cast<uintptr_t>(base) & 15) == 0 && (ld & 3) == 0; }

// false: no tensor map of the weights could be made, nothing was launched (a launch that fails is left to cudaGetLastError)
template <int MODE, int NJ, bool VEC>
bool launch_gemm_one(const GemmParams& p, long long M_max, int N, cudaStream_t st) {
  static std::atomic<unsigned long long> ready{0};           // devices whose copy of the kernel has its shared-memory limit raised
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (dev > 63 || !(ready.load(std::memory_order_acquire) & bit)) {
    cudaFuncSetAttribute(gemm_f32_kernel<MODE, NJ, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F32Smem<NJ>::kTotal);
    ready.fetch_or(bit, std::memory_order_release);
  }
  const long long mt = (M_max + TM - 1) / TM, nt = (N + 32 * NJ - 1) / (32 * NJ);
  // K shared by two or four CTAs while the tiles of the largest row count leave SMs idle (a step mostly has fewer rows
  // than its maximum) and every CTA keeps four blocks of K
  const int nb = MODE == 1 ? (p.jr.J + BK - 1) / BK : (p.op[0].K + BK - 1) / BK + (p.op[1].K + BK - 1) / BK;
  const unsigned split = (mt * nt <= 40 && nb >= 16) ? 4 : ((mt * nt <= 110 && nb >= 8) ? 2 : 1);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nt * mt), 1, split); cfg.blockDim = dim3(kThreadsF);
  cfg.dynamicSmemBytes = F32Smem<NJ>::kTotal; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = split;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = g_pdl_on ? 2 : 1;
  CUtensorMap tm0 = {}, tm1 = {};
  if (VEC) {
    const GemmOperand b0 = MODE == 1 ? GemmOperand{nullptr, nullptr, 0, p.W_out, p.jr.J, p.jr.J} : p.op[0];
    if (make_tmap_f32(&tm0, b0.B, N, b0.K, b0.ldB, 32 * NJ) != TW_OK) return false;
    if (p.op[1].K > 0 && make_tmap_f32(&tm1, p.op[1].B, N, p.op[1].K, p.op[1].ldB, 32 * NJ) != TW_OK) return false;
  }
  cudaLaunchKernelEx(&cfg, gemm_f32_kernel<MODE, NJ, VEC>, tm0, tm1, p);
  return true;
}
template <int MODE>
void launch_gemm_tiles(const GemmParams& p, bool vec, long long M_max, int N, cudaStream_t st) {
  if (N <= 128) {
    if (!vec || !launch_gemm_one<MODE, 2, true>(p, M_max, N, st)) launch_gemm_one<MODE, 2, false>(p, M_max, N, st);
  } else {
    if (!vec || !launch_gemm_one<MODE, 8, true>(p, M_max, N, st)) launch_gemm_one<MODE, 8, false>(p, M_max, N, st);
  }
}
}  // namespace

void launch_gemm_f32(const GemmOperand& op1, const GemmOperand& op2, const GemmOut& out,
                     const int* M_dev, int M_max, int N, cudaStream_t st) {
  if (M_max <= 0 || N <= 0) return;
  GemmParams p{};
  p.op[0] = op1; p.op[1] = op2; p.out = out; p.M_dev = M_dev; p.M_scale = 1; p.M_max = M_max; p.N = N; p.err = out.err;
  auto ok = [](const GemmOperand& o) { return o.K == 0 || ((o.K & 3) == 0 && row_aligned(o.A, o.ldA) && row_aligned(o.B, o.ldB)); };
  launch_gemm_tiles<0>(p, ok(op1) && ok(op2), M_max, N, st);
}

void launch_gemm_f32_table(const float* A, const float* B, const float* bias, float* C, int M, int N, int K, cudaStream_t st) {
  gemm_f32_table_kernel<<<dim3((N + 63) / 64, (M + 63) / 64), 256, 0, st>>>(A, B, bias, C, M, N, K);
}

int launch_joiner_f32(const JoinerRows& rows, const float* W_out, const float* b_out, float* z, float* A_buf, int* err, cudaStream_t st) {
  if (rows.R_max <= 0) return 0;
  GemmParams p{};
  p.err = err;
  const long long M_max = (long long)rows.R_max * rows.S;
  // The operand (a tanhf per element) formed anew in every column tile, or once in a pass of its own, which costs a launch and a
  // round trip through L2: 1 to 2 us.  The pass from one 16 x 64 output tile per SM on, which is a quarter of that many CTAs
  // for V > 128.  Measured, without / with it, tw_joiner_expand: V = 1024, J = 640: 129 GEMM rows 30.2 / 30.8 us, 192 26.8 /
  // 27.6, 321 44.6 / 43.1, 768 70 / 64; V = 501: 480 27.5 / 28.0, 768 45.3 / 43.6; V = 4096, J = 1024: 33 42.5 / 42.8, 81
  // 67.8 / 64.4; V = 128: 1536 13.6 / 12.1.
  const long long tiles = (M_max + TM - 1) / TM * ((rows.V + 63) / 64);
  const bool vec = (rows.J & 3) == 0 && row_aligned(W_out, rows.J);
  if (A_buf != nullptr && tiles > sm_count()) {
    launch_pdl(joiner_A_f32_kernel, dim3((unsigned)((M_max + 7) / 8)), dim3(256), 0, st, rows, A_buf);
    p.op[0] = GemmOperand{A_buf, nullptr, rows.J, W_out, rows.J, rows.J};
    p.out = GemmOut{z, nullptr, rows.V, b_out};
    p.M_dev = rows.R_dev; p.M_scale = rows.S; p.M_max = (int)M_max; p.N = rows.V;
    launch_gemm_tiles<0>(p, vec, M_max, rows.V, st);
    return 2;
  }
  p.jr = rows; p.W_out = W_out; p.b_out = b_out; p.z = z;
  launch_gemm_tiles<1>(p, vec, M_max, rows.V, st);
  return 1;
}

void launch_log_softmax(const JoinerRows& rows, int blank, float* z, cudaStream_t st) {
  if (rows.R_max <= 0) return;
  log_softmax_kernel<<<rows.R_max * rows.S, 256, 0, st>>>(rows, blank, z);
}

void launch_expand_f32(const float* logp, const float* ld_old, const int* row_slen, const int* R_dev,
                       int R_max, int S, int V, int blank, float* ldphi, float* ldnb, float* la,
                       double* ldphi_d, double* la_d, const CandOut& cand, cudaStream_t st, const StepWords& words, const int* err) {
  if (R_max <= 0) return;
  expand_f32_kernel<<<R_max, 256, 0, st>>>(logp, ld_old, row_slen, R_dev, R_max, S, V, blank, ldphi,
                                           ldnb, la, ldphi_d, la_d, cand, words, err);
}

void launch_permute_rows_f32(const float* src, const int* perm, long long rows, int cols, float* dst, cudaStream_t st) {
  permute_rows_f32_kernel<<<(unsigned)rows, 256, 0, st>>>(src, perm, rows, cols, dst);
}

void launch_rows_from_groups(const int* row_group, const int* seg_len, int R, int G, int S, int* row_e0,
                             int* row_slen, int* clear, cudaStream_t st) {
  if (R <= 0) return;
  launch_pdl(rows_from_groups_kernel, dim3((R + 255) / 256), dim3(256), 0, st, row_group, seg_len, R, G, S, row_e0, row_slen, clear);
}

}  // namespace tw
