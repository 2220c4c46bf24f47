// The joiner's A operand act(E + Pp) as bf16, and where a row of it lies in the fused joiner kernel's tile layout.
#pragma once
#include "bf16_path.cuh"

namespace tw {

__device__ __forceinline__ float tanh_fast2(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float act2(float x, int act) { return act == TW_ACT_RELU ? fmaxf(x, 0.f) : tanh_fast2(x); }

// eight operand values act(e + p) as bf16
__device__ __forceinline__ uint4 act8(const float e[8], const float p[8], int act) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(act2(e[2 * i] + p[2 * i], act), act2(e[2 * i + 1] + p[2 * i + 1], act));
    w[i] = *reinterpret_cast<const uint32_t*>(&v);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint4 act8(const float4& e0, const float4& e1, const float4& p0, const float4& p1, int act) {
  const float e[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w}, p[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
  return act8(e, p, act);
}

// Operand row of frame t of joiner row r: a tile of 128 rows holds 4 (32 / S) hypotheses, the S frames of one adjacent
__device__ __forceinline__ long long operand_row(int r, int t, int S) {
  const int HPW = 32 / S, HPT = 4 * HPW;
  const int tile = r / HPT, hw = r - tile * HPT, q = hw / HPW;
  return (long long)tile * 128 + q * 32 + (hw - q * HPW) * S + t;
}

}  // namespace tw
