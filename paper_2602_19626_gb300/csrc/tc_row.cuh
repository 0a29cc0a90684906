// Whole-row arithmetic of the tensor-core path shared by the kernels that
// make a GEMM operand or finish a GEMM's rows: the RMSNorm of a row held by
// one warp, the E4M3 row scale and the SwiGLU of adjacent accumulator lanes.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "internal.h"

namespace nc {

// SiLU of the tensor-core path: a * (1 / (1 + e^-a)) with the fast exponential
// and a correctly rounded reciprocal (1 / inf = 0 for very negative a).  The
// decode step and the prefill forward run this same code.
__device__ __forceinline__ float silu_tc(float a) { return a * __frcp_rn(1.0f + __expf(-a)); }

// SwiGLU of two adjacent batch columns n, n + 1: rows 2j (gate) and 2j + 1
// (up) sit on adjacent lanes; the even lane computes h_j of column n, the odd
// lane h_j of column n + 1, each from one exchanged value; y0, y1 already
// carry the FP8 scales.  mine: the lane's row r is one of the M.
__device__ __forceinline__ void swiglu_pair(bool mine, int M, float* h_out, void* h16, int r, int n, int B, float y0, float y1) {
  const bool odd = r & 1;
  const float got = __shfl_xor_sync(0xffffffffu, odd ? y0 : y1, 1);
  const float gate = odd ? got : y0, up = odd ? y1 : got;
  const int col = n + (odd ? 1 : 0);
  if (mine && col < B) {
    const float h = silu_tc(gate) * up;
    if (h16)
      static_cast<__nv_bfloat16*>(h16)[(size_t)col * (M / 2) + (r >> 1)] = __float2bfloat16_rn(h);
    else
      h_out[(size_t)col * (M / 2) + (r >> 1)] = h;
  }
}

// A row of up to 32 kRowVals columns over one warp, column lane + 32 i in
// value i.
constexpr int kRowVals = 20;                 // 640 columns: the full model's 576 in whole 128-byte E4M3
                                             // blocks; wider rows take the kernels of a CTA per row

__device__ __forceinline__ void load_row(const float* xr, int cols, int lane, float (&x)[kRowVals]) {
#pragma unroll
  for (int i = 0; i < kRowVals; ++i) x[i] = lane + 32 * i < cols ? __ldcg(xr + lane + 32 * i) : 0.f;
}
__device__ __forceinline__ void load_gain(const float* gain, int cols, int lane, float (&g)[kRowVals]) {
#pragma unroll
  for (int i = 0; i < kRowVals; ++i) g[i] = lane + 32 * i < cols ? __ldg(gain + lane + 32 * i) : 0.f;
}

// x <- x / rms(x) * gain.  The sum of squares has the order of a 256-thread
// row: thread t sums columns t, t + 256, .. by fused multiply-adds, the 32
// threads of a warp by the xor tree, the eight warps in order.  Lane l holds
// the columns of threads l, l + 32, .. (value i: thread l + 32 (i mod 8)).
__device__ __forceinline__ void norm_row(float (&x)[kRowVals], const float (&gain)[kRowVals], int cols, int lane,
                                         float eps) {
  float p[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    p[w] = 0.f;
#pragma unroll
    for (int i = w; i < kRowVals; i += 8) p[w] = fmaf(x[i], x[i], p[w]);   // zeros past the row add nothing
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
#pragma unroll
    for (int w = 0; w < 8; ++w) p[w] += __shfl_xor_sync(0xffffffffu, p[w], o);
  }
  float t = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) t += p[w];
  const float inv = 1.0f / sqrtf(t / (float)cols + eps);
#pragma unroll
  for (int i = 0; i < kRowVals; ++i) x[i] = x[i] * inv * gain[i];
}

// The E4M3 scale of a row whose lanes hold maxima m: amax / 448.
__device__ __forceinline__ float fp8_scale(float m) {
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m > 0.f ? __fdiv_rn(m, 448.0f) : 1.0f;
}

// Four values over the scale s as E4M3 bytes.
__device__ __forceinline__ uint32_t fp8x4(const float4& v, float s) {
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v.x, s), __fdiv_rn(v.y, s)), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(__fdiv_rn(v.z, s), __fdiv_rn(v.w, s)), __NV_SATFINITE, __NV_E4M3);
  return lo | (hi << 16);
}

}  // namespace nc
