// Pieces shared by the tensor-core attention over a BF16 KV cache of the
// prefill (k_attn_t5.cu) and of the decode step (k_attn_dec.cu): the chunking
// of the window, the K / V loads, the exponential and the chunk merge, so
// that both compute the same bits.
#pragma once

#include <cuda_bf16.h>

#include "model_dev.cuh"
#include "tc5.cuh"

namespace nc {
namespace t5 {

using namespace dev;
using namespace tc5;

constexpr int kT5Threads = 256;              // 8 warps
constexpr int kT5Chunk = 256;                // positions per chunk (one CTA)
constexpr int kT5Block = 64;                 // positions per block (K of P V)
constexpr int kT5Blocks = kT5Chunk / kT5Block;
constexpr int kT5MaxRanks = 8;               // chunks of a window of at most 2,048 positions
constexpr int kRowB = 128;                   // bytes of one swizzled row: 64 BF16
constexpr int kGroups = kHeadDim / 4;        // float4 groups of an output row

constexpr float kLog2e = 1.4426950408889634f;

// 2^x (PTX ex2.approx, subnormal results flushed to zero).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float exp_fast(float x) { return ex2_approx(__fmul_rn(x, kLog2e)); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// Byte offset of 16-byte segment `seg` of row `row` in the 128-byte swizzle
// layout (rows of 128 bytes, 8-row atoms at 1024-byte aligned addresses).
__device__ __forceinline__ int swz(int row, int seg) { return row * kRowB + ((seg ^ (row & 7)) << 4); }

__device__ __forceinline__ void cp_async16(uint8_t* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Whether block bb of the chunk at c_lo is one TMA box: its 64 ring rows
// contiguous (no wrap) and the slots' tensor maps present.
__device__ __forceinline__ bool kv_block_tma(const Dims& D, int c_lo, int bb) {
  return D.kv_tmap != nullptr && ((c_lo + bb * kT5Block) & (D.L - 1)) + kT5Block <= D.L;
}

// The K and V rows of the chunk's first nblk blocks: TMA boxes of 64 ring
// rows (thread 0; K completes on bar_k, V on bar_v, each arrived on once),
// and the blocks that wrap around the ring by 16-byte copies of the
// positions <= last other than `own` (which the caller writes), zero past
// last (every thread).
__device__ __forceinline__ void load_kv(const Dims& D, const StreamDev& st, int slot, int layer, int g, int c_lo, int nblk, int last,
                        int own, uint8_t* kt, uint8_t* vt, uint64_t* bar_k, uint64_t* bar_v, int tid) {
  if (tid == 0) {
    uint32_t n = 0;
    for (int bb = 0; bb < nblk; ++bb) n += kv_block_tma(D, c_lo, bb);
    mbar_expect_tx(bar_k, n * kT5Block * kRowB);
    mbar_expect_tx(bar_v, n * kT5Block * kRowB);
    if (n) {
      const void* map = static_cast<const uint8_t*>(D.kv_tmap) + (size_t)slot * kTmapBytes;
      const int rk = (layer * 2 * D.hkv + g) * D.L, rv = (layer * 2 * D.hkv + D.hkv + g) * D.L;
      for (int bb = 0; bb < nblk; ++bb) {
        if (!kv_block_tma(D, c_lo, bb)) continue;
        const int r = (c_lo + bb * kT5Block) & (D.L - 1);
        tma_load_2d(kt + bb * kT5Block * kRowB, map, bar_k, 0, rk + r);
        tma_load_2d(vt + bb * kT5Block * kRowB, map, bar_v, 0, rv + r);
      }
    }
  }
  const __nv_bfloat16* kv = static_cast<const __nv_bfloat16*>(st.kv);
  const __nv_bfloat16* kp = kv + attn_plane_off(D, layer, g);
  const __nv_bfloat16* vp = kv + attn_plane_off(D, layer, D.hkv + g);
  for (int bb = 0; bb < nblk; ++bb) {
    if (kv_block_tma(D, c_lo, bb)) continue;
    for (int e = tid; e < kT5Block * 8; e += kT5Threads) {
      const int row = bb * kT5Block + (e >> 3), seg = e & 7;
      const int p = c_lo + row;
      if (p == own) continue;                      // written by the caller
      uint8_t* dk = kt + swz(row, seg);
      uint8_t* dv = vt + swz(row, seg);
      if (p <= last) {
        const size_t ri = (size_t)(p & (D.L - 1)) * kHeadDim + seg * 8;
        cp_async16(dk, kp + ri);
        cp_async16(dv, vp + ri);
      } else {
        *reinterpret_cast<uint4*>(dk) = make_uint4(0, 0, 0, 0);
        *reinterpret_cast<uint4*>(dv) = make_uint4(0, 0, 0, 0);
      }
    }
  }
}

// Dims 4 i .. 4 i + 3 of a pair's output merged over its ncp chunks, in chunk
// order: M = max M_c, f_c = exp(M_c - M), O = sum O_c f_c / sum l_c f_c; zero
// when the row has no chunk.  ml(c) gives (M_c, l_c), o(c) the dims of O_c.
template <typename ML, typename O>
__device__ __forceinline__ float4 merge_chunks(int ncp, ML ml, O oc) {
  float2 v[kT5MaxRanks];
  float4 u[kT5MaxRanks];
#pragma unroll
  for (int c = 0; c < kT5MaxRanks; ++c) {
    if (c < ncp) {
      v[c] = ml(c);
      u[c] = oc(c);
    }
  }
  float M = -INFINITY;
#pragma unroll
  for (int c = 0; c < kT5MaxRanks; ++c)
    if (c < ncp) M = fmaxf(M, v[c].x);
  float l = 0.f;
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int c = 0; c < kT5MaxRanks; ++c) {
    if (c < ncp) {
      const float f = exp_fast(__fsub_rn(v[c].x, M));
      l = __fmaf_rn(v[c].y, f, l);
      o.x = __fmaf_rn(u[c].x, f, o.x);
      o.y = __fmaf_rn(u[c].y, f, o.y);
      o.z = __fmaf_rn(u[c].z, f, o.z);
      o.w = __fmaf_rn(u[c].w, f, o.w);
    }
  }
  if (ncp) o = make_float4(__fdiv_rn(o.x, l), __fdiv_rn(o.y, l), __fdiv_rn(o.z, l), __fdiv_rn(o.w, l));
  return o;
}

__device__ __forceinline__ void store_out(const AttnIO& io, size_t off, float4 o) {
  if (io.out16) {
    *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(io.out16) + off) =
        make_uint2(pack_bf16(o.x, o.y), pack_bf16(o.z, o.w));
  } else {
    *reinterpret_cast<float4*>(io.attn_out + off) = o;
  }
}

}  // namespace t5
}  // namespace nc
