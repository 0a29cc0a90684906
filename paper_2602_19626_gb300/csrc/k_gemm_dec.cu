// tcgen05 projections of a decode step: few rows, so the kernel is bound by
// latency, not by bytes or products.
//
// Y[n][m] = sum_k W[m][k] X[n][k] as in k_gemm_tc.cu, with the same steps over
// K (blocks of 128 bytes, four instructions each, in order), so every output
// element has the same bits.  What differs is everything around the products:
//   - a CTA stores kDecM = 32 weight rows instead of 128, so a 576-row
//     projection spreads over 18 SMs instead of 5 and its weights arrive in a
//     quarter of the time.  The MMA takes M = 64 (the products are those of
//     M = 128, at 29 instead of 43 cycles each): the rows past the 32 are
//     whatever follows in shared memory (later K blocks, then the operand; in
//     bounds by the layout), and their accumulator lanes are never read;
//   - the whole K of the 32 rows sits in shared memory, requested before the
//     wait on the predecessor, so that no copy of weights is left after it;
//   - the operand is made in the prologue where that takes arithmetic on
//     whole rows: the RMSNorm (QKV, gate/up) and the E4M3 row scale (every
//     projection with FP8 weights).  Each CTA repeats it for its rows: a few
//     KB from L2, against a kernel of its own in the chain (5 us alone).
//     A warp owns a row; the sums keep the order of the row kernel.
//
// Measured (GB300, full model, nc_decode, time per token step with the
// separate operand kernels and 128-row tiles -> with these, products issued
// by an elected lane in both this kernel and the attention): one BF16 stream
// 1,076 -> 703 us; 48 FP8 streams 1,315 -> 1,126 us.
// What is left of a projection (one row, K = 576, from the predecessor's end
// to its own): 0.7 us operand, 0.5 us products, 0.4 us epilogue, about 1 us
// between kernels.
//
// Every wait is bounded as in k_gemm_tc.cu; nothing a CTA issued is in flight
// when it exits.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "internal.h"
#include "tc5.cuh"
#include "tc_row.cuh"

namespace nc {

namespace {

using namespace tc5;

constexpr int kDecM = 32;                    // weight rows of a CTA
constexpr int kBlkBytes = 128;               // a K block of one row: one swizzle row
constexpr int kABlk = kDecM * kBlkBytes;     // bytes of a K block of the CTA's weights
constexpr int kMmaM = 64;                    // rows 16 q .. 16 q + 15 in TMEM lanes 32 q ..

// Compile-time (KB, EPI) of a generic lambda.
template <int KB_, int EPI_>
struct Pick {
  static constexpr int kb = KB_, epi = EPI_;
};

// Bytes after the barriers' 1024: the weights' blocks, the operand's, and
// what the MMA's 64 rows read past the last weight block.
__host__ __device__ inline size_t dec_smem_bytes(int nk, int bn) {
  const size_t a = (size_t)nk * kABlk, b = (size_t)nk * bn * kBlkBytes;
  const size_t over = (size_t)(nk - 1) * kABlk + (size_t)kMmaM * kBlkBytes;   // end of the last block's read
  return 1024 + 1024 + (a + b > over ? a + b : over);
}

// Byte offset of column c (of ESZ bytes) of operand row r.
template <int ESZ, int BN>
__device__ __forceinline__ int op_off(int r, int c) {
  constexpr int kPer = kBlkBytes / ESZ;
  const int kb = c / kPer, x = (c % kPer) * ESZ;
  return kb * (BN * kBlkBytes) + r * kBlkBytes + ((((x >> 4) ^ (r & 7)) << 4) | (x & 15));
}

// BN batch rows per CTA, NW warps, RPW rows per warp at a time in the
// prologue.
template <int KB, int EPI, int PRO, int BN, int NW, int RPW>
__global__ void __launch_bounds__(NW * 32, 1)
    k_gemm_dec(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, TcDec g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bar_a = reinterpret_cast<uint64_t*>(base);     // every weight block
  uint64_t* bar_b = bar_a + 1;                             // every operand block (PRO_TMA)
  uint64_t* done = bar_a + 2;                              // every product
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_a + 3);
  float* xsc = reinterpret_cast<float*>(base + 64);        // [BN] E4M3 row scales
  constexpr int kBBlk = BN * kBlkBytes;                    // bytes of a K block of the operand
  // epilogue warps: lane quarters 0 and 1 (weight rows 0 .. 15, 16 .. 31 on
  // 16 lanes each), kCols columns per warp
  constexpr int kCols = BN * 4 / NW < 16 ? 16 : BN * 4 / NW;
  constexpr int kPer = KB ? 64 : 128;                      // elements per K block
  const int nk = (g.K + kPer - 1) / kPer;
  uint8_t* sA = base + 1024;
  uint8_t* sB = sA + (size_t)nk * kABlk;

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kDecM, n0 = blockIdx.y * BN;
  // the row count was written several launches back
  const int B = *g.nB;
  if (n0 >= B) return;                                     // uniform across the CTA
  const int nb = min(BN, B - n0);
  if (threadIdx.x == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(bar_a + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(bar_a, (uint32_t)nk * kABlk);
    for (int kb = 0; kb < nk; ++kb) tma_load_2d(sA + (size_t)kb * kABlk, &tA, bar_a, kb * kPer, m0);
    if (PRO == DPRO_TMA) mbar_expect_tx(bar_b, (uint32_t)nk * kBBlk);
  }
  if (warp == 1) tmem_alloc(tmem_slot, BN);
  const int quarter = warp & 3, c_ep = (warp >> 2) * kCols;
  const bool ep = quarter < 2 && c_ep < BN;
  const int r = m0 + 16 * quarter + (lane & 15);
  const bool mine = ep && lane < 16 && r < g.M;            // this lane's weight row is real
  float ws = 1.f;
  if (!KB && mine) ws = g.w_scale[r];
  float gain[kRowVals];
  if (PRO == DPRO_RMS) load_gain(g.gain, g.K, lane, gain);
  if (PRO == DPRO_TMA && threadIdx.x == 0) prefetch_tmap(&tB);
  pdl_wait();
  pdl_trigger();
  if (PRO == DPRO_TMA && threadIdx.x == 0)
    for (int kb = 0; kb < nk; ++kb) tma_load_2d(sB + (size_t)kb * kBBlk, &tB, bar_b, kb * kPer, n0);
  // the epilogue's residuals, beside the prologue
  float pre[kCols];
  if (EPI == EPI_RESID) {
#pragma unroll
    for (int i = 0; i < kCols; ++i) {
      const int n = n0 + c_ep + i;
      pre[i] = (mine && n < B) ? __ldcg(g.y + (size_t)n * g.M + r) : 0.f;
    }
  }
  if (PRO == DPRO_RMS) {
    // rows warp, warp + NW, ..: RPW of them at a time
    for (int r0 = warp; r0 < nb; r0 += RPW * NW) {
      float x[RPW][kRowVals];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int j = r0 + q * NW;
        load_row(g.x + (size_t)(n0 + min(j, nb - 1)) * g.K, g.K, lane, x[q]);
      }
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int j = r0 + q * NW;
        if (j >= nb) break;                                // uniform across the warp
        norm_row(x[q], gain, g.K, lane, g.eps);            // zero past the row
        // column lane + 32 i: K block 32 i / kPer, and in its 128 bytes the
        // segment of (lane, i mod kStep), the same for every block
        constexpr int kStep = kPer / 32;
        if (KB) {
#pragma unroll
          for (int i = 0; i < kRowVals; ++i)
            if (i < nk * kStep)
              *reinterpret_cast<__nv_bfloat16*>(sB + (i / kStep) * kBBlk + op_off<2, BN>(j, lane + 32 * (i % kStep))) =
                  __float2bfloat16_rn(x[q][i]);
        } else {
          float m = 0.f;
#pragma unroll
          for (int i = 0; i < kRowVals; ++i) m = fmaxf(m, fabsf(x[q][i]));
          const float s = fp8_scale(m);
          if (lane == 0) xsc[j] = s;
#pragma unroll
          for (int i = 0; i < kRowVals; ++i)
            if (i < nk * kStep)
              sB[(i / kStep) * kBBlk + op_off<1, BN>(j, lane + 32 * (i % kStep))] =
                  __nv_cvt_float_to_fp8(__fdiv_rn(x[q][i], s), __NV_SATFINITE, __NV_E4M3);
        }
      }
    }
  } else if (PRO == DPRO_FP8) {
    // FP32 rows to E4M3 by the row's maximum, four columns per lane
    const int nv = g.K / 4;
    for (int r0 = warp; r0 < nb; r0 += RPW * NW) {
      float4 v[RPW][kPlainVecs];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const float4* xr =
            reinterpret_cast<const float4*>(g.x + (size_t)(n0 + min(r0 + q * NW, nb - 1)) * g.K);
#pragma unroll
        for (int i = 0; i < kPlainVecs; ++i)
          v[q][i] = lane + 32 * i < nv ? __ldcg(xr + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int j = r0 + q * NW;
        if (j >= nb) break;                                // uniform across the warp
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < kPlainVecs; ++i)
          m = fmaxf(m, fmaxf(fmaxf(fabsf(v[q][i].x), fabsf(v[q][i].y)), fmaxf(fabsf(v[q][i].z), fabsf(v[q][i].w))));
        const float s = fp8_scale(m);
        if (lane == 0) xsc[j] = s;
#pragma unroll
        for (int i = 0; i < kPlainVecs; ++i) {
          const int c = 4 * (lane + 32 * i);
          if (c < nk * kPer) {
            const uint32_t w = c < g.K ? fp8x4(v[q][i], s) : 0u;
            *reinterpret_cast<uint32_t*>(sB + op_off<1, BN>(j, c)) = w;
          }
        }
      }
    }
  }
  fence_proxy_async();                                     // the operand, read by the tensor core
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = uniform(*tmem_slot);
  bool ok = true;
  if (warp == 0) {
    ok = mbar_wait(bar_a, 0);
    if (PRO == DPRO_TMA) ok = mbar_wait(bar_b, 0) && ok;
    ok = __all_sync(0xffffffffu, ok);
    fence_after_sync();
    const uint64_t da = sdesc_sw128(uniform(smem_u32(sA))), db = sdesc_sw128(uniform(smem_u32(sB)));
    if (elect_one()) {
      if (ok) {
        const uint32_t id = idesc(KB, kMmaM, BN);
        for (int kb = 0; kb < nk; ++kb) {
          // descriptor addresses count 16 bytes
          const uint64_t a = da + (uint64_t)(kb * (kABlk / 16)), b = db + (uint64_t)(kb * (kBBlk / 16));
#pragma unroll
          for (int k = 0; k < 4; ++k) mma_issue(KB, tmem, a + 2 * k, b + 2 * k, id, (kb | k) ? 1u : 0u);
        }
      }
      mma_commit(done);
    }
    __syncwarp();
  }
  ok = __syncthreads_and(ok && (!ep || mbar_wait(done, 0)));
  fence_after_sync();
  if (ok && ep) {
#pragma unroll
    for (int c0 = 0; c0 < kCols; c0 += 16) {
      if (c_ep + c0 >= nb) break;                          // uniform across the warp
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(c_ep + c0), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int n = n0 + c_ep + c0 + i;
        const float sc = KB ? 1.f : __fmul_rn(ws, n < B ? xsc[c_ep + c0 + i] : 0.f);
        if (!KB) v[i] = __fmul_rn(v[i], sc);
        if (EPI == EPI_RESID) v[i] = __fadd_rn(pre[c0 + i], v[i]);
        if (EPI != EPI_SWIGLU && mine && n < B) g.y[(size_t)n * g.M + r] = v[i];
      }
      if (EPI == EPI_SWIGLU) {
#pragma unroll
        for (int i = 0; i < 16; i += 2) swiglu_pair(mine, g.M, g.h_out, g.h16, r, n0 + c_ep + c0 + i, B, v[i], v[i + 1]);
      }
    }
  }
  if (!ok && threadIdx.x == 0) {
    // gave up: the products issued were committed to `done`; wait, with the
    // same bound, for the copies, so that none lands in a CTA that has exited
    mbar_wait(bar_a, 0);
    if (PRO == DPRO_TMA) mbar_wait(bar_b, 0);
    mbar_wait(done, 0);
    if (g.status) atomicOr(g.status, ST_TIMEOUT);
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, BN);
}

template <int KB, int EPI, int PRO, int BN, int NW, int RPW>
cudaError_t dec_t(const TcDec& g, cudaStream_t s, bool pdl) {
  auto kern = k_gemm_dec<KB, EPI, PRO, BN, NW, RPW>;
  const int nk = (g.K + (KB ? 64 : 128) - 1) / (KB ? 64 : 128);
  const dim3 grid((g.M + kDecM - 1) / kDecM, (g.Bmax + BN - 1) / BN);
  const CUtensorMap* a = reinterpret_cast<const CUtensorMap*>(g.tmap_a);
  const CUtensorMap* b = reinterpret_cast<const CUtensorMap*>(g.tmap_b ? g.tmap_b : g.tmap_a);
  return launch_kernel(kern, grid, dim3(NW * 32), dec_smem_bytes(nk, BN), s, pdl, *a, *b, g);
}

template <int KB, int EPI, int PRO, int BN, int NW, int RPW>
cudaError_t dec_prepare_t() {
  return cudaFuncSetAttribute(k_gemm_dec<KB, EPI, PRO, BN, NW, RPW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kDecSmemMax);
}

// The variants of a row-making prologue: one row per warp and 8 warps up to 8
// rows; 16 warps of two rows at a time for more, in tiles of 32 or (above 32
// rows) 64 rows.  Measured (GB300, full model, one nc_step_probe, in us):
//   8 warps, then 16 warps of two rows: BF16 8 rows 551, 599; 16: 636, 661;
//   24: 697, 686; 32: 762, 710; FP8 8 rows 722, 759; 16: 871, 845
//   above 32 rows 64-row tiles, then 32-row tiles of 16 and of 8 warps: BF16
//   48 rows 849, 871, 796; 64: 905, 934, 859; 32 active rows in a launch for
//   64: 721, 722, 771
// The E4M3 rows of a residual projection, 8 warps, then 16: 8 rows 722, 723;
// 16: 981, 871.
template <typename F>
cudaError_t dec_rms(int kind_bf16, int epi, F f) {
  if (epi == EPI_STORE) return kind_bf16 ? f(Pick<1, EPI_STORE>()) : f(Pick<0, EPI_STORE>());
  if (epi == EPI_SWIGLU) return kind_bf16 ? f(Pick<1, EPI_SWIGLU>()) : f(Pick<0, EPI_SWIGLU>());
  return cudaErrorInvalidValue;
}

}  // namespace

bool gemm_dec_fits(int kind_bf16, int K, int pro) {
  const int per = kind_bf16 ? 64 : 128;
  const int nk = (K + per - 1) / per;
  if (pro == DPRO_RMS && nk * per > 32 * kRowVals) return false;
  if (pro == DPRO_FP8 && nk * per > 128 * kPlainVecs) return false;
  return dec_smem_bytes(nk, pro == DPRO_RMS ? 64 : 32) <= (size_t)kDecSmemMax;
}

cudaError_t prepare_dec_kernels() {
  cudaError_t e = cudaSuccess;                     // attributes of the current device's kernels
  auto also = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
  for (int kb = 0; kb < 2; ++kb)
    for (int epi : {(int)EPI_STORE, (int)EPI_SWIGLU})
      also(dec_rms(kb, epi, [&](auto k) {
        constexpr int KB = decltype(k)::kb, EPI = decltype(k)::epi;
        cudaError_t r = dec_prepare_t<KB, EPI, DPRO_RMS, 32, 8, 1>();
        if (r == cudaSuccess) r = dec_prepare_t<KB, EPI, DPRO_RMS, 32, 16, 2>();
        return r == cudaSuccess ? dec_prepare_t<KB, EPI, DPRO_RMS, 64, 16, 2>() : r;
      }));
  also(dec_prepare_t<1, EPI_RESID, DPRO_TMA, 32, 8, 1>());
  also(dec_prepare_t<0, EPI_RESID, DPRO_FP8, 32, 8, 1>());
  also(dec_prepare_t<0, EPI_RESID, DPRO_FP8, 32, 16, 1>());
  return e;
}

cudaError_t launch_gemm_dec(const TcDec& g, int kind_bf16, int epi, int pro, cudaStream_t s, bool pdl) {
  if (pro == DPRO_RMS)
    return dec_rms(kind_bf16, epi, [&](auto k) {
      constexpr int KB = decltype(k)::kb, EPI = decltype(k)::epi;
      if (g.Bmax <= 8) return dec_t<KB, EPI, DPRO_RMS, 32, 8, 1>(g, s, pdl);
      if (g.Bmax <= 32) return dec_t<KB, EPI, DPRO_RMS, 32, 16, 2>(g, s, pdl);
      return dec_t<KB, EPI, DPRO_RMS, 64, 16, 2>(g, s, pdl);
    });
  if (epi != EPI_RESID) return cudaErrorInvalidValue;
  if (pro == DPRO_TMA && kind_bf16) return dec_t<1, EPI_RESID, DPRO_TMA, 32, 8, 1>(g, s, pdl);
  if (pro == DPRO_FP8 && !kind_bf16)
    return g.Bmax <= 8 ? dec_t<0, EPI_RESID, DPRO_FP8, 32, 8, 1>(g, s, pdl)
                       : dec_t<0, EPI_RESID, DPRO_FP8, 32, 16, 1>(g, s, pdl);
  return cudaErrorInvalidValue;
}

}  // namespace nc
