// Attention of a decode step over a BF16 KV cache on the tcgen05 tensor
// cores (Sec. 3.2 model, Sec. 3.9 sliding window): one query row per stream.
//
// The kernel is bound by latency: a row's grp <= 4 query heads per KV head
// are a few hundred thousand products.  The window is cut into the chunks and
// blocks of the prefill attention (k_attn_t5.cu), CTA (c, g, j) computes chunk
// c of row j and KV head g with the same products, partial sums and merge, so
// the two give the same bits; the work is laid out for one row:
//   - the scores are transposed, S^T = K Q^T: the 256 positions are the MMA's
//     M (two tiles of 128), the heads its N (16 columns, grp of them real), so
//     each of the 256 threads holds one position's scores and forms its own
//     exponentials, where a tile of (row, head) pairs left all but grp lanes
//     of two warps idle over 64 positions each;
//   - the numerators go to shared memory twice: as the P operand (BF16, one
//     8-row swizzle atom per block of 64 positions: the MMA's M = 64 reads on
//     into the next atoms and the keys, rows whose results are not read), and
//     in FP32 for the sums, which grp warps take while P V runs: lane 8 b + q
//     adds the eight numerators q, q + 8, .. of block b in order, a fixed tree
//     adds the eight partial sums, blocks 0 + 2 and 1 + 3, then both;
//   - the chunks of a row are a cluster (1, 2, 4 or 8 CTAs by the longest
//     stream the launch may hold): each CTA stores (O_c, M_c, l_c) into rank
//     0's shared memory and rank 0 merges them in chunk order.  A window of
//     one chunk merges in its own CTA, with no exchange.
// The cached K and V, and the rotation of the fed position, are loaded before
// the wait on the QKV projection; the CTA of the chunk that holds the fed
// position rotates its k, rounds k and v to BF16 and puts them into the ring
// and into its tiles.
//
// Measured (GB300, full model, nc_decode, time per token step, with the pair
// tiles and the partials merged through global memory -> this kernel): one
// BF16 stream of 300 tokens 703 -> 556 us; 48 FP8 streams of up to 160 tokens
// 1,126 -> 976 us.
//
// Every wait is bounded as in k_attn_t5.cu.
#include <algorithm>

#include <cooperative_groups.h>

#include "attn_t5.cuh"

namespace cg = cooperative_groups;

namespace nc {

namespace {

using namespace t5;

constexpr int kSCols = 16;                   // N of a score tile (the heads, padded)
constexpr uint32_t kDecCols = 128;           // TMEM: S^T tiles at 0 and 16, O_c at 32 .. 95

// Shared memory, byte offsets from a 1024-byte aligned base.
struct DecLayout {
  static constexpr int bars = 0;                           // 5 mbarriers
  static constexpr int slot = 64;                          // TMEM address
  static constexpr int red = 128;                          // [8 warps][kMaxGroup] floats: chunk maxima
  static constexpr int sum = red + kT5Threads / 32 * kMaxGroup * 4;   // [kMaxGroup] floats: l_c
  static constexpr int q = 1024;                           // [16 heads][128 B]
  static constexpr int p = q + kSCols * kRowB;             // [4 blocks][8 rows][128 B]
  static constexpr int k = p + kT5Blocks * 8 * kRowB;      // [256 positions][128 B]
  static constexpr int v = k + kT5Chunk * kRowB;           // [256 positions][128 B]
  static constexpr int e = v + kT5Chunk * kRowB;           // [kMaxGroup][256] floats: numerators
  static constexpr int part = e + kMaxGroup * kT5Chunk * 4;           // [8 chunks][kMaxGroup][64] floats
  static constexpr int ml = part + kT5MaxRanks * kMaxGroup * kHeadDim * 4;   // [8][kMaxGroup] (M_c, l_c)
  static constexpr int total = ml + kT5MaxRanks * kMaxGroup * 8;
};
static_assert(DecLayout::p % 1024 == 0 && DecLayout::k % 1024 == 0, "swizzle atoms");
static_assert(DecLayout::p + (kT5Blocks - 1) * 1024 + 64 * kRowB <= DecLayout::v, "P reads stay in P and K");
constexpr size_t kDecSmem = DecLayout::total + 1024;       // + alignment slack

template <int S>
__global__ void __launch_bounds__(kT5Threads, 2) k_attn_dec(Dims D, Batch b, int layer, AttnIO io) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  using Ly = DecLayout;
  uint64_t* bar_k = reinterpret_cast<uint64_t*>(sm + Ly::bars);   // the K boxes
  uint64_t* bar_v = bar_k + 1;                                     // the V boxes
  uint64_t* bar_s = bar_k + 2;                                     // the score products
  uint64_t* bar_o = bar_k + 3;                                     // P V
  uint64_t* bar_done = bar_k + 4;                                  // every product issued (give-up path)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + Ly::slot);
  float* red = reinterpret_cast<float*>(sm + Ly::red);
  float* lsum = reinterpret_cast<float*>(sm + Ly::sum);
  uint8_t* qt = sm + Ly::q;
  uint8_t* pt = sm + Ly::p;
  uint8_t* kt = sm + Ly::k;
  uint8_t* vt = sm + Ly::v;
  float* es = reinterpret_cast<float*>(sm + Ly::e);
  float* part = reinterpret_cast<float*>(sm + Ly::part);
  float2* ml = reinterpret_cast<float2*>(sm + Ly::ml);

  const int rank = blockIdx.x, g = blockIdx.y, j = blockIdx.z;    // chunk, KV head, row
  const int grp = D.hq / D.hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = uniform_warp();
  // the row count and the row's slot and position were written at least two
  // launches back: read before the wait
  if (j >= *b.nB) return;
  const int slot = b.slots[j];
  StreamDev& st = b.st[slot];
  const int a = st.n_coded, start = window_start(D, st);
  const int nch = (a - start) / kT5Chunk + 1;
  if (rank >= nch) return;                         // an exited CTA counts as arrived at the cluster's barriers
  const int c_lo = start + rank * kT5Chunk;
  const int nblk = min(kT5Blocks, (a - c_lo) / kT5Block + 1);
  const bool owner = rank == nch - 1;              // the chunk holds position a
  // rank 0 must have started before its shared memory is written remotely
  if (S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(bar_k + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(tmem_slot, kDecCols);
  __syncthreads();                                 // the barriers are initialised
  load_kv(D, st, slot, layer, g, c_lo, nblk, a, a, kt, vt, bar_k, bar_v, tid);
  const float2 cs = rope_cs(D, a, lane);
  pdl_wait();
  pdl_trigger();

  // ---- the rotated, 1/8-scaled queries (warp h: head h), the fed k and v
  bool ok = true;
  const float* row = io.qkv + (size_t)j * D.qkv_rows;
  if (warp < grp) {
    const float* src = row + (g * grp + warp) * kHeadDim;
    const float2 rr = rope_rotate(__ldcg(src + lane), __ldcg(src + lane + kHeadDim / 2), cs);
    // the 1/sqrt(64) score scale is a power of two: exact
    *reinterpret_cast<__nv_bfloat16*>(qt + swz(warp, lane >> 3) + (lane & 7) * 2) = __float2bfloat16_rn(rr.x * 0.125f);
    *reinterpret_cast<__nv_bfloat16*>(qt + swz(warp, (lane + 32) >> 3) + (lane & 7) * 2) =
        __float2bfloat16_rn(rr.y * 0.125f);
  } else if (owner && warp >= 6) {
    const int R = a - c_lo;
    const bool boxed = kv_block_tma(D, c_lo, R / kT5Block);
    const size_t ri = (size_t)(a & (D.L - 1)) * kHeadDim;
    if (warp == 6) {                               // dims lane and lane + 32 of k
      const float* src = row + D.hq * kHeadDim + g * kHeadDim;
      const float2 rr = rope_rotate(__ldcg(src + lane), __ldcg(src + lane + kHeadDim / 2), cs);
      __nv_bfloat16* kv = static_cast<__nv_bfloat16*>(st.kv) + attn_plane_off(D, layer, g) + ri;
      const __nv_bfloat16 k0 = __float2bfloat16_rn(rr.x), k1 = __float2bfloat16_rn(rr.y);
      kv[lane] = k0;
      kv[lane + kHeadDim / 2] = k1;
      if (boxed) ok = mbar_wait(bar_k, 0);         // the tile's row after its box has landed
      *reinterpret_cast<__nv_bfloat16*>(kt + swz(R, lane >> 3) + (lane & 7) * 2) = k0;
      *reinterpret_cast<__nv_bfloat16*>(kt + swz(R, (lane + 32) >> 3) + (lane & 7) * 2) = k1;
    } else {                                       // dims 2 lane, 2 lane + 1 of v
      const int d0 = 2 * lane;
      const float2 x = __ldcg(reinterpret_cast<const float2*>(row + (D.hq + D.hkv) * kHeadDim + g * kHeadDim + d0));
      const uint32_t v2 = pack_bf16(x.x, x.y);
      *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(st.kv) + attn_plane_off(D, layer, D.hkv + g) + ri + d0) =
          v2;
      if (boxed) ok = mbar_wait(bar_v, 0);
      *reinterpret_cast<uint32_t*>(vt + swz(R, d0 >> 3) + (d0 & 7) * 2) = v2;
    }
  }
  cp_async_wait_all();
  fence_proxy_async();
  fence_before_sync();
  ok = __syncthreads_and(ok && mbar_wait(bar_k, 0));
  fence_after_sync();
  const uint32_t tmem = uniform(*tmem_slot);
  const uint64_t dk = sdesc_sw128(uniform(smem_u32(kt))), dq = sdesc_sw128(uniform(smem_u32(qt))),
                 dp = sdesc_sw128(uniform(smem_u32(pt))), dv = sdesc_sw128_mn(uniform(smem_u32(vt)));

  // ---- S^T = K Q^T, 128 positions per tile
  if (warp == 0) {
    if (elect_one()) {
      if (ok) {
        const uint32_t ids = idesc(1, 128, kSCols);
        for (int h = 0; h < (nblk > 2 ? 2 : 1); ++h)
#pragma unroll
          for (int k = 0; k < kHeadDim / 16; ++k)  // descriptor addresses count 16 bytes
            mma_issue(1, tmem + kSCols * h, dk + (uint64_t)(h * (128 * kRowB / 16) + 2 * k), dq + 2 * k, ids,
                      k ? 1u : 0u);
      }
      mma_commit(bar_s);
    }
    __syncwarp();
  }
  ok = mbar_wait(bar_s, 0) && ok;
  fence_after_sync();
  // thread tid holds position c_lo + tid: TMEM lane tid mod 128 of its tile
  const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const bool valid = c_lo + tid <= a;
  float s[kMaxGroup];
  if (warp < 4 || nblk > 2) {
    uint32_t r[4];
    tmem_ld4_nowait(tlane + kSCols * (warp >> 2), r);
    tmem_wait_ld();
#pragma unroll
    for (int h = 0; h < kMaxGroup; ++h) s[h] = __uint_as_float(r[h]);
  }
#pragma unroll
  for (int h = 0; h < kMaxGroup; ++h) {
    if (h < grp) {
      const float m = warp_max(valid ? s[h] : -INFINITY);
      if (lane == 0) red[warp * kMaxGroup + h] = m;
    }
  }
  __syncthreads();
  float Mc[kMaxGroup];
#pragma unroll
  for (int h = 0; h < kMaxGroup; ++h) {
    if (h < grp) {
      float m = red[h];
#pragma unroll
      for (int w = 1; w < kT5Threads / 32; ++w) m = fmaxf(m, red[w * kMaxGroup + h]);
      Mc[h] = m;
      const float mb = m > -INFINITY ? -__fmul_rn(m, kLog2e) : 0.f;
      const float e = valid ? ex2_approx(__fmaf_rn(s[h], kLog2e, mb)) : 0.f;
      es[h * kT5Chunk + tid] = e;
      *reinterpret_cast<__nv_bfloat16*>(pt + (tid >> 6) * (8 * kRowB) + swz(h, (tid & 63) >> 3) + (tid & 7) * 2) =
          __float2bfloat16_rn(e);
    }
  }
  fence_proxy_async();
  fence_before_sync();
  ok = __syncthreads_and(ok && mbar_wait(bar_v, 0));
  fence_after_sync();

  // ---- O_c = sum_b P_b V_b (M = 64: head h in TMEM lane h), and the sums
  if (warp == 0) {
    if (elect_one()) {
      if (ok) {
        const uint32_t ido = idesc(1, 64, kHeadDim, 1);
        for (int bb = 0; bb < nblk; ++bb)
#pragma unroll
          for (int k = 0; k < kT5Block / 16; ++k)
            mma_issue(1, tmem + 2 * kSCols, dp + (uint64_t)(bb * (8 * kRowB / 16) + 2 * k),
                      dv + (uint64_t)((bb * kT5Block + 16 * k) * (kRowB / 16)), ido, bb + k ? 1u : 0u);
      }
      mma_commit(bar_o);
    }
    __syncwarp();
  } else if (warp <= grp) {
    const float* eh = es + (warp - 1) * kT5Chunk + (lane >> 3) * kT5Block + (lane & 7);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc = __fadd_rn(acc, eh[8 * i]);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, o));
    acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, 16));   // blocks 0 + 2, 1 + 3
    acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, 8));
    if (lane == 0) lsum[warp - 1] = acc;
  }
  if (S > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");   // rank 0 has started
  ok = __syncthreads_and(ok && mbar_wait(bar_o, 0));
  fence_after_sync();

  // ---- the chunk's (O_c, M_c, l_c) to rank 0
  float* rpart = part;
  float2* rml = ml;
  if (S > 1) {
    cg::cluster_group cl = cg::this_cluster();
    rpart = cl.map_shared_rank(part, 0);
    rml = cl.map_shared_rank(ml, 0);
  }
  if ((warp & 3) == 0) {                           // warps 0, 4: dims 0 .. 31, 32 .. 63
    uint32_t r[32];
    tmem_ld32_nowait(tmem + 2 * kSCols + 8 * warp, r);
    tmem_wait_ld();
    if (lane < grp) {
      float4* dst = reinterpret_cast<float4*>(rpart + (rank * kMaxGroup + lane) * kHeadDim + 8 * warp);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        dst[i] = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]),
                             __uint_as_float(r[4 * i + 3]));
    }
  } else if (warp == 1) {
#pragma unroll
    for (int h = 0; h < kMaxGroup; ++h)
      if (h < grp && lane == h) rml[rank * kMaxGroup + h] = make_float2(Mc[h], lsum[h]);
  }
  // give-up path: every copy and product issued has completed before the
  // memory is freed
  if (!ok) {
    if (warp == 0 && elect_one()) mma_commit(bar_done);
    __syncwarp();
    mbar_wait(bar_done, 0);
    mbar_wait(bar_k, 0);
    mbar_wait(bar_v, 0);
    cp_async_wait_all();
    if (tid == 0) atomicOr(&st.status, ST_TIMEOUT);
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, kDecCols);
  if (S > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (rank > 0) return;
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (tid < grp * kGroups) {
    const int h = tid / kGroups, i = tid % kGroups;
    const float4 o = merge_chunks(
        nch, [&](int c) { return ml[c * kMaxGroup + h]; },
        [&](int c) { return *reinterpret_cast<const float4*>(part + (c * kMaxGroup + h) * kHeadDim + 4 * i); });
    store_out(io, (size_t)j * D.hq * kHeadDim + (g * grp + h) * kHeadDim + 4 * i, o);
  }
}

template <int S>
cudaError_t launch_dec_s(const Dims& D, const Batch& b, int layer, const AttnIO& io, cudaStream_t s) {
  const dim3 grid(S, D.hkv, b.Bmax);
  if (S == 1) return launch_kernel(k_attn_dec<S>, grid, dim3(kT5Threads), kDecSmem, s, D.pdl, D, b, layer, io);
  return launch_kernel_cluster(k_attn_dec<S>, grid, dim3(kT5Threads), kDecSmem, s, D.pdl, S, D, b, layer, io);
}

}  // namespace

cudaError_t prepare_attn_dec() {
  cudaError_t e = cudaSuccess;                     // attributes of the current device's kernels
  auto set = [&](auto kern) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecSmem);
  };
  set(k_attn_dec<1>);
  set(k_attn_dec<2>);
  set(k_attn_dec<4>);
  set(k_attn_dec<8>);
  return e;
}

int attn_dec_class(const Dims& D, const Batch& b) {
  // chunks of the longest window a row of this launch may reach
  const int64_t len = b.len_max > 0 && b.len_max < D.L ? b.len_max : D.L;
  const int nch = (int)((len + kT5Chunk - 1) / kT5Chunk);
  return nch <= 1 ? 0 : nch <= 2 ? 1 : nch <= 4 ? 2 : 3;
}

cudaError_t launch_attn_dec(const Dims& D, const Batch& b, int layer, const float* qkv, float* attn_out, void* out16,
                            cudaStream_t s) {
  const AttnIO io{qkv, attn_out, out16};
  switch (attn_dec_class(D, b)) {
    case 0: return launch_dec_s<1>(D, b, layer, io, s);
    case 1: return launch_dec_s<2>(D, b, layer, io, s);
    case 2: return launch_dec_s<4>(D, b, layer, io, s);
    default: return launch_dec_s<8>(D, b, layer, io, s);
  }
}

}  // namespace nc
