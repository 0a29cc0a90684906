// Prefill attention over a BF16 KV cache on the tcgen05 tensor cores,
// accumulators in tensor memory (Sec. 3.2 model, Sec. 3.9 sliding window).
//
// A tile is up to 128 (query row, head) pairs of one stream and KV head: the
// grp query heads sharing the KV head of a row of consecutive positions,
// pair p = r grp + h, cut into tiles of 128 consecutive pairs (a tile's
// first and last row may be split with its neighbours).  The pairs are the
// MMA's M = 128 rows, so each pair's products depend on its own query alone;
// a decode step's row (k_attn_dec.cu) takes the same products, partial sums
// and merge, and gives the same bits.
//
// The window [start, a] of a row is cut into chunks of 256 positions (chunk
// c = [start + 256 c, ...)), a chunk into four blocks of 64.  CTA (c, g, t)
// computes chunk c of tile t and KV head g with 8 warps; warp w reads TMEM
// lanes 32 (w mod 4) .. + 31 (one lane per pair) and belongs to warpgroup
// h = w / 4, which takes blocks h and h + 2:
//   - the K and V rows of the chunk's blocks go to shared memory in the
//     128-byte swizzle layout, a block of 64 ring rows per TMA copy (a block
//     that wraps around the ring by 16-byte asynchronous copies); rows past
//     the tile's last position hold whatever the ring holds there (zero from
//     allocation, else finite older entries), which the zero probabilities
//     of masked positions cancel; the pairs' rotated 1/8-scaled queries in
//     BF16, written by the append pass, go beside them;
//   - one lane issues the scores of every block as one product of N = 64
//     nblk columns (M 128, four K steps of 16 head dims; four instructions
//     for the chunk instead of sixteen), S_b in tensor-memory columns 64 b ..
//     64 b + 63;
//   - each pair's chunk maximum M_c over its unmasked scores (positions up
//     to its row's), then e = 2^(s log2 e - M_c log2 e) (PTX ex2.approx),
//     their FP32 sum l_c (per block eight interleaved partial sums and a
//     fixed tree; blocks h, h + 2 added in order per warpgroup, then the two
//     warpgroups' sums) and P_b = BF16(e) into shared memory (the key tile
//     and the query tile hold the P buffers once every score is computed);
//   - O_c = sum_b P_b V_b accumulates in columns 0 .. 63 (block 0's scores,
//     read by then; V read MN-major straight from its tile; blocks past the
//     row carry zero probabilities);
//   - (O_c, M_c, l_c) go to a global partials buffer (O_c as 16 float4
//     planes of the tile's pairs, so that a warp's stores and loads are
//     contiguous), and every output element is merged over the row's chunks
//     in chunk order: O = sum O_c f_c / sum l_c f_c, f_c = exp(M_c - max M_c)
//     by the merge kernel that follows.
// The rows were appended to the ring by k_kv_append_t5 before this kernel.
// About 84 KB of shared memory and 256 TMEM columns: two CTAs per SM.
//
// Every wait on an mbarrier is bounded; a wait that gives up raises
// ST_TIMEOUT in the stream's status word, skips the remaining products and,
// before the tensor memory is freed, waits (with the same bound) for the
// copies and products already issued.
#include <cuda_bf16.h>

#include <algorithm>

#include "attn_t5.cuh"

namespace nc {

namespace {

using namespace t5;

constexpr int kT5Pairs = 128;                // MMA M: (row, head) pairs per tile
constexpr uint32_t kT5Cols = 256;            // TMEM columns: S_b at 64 b; O_c at 0
constexpr int kPartRow = kHeadDim + 4;       // floats per (chunk, pair) partial: O_c[64], M_c, l_c, padding
constexpr int kMergePairs = 16;              // pairs of one merge CTA (x 16 groups = 256 threads)

// Shared memory, byte offsets from a 1024-byte aligned base.
struct T5Layout {
  static constexpr int q = 0;                              // [128 pairs][128 B]; later P buffer 2
  static constexpr int k = q + kT5Pairs * kRowB;           // [256 positions][128 B]; later P buffers 0, 1
  static constexpr int v = k + kT5Chunk * kRowB;           // [256 positions][128 B]
  static constexpr int red = v + kT5Chunk * kRowB;         // [2][128] floats: the warpgroups' maxima, then sums
  static constexpr int bars = red + 2 * kT5Pairs * 4;      // 6 mbarriers
  static constexpr int slot = bars + 64;                   // TMEM address
  static constexpr int arow = slot + 16;                   // [128] row positions
  static constexpr int total = arow + kT5Pairs * 4;
};
constexpr size_t kT5Smem = T5Layout::total + 1024;         // + alignment slack

// The tile of CTA z: pairs pb .. pb + npairs - 1 (pb counted from row0's
// first pair) of rows row0 .. row0 + nr - 1.  Stream j takes tps tiles of 128
// consecutive pairs of its pm rows.
struct T5Tile {
  int row0, nr, npairs, pb;
};
__device__ __forceinline__ T5Tile t5_tile(const Batch& b, int grp, int tps, int z) {
  T5Tile t;
  const int j = z / tps, sub = z % tps;
  const int p0 = sub * kT5Pairs;
  t.npairs = min(kT5Pairs, b.pm * grp - p0);
  const int r_lo = p0 / grp;
  t.nr = (p0 + t.npairs - 1) / grp - r_lo + 1;
  t.row0 = j * b.pm + r_lo;
  t.pb = p0 - r_lo * grp;
  return t;
}

// The maximum of the first nvalid of the 64 scores at TMEM column `col` of
// this thread's lane.
__device__ __forceinline__ float block_max(uint32_t tlane, uint32_t col, int nvalid) {
  uint32_t r[2][32];
  tmem_ld32_nowait(tlane + col, r[0]);
  tmem_ld32_nowait(tlane + col + 32, r[1]);
  tmem_wait_ld();
  float m = -INFINITY;
  if (nvalid == kT5Block) {
#pragma unroll
    for (int i = 0; i < kT5Block; ++i) m = fmaxf(m, __uint_as_float(r[i >> 5][i & 31]));
  } else {
#pragma unroll
    for (int i = 0; i < kT5Block; ++i)
      if (i < nvalid) m = fmaxf(m, __uint_as_float(r[i >> 5][i & 31]));
  }
  return m;
}

// The numerators of one block for this thread's pair: e = 2^(s log2 e + mb)
// (mb = -M_c log2 e) over the first nvalid of the 64 scores at TMEM column
// `col`, zero past them, rounded to BF16 into the pair's row of the P tile;
// returns their FP32 sum.
__device__ __forceinline__ float block_exp(uint32_t tlane, uint32_t col, int nvalid, float mb, uint8_t* ptile,
                                           int pair) {
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t r[32];
    tmem_ld32_nowait(tlane + col + 32 * half, r);
    tmem_wait_ld();
    float e[32];
    if (nvalid == kT5Block) {
#pragma unroll
      for (int i = 0; i < 32; ++i) e[i] = ex2_approx(__fmaf_rn(__uint_as_float(r[i]), kLog2e, mb));
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        e[i] = 32 * half + i < nvalid ? ex2_approx(__fmaf_rn(__uint_as_float(r[i]), kLog2e, mb)) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i & 7] = __fadd_rn(acc[i & 7], e[i]);
#pragma unroll
    for (int sg = 0; sg < 4; ++sg) {
      const uint4 u = make_uint4(pack_bf16(e[8 * sg], e[8 * sg + 1]), pack_bf16(e[8 * sg + 2], e[8 * sg + 3]),
                                 pack_bf16(e[8 * sg + 4], e[8 * sg + 5]), pack_bf16(e[8 * sg + 6], e[8 * sg + 7]));
      *reinterpret_cast<uint4*>(ptile + swz(pair, 4 * half + sg)) = u;
    }
  }
  return __fadd_rn(__fadd_rn(__fadd_rn(acc[0], acc[1]), __fadd_rn(acc[2], acc[3])),
                   __fadd_rn(__fadd_rn(acc[4], acc[5]), __fadd_rn(acc[6], acc[7])));
}

// Partials of tile-and-head tg: O_c of pair p, dims 4 i .. 4 i + 3, at float4
// (c 16 + i) tp + p; (M_c, l_c) at float4 16 kT5MaxRanks tp + c tp + p.
__device__ __forceinline__ float4* part_base(const Dims& D, size_t tg, int tp) {
  return reinterpret_cast<float4*>(D.attn_part) + tg * kT5MaxRanks * tp * (kPartRow / 4);
}

// Dims 4 i .. 4 i + 3 of pair p's output merged over its ncp chunks.
__device__ __forceinline__ float4 merge_item(const float4* part, int tp, int p, int i, int ncp) {
  const float4* ml = part + (size_t)kT5MaxRanks * kGroups * tp + p;
  return merge_chunks(
      ncp,
      [&](int c) {
        const float4 w = __ldcg(ml + (size_t)c * tp);
        return make_float2(w.x, w.y);
      },
      [&](int c) { return __ldcg(part + (size_t)(c * kGroups + i) * tp + p); });
}

__global__ void __launch_bounds__(kT5Threads, 2) k_attn_t5(Dims D, Batch b, int layer, int tps, AttnIO io) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  using Ly = T5Layout;
  const int grp = D.hq / D.hkv;
  uint8_t* qt = sm + Ly::q;
  uint8_t* kt = sm + Ly::k;
  uint8_t* vt = sm + Ly::v;
  float* red = reinterpret_cast<float*>(sm + Ly::red);
  uint64_t* bar_k = reinterpret_cast<uint64_t*>(sm + Ly::bars);   // the K boxes
  uint64_t* bar_v = bar_k + 1;                                     // the V boxes
  uint64_t* bar_s = bar_k + 2;                                     // every score product
  uint64_t* bar_o0 = bar_k + 3;                                    // P V of blocks 0, 1
  uint64_t* bar_o1 = bar_k + 4;                                    // P V of blocks 2, 3
  uint64_t* bar_done = bar_k + 5;                                  // every product issued
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + Ly::slot);
  int* a_row = reinterpret_cast<int*>(sm + Ly::arow);

  const int rank = blockIdx.x;                     // the chunk of the window
  const int g = blockIdx.y;
  const int tid = threadIdx.x, wg = tid >> 7, p = tid & (kT5Pairs - 1);
  const T5Tile T = t5_tile(b, grp, tps, blockIdx.z);
  // the row count and the rows' slots and positions were written at least
  // two launches back: read before the wait
  if (T.row0 >= *b.nB) return;
  const int slot = b.slots[T.row0];
  StreamDev& st = b.st[slot];
  if (tid < T.nr) a_row[tid] = b.pos[T.row0 + tid];
  __syncthreads();
  // the rows' positions rise up to their stream's end
  int a_max = a_row[T.nr - 1];
  for (int r = 0; a_max < 0 && r < T.nr; ++r) a_max = a_row[T.nr - 1 - r];
  const int start = a_max < 0 ? 0 : window_start_at(D, a_max);
  const int nch = a_max < 0 ? 0 : (a_max - start) / kT5Chunk + 1;
  if (rank >= nch) {
    // a tile of no window (every row past its stream's end): zeros, by rank 0
    if (nch == 0 && rank == 0 && p < T.npairs) {
      pdl_wait();
      const int rr = (T.pb + p) / grp, hh = (T.pb + p) % grp;
      for (int i = 0; i < 8; ++i)
        store_out(io, (size_t)(T.row0 + rr) * D.hq * kHeadDim + (g * grp + hh) * kHeadDim + 32 * wg + 4 * i,
                  make_float4(0.f, 0.f, 0.f, 0.f));
    }
    return;
  }
  const int c_lo = start + rank * kT5Chunk;
  const int nblk = min(kT5Blocks, (a_max - c_lo) / kT5Block + 1);
  // this thread's pair and its row's position (-1: padding or past the stream's end)
  const int my_r = (T.pb + p) / grp, my_h = (T.pb + p) % grp;
  const int my_a = p < T.npairs ? a_row[my_r] : -1;
  const bool mine = 32 * ((tid >> 5) & 3) < T.npairs;   // warp-uniform: the warp's lanes hold real pairs

  bool ok = true;
  if (tid == 0) {
    for (int i = 0; i < 6; ++i) mbar_init(bar_k + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) tmem_alloc(tmem_slot, kT5Cols);
  __syncthreads();                                 // the barriers are initialised
  // the rows were appended by the launch just before
  pdl_wait();
  pdl_trigger();
  {
    load_kv(D, st, slot, layer, g, c_lo, nblk, a_max, -1, kt, vt, bar_k, bar_v, tid);
    // the pairs' rotated, 1/8-scaled BF16 queries (zero for padding pairs):
    // warpgroup h writes dims 16 h .. 16 h + 15 and 32 + 16 h .. 32 + 16 h + 15
    if (mine) {
      uint4 s0 = make_uint4(0, 0, 0, 0), s1 = s0, s2 = s0, s3 = s0;
      if (my_a >= 0) {
        const uint4* src = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(D.q16) +
                                                          ((size_t)(T.row0 + my_r) * D.hq + g * grp + my_h) * kHeadDim);
        s0 = __ldcg(src + 2 * wg);
        s1 = __ldcg(src + 2 * wg + 1);
        s2 = __ldcg(src + 4 + 2 * wg);
        s3 = __ldcg(src + 4 + 2 * wg + 1);
      }
      *reinterpret_cast<uint4*>(qt + swz(p, 2 * wg)) = s0;
      *reinterpret_cast<uint4*>(qt + swz(p, 2 * wg + 1)) = s1;
      *reinterpret_cast<uint4*>(qt + swz(p, 4 + 2 * wg)) = s2;
      *reinterpret_cast<uint4*>(qt + swz(p, 4 + 2 * wg + 1)) = s3;
    }
    cp_async_wait_all();
    fence_proxy_async();
    fence_before_sync();
    // the queries, the copied rows and every K box are in place
    ok = __syncthreads_and(mbar_wait(bar_k, 0));
    fence_after_sync();
    const uint32_t tmem = uniform(*tmem_slot);
    const int warp = uniform_warp();
    const uint64_t dq = sdesc_sw128(uniform(smem_u32(qt))), dk = sdesc_sw128(uniform(smem_u32(kt))),
                   dv = sdesc_sw128_mn(uniform(smem_u32(vt)));
    const uint32_t tlane = tmem + ((uint32_t)(32 * ((tid >> 5) & 3)) << 16);
    if (warp == 0 && ok) {
      if (elect_one()) {
        const uint32_t ids = idesc(1, kT5Pairs, kT5Block * nblk);
#pragma unroll
        for (int k = 0; k < kHeadDim / 16; ++k)     // descriptor addresses count 16 bytes
          mma_issue(1, tmem, dq + 2 * k, dk + 2 * k, ids, k ? 1u : 0u);
        mma_commit(bar_s);
      }
      __syncwarp();
    }
    // every score product done (the key and query tiles hold the P buffers
    // from here) and every V box in place
    ok = __syncthreads_and(ok && mbar_wait(bar_s, 0) && mbar_wait(bar_v, 0));
    fence_after_sync();
    // the unmasked columns of this pair in each of the warpgroup's blocks
    int nv[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int bb = wg + 2 * k, blo = c_lo + bb * kT5Block;
      nv[k] = bb < nblk && my_a >= blo ? min(kT5Block, my_a - blo + 1) : 0;
    }
    // the chunk maximum: each warpgroup over its blocks, then both (the
    // TMEM loads are warp-collective: every lane of a warp takes them)
    float m = -INFINITY;
    if (ok && mine) {
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (wg + 2 * k < nblk) m = fmaxf(m, block_max(tlane, kT5Block * (wg + 2 * k), nv[k]));
    }
    red[wg * kT5Pairs + p] = m;
    __syncthreads();
    const float Mc = fmaxf(red[p], red[kT5Pairs + p]);
    const float mb = Mc > -INFINITY ? -__fmul_rn(Mc, kLog2e) : 0.f;
    __syncthreads();                               // the maxima are read: the sums take their place
    // stage 0: block h into P buffer h (the key tile); stage 1: block 2 into
    // the query tile, block 3 into P buffer 0 once P V of blocks 0, 1 is done
    float lh = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int bb = wg + 2 * k;
      uint8_t* pt = bb == 2 ? qt : kt + (bb & 1) * (kT5Pairs * kRowB);
      bool wok = true;
      if (ok && bb == 3 && bb < nblk) wok = __all_sync(0xffffffffu, mbar_wait(bar_o0, 0));
      if (ok && wok && mine && bb < nblk) lh = __fadd_rn(lh, block_exp(tlane, kT5Block * bb, nv[k], mb, pt, p));
      fence_proxy_async();
      fence_before_sync();
      ok = __syncthreads_and(ok && wok);
      fence_after_sync();
      if (warp == 0 && ok && 2 * k < nblk) {
        // O_c += P_b V_b for the stage's blocks, into columns 0 .. 63
        if (elect_one()) {
          const uint32_t ido = idesc(1, kT5Pairs, kHeadDim, 1);
          for (int b2 = 2 * k; b2 < min(2 * k + 2, nblk); ++b2) {
            const uint64_t dp = b2 == 2 ? dq : dk + (uint64_t)((b2 & 1) * (kT5Pairs * kRowB / 16));
#pragma unroll
            for (int s = 0; s < kT5Block / 16; ++s)
              mma_issue(1, tmem, dp + 2 * s, dv + (uint64_t)((b2 * kT5Block + 16 * s) * (kRowB / 16)), ido,
                        b2 + s ? 1u : 0u);
          }
          mma_commit(k ? bar_o1 : bar_o0);
        }
        __syncwarp();
      }
    }
    red[wg * kT5Pairs + p] = lh;
    // every product done
    ok = __syncthreads_and(ok && mbar_wait(nblk > 2 ? bar_o1 : bar_o0, 0));
    fence_after_sync();
    const float Lc = __fadd_rn(red[p], red[kT5Pairs + p]);
    // the chunk's (O_c, M_c, l_c) of the present pairs: warpgroup h takes
    // dims 32 h .. 32 h + 31.  A tile of one chunk is merged here (merge_chunks
    // of one chunk, whose factor is exp(0) = 1); else they go to the partials.
    const int tp = min(kT5Pairs, b.pm * grp);      // pairs a tile can hold
    float4* part = part_base(D, (size_t)blockIdx.z * D.hkv + g, tp);
    if (ok && mine) {
      uint32_t r[32];
      tmem_ld32_nowait(tlane + 32 * wg, r);
      tmem_wait_ld();
      if (nch == 1) {
        if (p < T.npairs) {
          const size_t off = (size_t)(T.row0 + my_r) * D.hq * kHeadDim + (g * grp + my_h) * kHeadDim + 32 * wg;
          const float l = my_a >= 0 ? __fmaf_rn(Lc, 1.f, 0.f) : 1.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              o[q] = my_a >= 0 ? __fdiv_rn(__fmaf_rn(__uint_as_float(r[4 * i + q]), 1.f, 0.f), l) : 0.f;
            store_out(io, off + 4 * i, make_float4(o[0], o[1], o[2], o[3]));
          }
        }
      } else if (p < T.npairs && my_a >= c_lo) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          __stcg(part + (size_t)(rank * kGroups + 8 * wg + i) * tp + p,
                 make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]),
                             __uint_as_float(r[4 * i + 3])));
        if (wg == 0)
          __stcg(part + (size_t)kT5MaxRanks * kGroups * tp + (size_t)rank * tp + p, make_float4(Mc, Lc, 0.f, 0.f));
      }
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
    if (tid < 32) tmem_dealloc(tmem, kT5Cols);
  }
}

// The prefill merge: CTA (t, g, s) merges pairs 16 s .. 16 s + 15 of tile t
// and KV head g; thread (pair, group) = (tid % 16, tid / 16).
__global__ void __launch_bounds__(kT5Threads) k_attn_merge(Dims D, Batch b, int tps, AttnIO io) {
  const int grp = D.hq / D.hkv;
  const int g = blockIdx.y;
  const T5Tile T = t5_tile(b, grp, tps, blockIdx.x);
  const int p = blockIdx.z * kMergePairs + (threadIdx.x % kMergePairs), i = threadIdx.x / kMergePairs;
  if (T.row0 >= *b.nB) return;
  // the positions were written several launches back; a tile of one chunk was
  // merged, and one of none (all rows past their streams' ends) zeroed, by
  // its attention CTA
  int a_max = b.pos[T.row0 + T.nr - 1];
  for (int r = 1; a_max < 0 && r < T.nr; ++r) a_max = b.pos[T.row0 + T.nr - 1 - r];
  const bool one = a_max < 0 || (a_max - window_start_at(D, a_max)) / kT5Chunk == 0;
  pdl_wait();
  pdl_trigger();
  if (one || p >= T.npairs) return;
  const int my_r = (T.pb + p) / grp, my_h = (T.pb + p) % grp;
  const int a = b.pos[T.row0 + my_r];
  const int ncp = a < 0 ? 0 : (a - window_start_at(D, a)) / kT5Chunk + 1;
  const int tp = min(kT5Pairs, b.pm * grp);
  const float4* part = part_base(D, (size_t)blockIdx.x * D.hkv + g, tp);
  store_out(io, (size_t)(T.row0 + my_r) * D.hq * kHeadDim + (g * grp + my_h) * kHeadDim + 4 * i,
            merge_item(part, tp, p, i, ncp));
}

// Prefill append: row j's k (rotated at its position a) and v, rounded to
// BF16, into the ring of `layer`, and its query heads, rotated, scaled by 1/8
// and rounded to BF16, into q16 (the attention's decode step does the same
// arithmetic for its one row).  A warp takes a row, lane i mod 16 the rotation
// pairs 2 i and 2 i + 1 of every second head, so a position's rotations are
// formed once and all heads' loads are in flight together.  Bound by latency:
// with the loops unrolled for the full model's nine and three heads a launch
// of 4,096 rows takes 8.9 us, with loops over any heads 10.0 (512 rows 8.7 and
// 9.7; GB300, each launch alone and cold).
constexpr int kAppendThreads = 128, kAppendRows = kAppendThreads / 32;
template <int HQ, int HKV>
__global__ void __launch_bounds__(kAppendThreads) k_kv_append_t5(Dims D, Batch b, int layer, const float* qkv) {
  const int hq = HQ ? HQ : D.hq, hkv = HKV ? HKV : D.hkv;
  const int j = blockIdx.x * kAppendRows + (threadIdx.x >> 5), dd = 2 * (threadIdx.x & 15);
  const int half = (threadIdx.x >> 4) & 1;
  pdl_wait();
  pdl_trigger();
  if (j >= *b.nB) return;
  const int a = b.pos[j];
  if (a < 0) return;
  StreamDev& st = b.st[b.slots[j]];
  const float* row = qkv + (size_t)j * D.qkv_rows;
  __nv_bfloat16* ring = static_cast<__nv_bfloat16*>(st.kv) + attn_plane_off(D, layer, 0) +
                        (size_t)(a & (D.L - 1)) * kHeadDim;
  const size_t plane = (size_t)D.L * kHeadDim;
  __nv_bfloat16* q16 = static_cast<__nv_bfloat16*>(D.q16) + (size_t)j * hq * kHeadDim;
  const float2 c0 = rope_cs(D, a, dd), c1 = rope_cs(D, a, dd + 1);
  auto put = [](__nv_bfloat16* dst, float x, float y) { *reinterpret_cast<uint32_t*>(dst) = pack_bf16(x, y); };
#pragma unroll
  for (int i = 0; i < (hq + hkv + 1) / 2; ++i) {   // the query heads, then the keys
    const int h = 2 * i + half;
    if (h >= hq + hkv) break;
    const float* src = row + h * kHeadDim + dd;
    const float2 x = __ldcg(reinterpret_cast<const float2*>(src));
    const float2 y = __ldcg(reinterpret_cast<const float2*>(src + kHeadDim / 2));
    const float2 r0 = rope_rotate(x.x, y.x, c0), r1 = rope_rotate(x.y, y.y, c1);
    if (h < hq) {
      put(q16 + h * kHeadDim + dd, r0.x * 0.125f, r1.x * 0.125f);
      put(q16 + h * kHeadDim + dd + kHeadDim / 2, r0.y * 0.125f, r1.y * 0.125f);
    } else {
      __nv_bfloat16* dst = ring + (size_t)(h - hq) * plane + dd;
      put(dst, r0.x, r1.x);
      put(dst + kHeadDim / 2, r0.y, r1.y);
    }
  }
#pragma unroll
  for (int i = 0; i < (hkv + 1) / 2; ++i) {
    const int h = 2 * i + half;
    if (h >= hkv) break;
    const float4 v = __ldcg(reinterpret_cast<const float4*>(row + (hq + hkv + h) * kHeadDim + 2 * dd));
    *reinterpret_cast<uint2*>(ring + (size_t)(hkv + h) * plane + 2 * dd) =
        make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
  }
}

}  // namespace

size_t attn_t5_scratch(const Dims& D, int prefill_rows) {
  const int grp = D.hq / D.hkv;
  // a prefill chunk of n streams and m <= prefill_rows / n positions each
  // takes n ceil(m grp / 128) tiles of min(128, m grp) pairs: at most
  // 2 prefill_rows grp pairs (n < 128 prefill_rows / (m grp 128) when m grp > 128)
  const size_t pf_pairs = prefill_rows >= 2 ? 2 * (size_t)prefill_rows * grp : 0;
  return pf_pairs * (size_t)D.hkv * kT5MaxRanks * kPartRow;
}

cudaError_t prepare_attn_t5() {                    // the limit of the current device's context
  return cudaFuncSetAttribute(k_attn_t5, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kT5Smem);
}

cudaError_t launch_attn_t5(const Dims& D, const Batch& b, int layer, const float* qkv, float* attn_out, void* out16,
                           cudaStream_t s) {
  if (!b.pos) return launch_attn_dec(D, b, layer, qkv, attn_out, out16, s);
  if (!D.attn_part || !D.q16) return cudaErrorInvalidValue;
  const int grp = D.hq / D.hkv;
  if (grp > kT5Pairs) return cudaErrorInvalidValue;
  const int tps = (b.pm * grp + kT5Pairs - 1) / kT5Pairs, tiles = (b.Bmax / b.pm) * tps;
  const size_t tp = std::min(kT5Pairs, b.pm * grp);
  if ((size_t)tiles * D.hkv * kT5MaxRanks * tp * kPartRow > D.attn_part_cap) return cudaErrorInvalidValue;
  const AttnIO io{qkv, attn_out, out16};
  // chunks of the longest window of the launch: a CTA without a chunk costs
  // its launch and three dependent loads, more than a third of the kernel
  // when all eight were launched for windows of one
  const int64_t len = b.len_max > 0 && b.len_max < D.L ? b.len_max : D.L;
  const int nch = (int)((len + kT5Chunk - 1) / kT5Chunk);
  cudaError_t e = launch_kernel(k_attn_t5, dim3(nch, D.hkv, tiles), dim3(kT5Threads), kT5Smem, s, D.pdl, D, b,
                                layer, tps, io);
  if (e == cudaSuccess && nch > 1)
    e = launch_kernel(k_attn_merge, dim3(tiles, D.hkv, kT5Pairs / kMergePairs), dim3(kT5Threads), 0, s, D.pdl, D, b,
                      tps, io);
  return e;
}

cudaError_t launch_kv_append_t5(const Dims& D, const Batch& b, int layer, const float* qkv, cudaStream_t s) {
  if (!D.q16) return cudaErrorInvalidValue;
  const dim3 grid((b.Bmax + kAppendRows - 1) / kAppendRows);
  if (D.hq == 9 && D.hkv == 3)                     // the full model's heads: the loops unrolled
    return launch_kernel(k_kv_append_t5<9, 3>, grid, dim3(kAppendThreads), 0, s, D.pdl, D, b, layer, qkv);
  return launch_kernel(k_kv_append_t5<0, 0>, grid, dim3(kAppendThreads), 0, s, D.pdl, D, b, layer, qkv);
}

}  // namespace nc
