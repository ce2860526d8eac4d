// Nearest-parent search with the tensor cores as a filter (Sec. IV-E
// "Parents"), exact in its result.
//
// The squared distance of query q and node n under the velocity weight w is
// |q'|^2 + (|n'|^2 - 2 q'.n') with x' = (positions, sqrt(w) velocities).  The
// bracket, the pair's score, is a contraction (knn_scales may shrink x' by a power
// of two, which changes no digit of it): each value is split into two
// f16 terms (hi + lo, 22 bits), the cross products hi hi, hi lo and lo hi of
// the 14 components and the node's squared norm in three f16 terms make a
// row of KT_K = 48 columns, and tcgen05.mma scores 128 nodes against 128
// queries at a time.  Three steps:
//   pack    nodes and queries into operand images (knn_pack_node / _query)
//   mins    every (query, group of 32 consecutive nodes): the least score of
//           the group, read from tensor memory (knn_mins)
//   select  a warp per query: groups that can hold one of its k nearest
//           nodes, by the score's error bound, are scored exactly in FP32
//           (knn_dist's operations in their order) and kept in (d, index)
//           order (knn_select)
// so the list is the one the full FP32 scan gives, ties and all.
//
// Error bound.  With f = |q'| + |n'|: dropped products and split remainders
// at most 3 2^-22 2 |q'||n'|, the FP32 sums of 48 products 2^-18.3 f^2 at
// worst, the norm 2^-21 |n'|^2, the exact distance's own rounding 2^-20 f^2;
// in all less than KT_C f^2 with KT_C = 2^-16, plus KT_ABS for f16's
// subnormal range.  Since |n'| <= |q'| + sqrt(d), f^2 <= 8 |q'|^2 + 2 d.
// If k groups have least scores up to tau, k nodes have d <= Dmax =
// (tau + |q'|^2 + 8 C |q'|^2 + ABS) / (1 - 2 C), and every node with d <=
// Dmax has a score of at most Dmax (1 + 2 C) + 8 C |q'|^2 + ABS - |q'|^2.
//
// States outside the split's range (not finite, or |x'|^2 > KT_MAX2) never
// depend on a score: such a node gets a score below KT_FORCED, which makes
// its group one that is always scored exactly and never counted towards
// tau, and such a query scores every group exactly.  Rows past the last
// node score above KT_EMPTY.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "fn_umma.cuh"
#include "knn_core.cuh"

namespace fn {

constexpr int KT_K = 48;                           // operand columns
constexpr int KT_ROWS = 128;                       // rows of an operand tile
constexpr int KT_TILE = KT_ROWS * KT_K * 2;        // 12 KB
constexpr int KT_QT = 2 * KT_ROWS;                 // queries per work unit
constexpr int KT_GROUP = 32;                       // nodes per group
constexpr float KT_MAX2 = 16384.f;
constexpr float KT_FORCED = -1e5f, KT_EMPTY = 1e5f;
constexpr float KT_C = 1.52587890625e-5f;          // 2^-16
constexpr float KT_ABS = 9.5367431640625e-7f;      // 2^-20
constexpr int KT_RING = 4;                         // node tiles in flight
constexpr int KT_WARPS = 16;                       // read-back warps
constexpr int KT_THREADS = 32 * (KT_WARPS + 2);    // and the MMA warp, the copy warp
constexpr int KT_BLK = 16;                         // node tiles per block of a row of minima
constexpr int kKtBars = 2 * KT_RING + 2 + 2 + 2;   // tile full / free, A full, D full / free
constexpr int kKtOffB = 2 * 2 * KT_TILE;           // after two query images
constexpr int kKtOffOut = kKtOffB + KT_RING * KT_TILE;      // minima waiting to be written
constexpr int kKtOffBar = kKtOffOut + KT_WARPS * 32 * 33 * 4;
constexpr int kKtSmem = kKtOffBar + kKtBars * 8 + 16;       // above half an SM's: one CTA
static_assert(kKtSmem > 120 * 1024 && kKtSmem <= 227 * 1024, "one CTA per SM (all of TMEM)");

// instruction descriptor: FP32 accumulator, f16 operands, both K-major, 128 x 128
constexpr uint32_t kKtIdesc = (1u << 4) | ((uint32_t)(KT_ROWS >> 3) << 17) |
                              ((uint32_t)(KT_ROWS >> 4) << 24);

__device__ __forceinline__ uint32_t h2(__half a, __half b) {
  return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

// one operand row (48 halfs) into its place of a tile image: 8 x 8 core
// matrices of 128 B, K-adjacent ones 128 B apart, 8-row groups 768 B apart
__device__ __forceinline__ void knn_store_row(uint8_t* tile, int r, const __half (&v)[KT_K]) {
  uint8_t* p = tile + (r >> 3) * (KT_K / 8) * 128 + (r & 7) * 16;
#pragma unroll
  for (int c = 0; c < KT_K / 8; ++c)
    *reinterpret_cast<uint4*>(p + c * 128) =
        make_uint4(h2(v[8 * c], v[8 * c + 1]), h2(v[8 * c + 2], v[8 * c + 3]),
                   h2(v[8 * c + 4], v[8 * c + 5]), h2(v[8 * c + 6], v[8 * c + 7]));
}

// Scales (position, velocity) = c (1, sqrt(w)) of x', c the largest power of two up
// to 1 that brings states with |q|^2 + w |qd|^2 <= r2 into the split's range (not
// below 2^-50: distances of states in range stay finite in FP32, as those that
// overflow tie).
// A weight of 1e4 without it leaves every node to the exact scores: 60000 nodes and
// 256 queries 1175 us, now 44.
inline float2 knn_scales(float w, double r2) {
  float c = 1.f;
  if (r2 < INFINITY)
    while (c > 1e-15f && (double)c * c * r2 > KT_MAX2) c *= 0.5f;
  return make_float2(c, c * std::sqrt(w));
}

// x' and |x'|^2 of a state; returns whether the split covers it
__device__ __forceinline__ bool knn_scaled(const float* x, float2 sc, float (&s)[14], float& n2) {
  n2 = 0.f;
#pragma unroll
  for (int j = 0; j < 14; ++j) {
    s[j] = (j < 7 ? sc.x : sc.y) * x[j];
    n2 = fmaf(s[j], s[j], n2);
  }
  return n2 <= KT_MAX2;   // false for NaN
}

// present = false: a row past the last node (x unused)
__device__ __forceinline__ void knn_pack_node(uint8_t* tile, int r, const float* x, float2 sc,
                                              bool present) {
  __half v[KT_K];
#pragma unroll
  for (int j = 0; j < KT_K; ++j) v[j] = __float2half_rn(0.f);
  float s[14], n2 = 0.f;
  const bool in = present && knn_scaled(x, sc, s, n2);
  if (in) {
#pragma unroll
    for (int j = 0; j < 14; ++j) {
      const __half hi = __float2half_rn(s[j]);
      v[j] = hi;
      v[14 + j] = __float2half_rn(s[j] - __half2float(hi));
      v[28 + j] = hi;
    }
    v[42] = __float2half_rn(n2);
    const float r1 = n2 - __half2float(v[42]);
    v[43] = __float2half_rn(r1);
    v[44] = __float2half_rn(r1 - __half2float(v[43]));
  } else {
    v[42] = v[43] = v[44] = __float2half_rn(present ? -65504.f : 65504.f);
  }
  knn_store_row(tile, r, v);
}
__device__ __forceinline__ void knn_pack_query(uint8_t* tile, int r, const float* x, float2 sc,
                                               bool present) {
  __half v[KT_K];
#pragma unroll
  for (int j = 0; j < KT_K; ++j) v[j] = __float2half_rn(0.f);
  float s[14], n2;
  if (present && knn_scaled(x, sc, s, n2)) {
#pragma unroll
    for (int j = 0; j < 14; ++j) {
      const float a = -2.f * s[j];
      const __half hi = __float2half_rn(a);
      v[j] = v[14 + j] = hi;
      v[28 + j] = __float2half_rn(a - __half2float(hi));
    }
    v[42] = v[43] = v[44] = __float2half_rn(1.f);
  }
  knn_store_row(tile, r, v);
}

__device__ __forceinline__ float min3f(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// least of a group's 32 scores
__device__ __forceinline__ float min32(const uint32_t (&v)[32]) {
  float m = __uint_as_float(v[0]);
#pragma unroll
  for (int j = 1; j < 31; j += 2) m = min3f(m, __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
  return fminf(m, __uint_as_float(v[31]));
}

// A query's row of group minima: four words (a float4) per node tile, in
// blocks of KT_BLK tiles, the even tiles first, then the odd ones, as the
// two sets of warps that read the accumulators back write them.
__host__ __device__ __forceinline__ int kt_row_f4(int ntiles) {
  return (ntiles + KT_BLK - 1) / KT_BLK * KT_BLK;
}
// tile of float4 j of a row (tiles past the last one are not written)
__device__ __forceinline__ int kt_f4_tile(int j) {
  return (j & ~(KT_BLK - 1)) + ((j & (KT_BLK / 2 - 1)) << 1) + ((j >> 3) & 1);
}
static_assert(KT_BLK == 16, "kt_f4_tile");

// A run of work units: 256 queries (two operand tiles at a) against node
// tiles nt .. nt + left of a tree (b: tile nt); the rows of minima are at
// g + r * stride for r < rows.
struct KtUnit {
  const uint8_t* a;
  const uint8_t* b;
  float* g;
  long stride;
  int rows, nt, left;
};

// Units [u0, u1) (pairs of 256 queries and a node tile) on one CTA of
// KT_THREADS; W(u) gives the run that starts at unit u.  Warp 17's first lane
// streams node tiles (cp.async.bulk, a ring of KT_RING) and query images
// (two), warp 16's issues the MMAs into the accumulator pair (2 x 128
// columns each; both: all of tensor memory) of the tile's parity, and warps
// 0-15 read them back (warp w: tiles of parity w / 8, lane quarter w % 4 of
// the query half (w / 4) % 2) and reduce them, one three-input minimum per
// two scores.  Sharing a node tile between two query halves keeps the
// operand traffic (12 KB per 256 x 128 scores) below what L2 gives; two sets
// of eight warps, so that one set's tensor-memory loads overlap the other's
// minima (one set on every tile: 76 us, 8192 queries on 65536 nodes; two:
// 71).  What is left is the round trip of an accumulator pair (MMA, commit,
// load, release; the MMAs alone take 25 us).  A thread holds a query's row, so its four minima per tile go through
// shared memory and leave as rows of up to 32 words.  Waits are bounded: on
// a timeout *err is raised and the select step scores every group exactly.
template <class Work>
__device__ __forceinline__ void knn_mins(uint8_t* smem, const Work& W, long u0, long u1,
                                         int* err) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (u0 >= u1) return;                               // block-uniform
  const uint32_t base = su32(smem), bar0 = base + kKtOffBar;
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(smem + kKtOffBar + kKtBars * 8);
  volatile int* s_fail = reinterpret_cast<volatile int*>(s_tmem + 1);
  auto b_full = [&](int s) { return bar0 + 8u * s; };
  auto b_free = [&](int s) { return bar0 + 8u * (KT_RING + s); };
  auto a_full = [&](int s) { return bar0 + 8u * (2 * KT_RING + s); };
  auto d_full = [&](int s) { return bar0 + 8u * (2 * KT_RING + 2 + s); };
  auto d_free = [&](int s) { return bar0 + 8u * (2 * KT_RING + 4 + s); };
  if (warp == KT_WARPS) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32((const void*)s_tmem)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < 2 * KT_RING + 4; ++i) mbar_init(bar0 + 8u * i, 1);
    for (int i = 0; i < 2; ++i) mbar_init(d_free(i), KT_WARPS / 2);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  auto run = [&](const KtUnit& t, long u) { return (int)min((long)t.left + 1, u1 - u); };
  if (warp == KT_WARPS + 1) {
    if (lane == 0) {
      int i = 0;             // node tiles requested
      int done = 0;          // of them, read by their MMAs
      int seg = 0;           // query images requested
      int seg_last = 0;      // node tiles requested when the newest image was
      bool ok = true;
      auto wait_done = [&](int upto) {   // the first upto tiles' MMAs have completed
        for (; ok && done < upto; done += ok)
          ok = mbar_wait(b_free(done % KT_RING), (done / KT_RING) & 1, s_fail);
      };
      for (long u = u0; ok && u < u1;) {
        const KtUnit t = W(u);
        const int n = run(t, u);
        wait_done(seg_last);             // the image two back is no longer read
        if (!ok) break;
        seg_last = i;
        mbar_expect_tx(a_full(seg & 1), 2 * KT_TILE);
        bulk_g2s(base + (seg & 1) * 2 * KT_TILE, t.a, 2 * KT_TILE, a_full(seg & 1));
        ++seg;
        for (int c = 0; c < n; ++c, ++i) {
          wait_done(i - KT_RING + 1);
          if (!ok) break;
          mbar_expect_tx(b_full(i % KT_RING), KT_TILE);
          bulk_g2s(base + kKtOffB + (i % KT_RING) * KT_TILE, t.b + (long)c * KT_TILE, KT_TILE,
                   b_full(i % KT_RING));
        }
        u += n;
      }
      // the copies end before the shared memory goes away
      for (int l = max(0, i - KT_RING); l < i; ++l)
        mbar_wait(b_full(l % KT_RING), (l / KT_RING) & 1);
      for (int l = max(0, seg - 2); l < seg; ++l) mbar_wait(a_full(l & 1), (l >> 1) & 1);
    }
    __syncwarp();
  } else if (warp == KT_WARPS) {
    if (lane == 0) {
      // descriptors differ in the start address only (16-byte units, below
      // 2^14: shared memory ends before any carry)
      const uint64_t desc0 = sdesc(base, 128, (KT_K / 8) * 128);
      int i = 0, seg = 0, use[2] = {0, 0};
      bool ok = true;
      for (long u = u0; ok && u < u1; ++seg) {
        const KtUnit t = W(u);
        const int n = run(t, u);
        u += n;
        ok = mbar_wait(a_full(seg & 1), (seg >> 1) & 1, s_fail);
        const uint64_t da = desc0 + (uint32_t)((seg & 1) * 2 * KT_TILE >> 4);
        for (int c = 0; ok && c < n; ++c) {
          const int p = (t.nt + c) & 1, use_p = p ? use[1] : use[0];
          if (use_p > 0) ok = mbar_wait(d_free(p), (use_p - 1) & 1, s_fail);
          if (ok) ok = mbar_wait(b_full(i % KT_RING), (i / KT_RING) & 1, s_fail);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)p * 2 * KT_ROWS;
          const uint64_t db = desc0 + (uint32_t)((kKtOffB + (i % KT_RING) * KT_TILE) >> 4);
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < KT_K / 16; ++k)
              umma_f16(d + h * KT_ROWS, da + ((h * KT_TILE + k * 256) >> 4), db + (k * 256 >> 4),
                       kKtIdesc, k > 0);
          umma_commit(d_full(p));
          umma_commit(b_free(i % KT_RING));
          if (p) ++use[1];
          else ++use[0];
          ++i;
        }
      }
      // every issued MMA ends before tensor memory and the operands go away
      if (i > 0) mbar_wait(b_free((i - 1) % KT_RING), ((i - 1) / KT_RING) & 1);
    }
    __syncwarp();
  } else {
    const int half = (warp >> 2) & 1, par = warp >> 3;
    const int row0 = half * KT_ROWS + (warp & 3) * 32;      // the warp's first query row
    const uint32_t at =
        tmem + ((uint32_t)((warp & 3) * 32) << 16) + (2 * par + half) * KT_ROWS;
    float* out = reinterpret_cast<float*>(smem + kKtOffOut) + warp * 32 * 33;   // [32][33]
    const uint32_t full = d_full(par), free = d_free(par);
    uint32_t phase = 0;
    bool ok = true;
    for (long u = u0; ok && u < u1;) {
      const KtUnit t = W(u);
      const int n = run(t, u), end = t.nt + n, rows = t.rows - row0;
      u += n;
      float* g = t.g + row0 * t.stride + 32 * par;
      int nt = t.nt + ((t.nt ^ par) & 1), lo = 4 * ((nt & (KT_BLK - 1)) >> 1);
      for (; nt < end; nt += 2) {
        ok = mbar_wait(full, phase, s_fail);
        phase ^= 1u;
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        tc_fence_after();
        uint32_t v0[32], v1[32], v2[32], v3[32];
        tmem_ld32_async(at, v0);
        tmem_ld32_async(at + 32, v1);
        tmem_ld32_async(at + 64, v2);
        tmem_ld32_async(at + 96, v3);
        tmem_ld_wait();
        tmem_use(v0); tmem_use(v1); tmem_use(v2); tmem_use(v3);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(free);
        const int hi = 4 * ((nt & (KT_BLK - 1)) >> 1) + 4;
        float* o = out + lane * 33 + hi - 4;
        o[0] = min32(v0);
        o[1] = min32(v1);
        o[2] = min32(v2);
        o[3] = min32(v3);
        if (hi == 32 || nt + 2 >= end) {                    // the block or the run ends
          float* gb = g + (nt / KT_BLK) * (4 * KT_BLK);
          const int wd = hi - lo;
          __syncwarp();
          if (wd == 32) {
            float* gl = gb + lane;
#pragma unroll 8
            for (int r = 0; r < 32; ++r, gl += t.stride)
              if (r < rows) *gl = out[r * 33 + lane];
          } else {
            for (int x = lane; x < 32 * wd; x += 32) {
              const int r = x / wd, c = lo + x - r * wd;
              if (r < rows) gb[r * t.stride + c] = out[r * 33 + c];
            }
          }
          __syncwarp();
          lo = 0;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*s_fail && tid == 0) atomicExch(err, 1);
  tc_fence_after();
  if (warp == KT_WARPS)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// ---------------------------------------------------------------------------
// select
// ---------------------------------------------------------------------------
// (d, index) as one ordered word: d >= 0, so its bits order as it does
__device__ __forceinline__ unsigned long long knn_key(float d, int i) {
  return ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)i;
}
constexpr unsigned long long KT_NONE = (0x7f800000ull << 32) | 0x7fffffffull;   // (inf, max)

__device__ __forceinline__ unsigned long long knn_cas(unsigned long long x, int o, bool lo) {
  const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
  return (x < y) == lo ? x : y;
}

// The warp's list of the k <= 16 best keys, ascending on lanes 0 .. k - 1
// (other lanes hold worse ones); only keys below kth enter: the k-th entry,
// or a bound that at least k nodes are known to meet.
struct KeyList {
  unsigned long long key = KT_NONE, kth = KT_NONE;
  // offer one key per lane (KT_NONE where a lane has none)
  __device__ __forceinline__ void offer(unsigned long long c, int k) {
    const int lane = threadIdx.x & 31;
    unsigned m = __ballot_sync(0xffffffffu, c < kth);
    if (__popc(m) > 5) {
      // sort the 32 offered keys, then merge: the 16 least of an ascending
      // and a descending run of 16 form a bitonic run
#pragma unroll
      for (int s = 2; s <= 32; s <<= 1)
#pragma unroll
        for (int o = s >> 1; o > 0; o >>= 1)
          c = knn_cas(c, o, ((lane & o) == 0) == ((lane & s) == 0));
      const unsigned long long r = __shfl_sync(0xffffffffu, c, 15 - (lane & 15));
      if (lane < 16 && r < key) key = r;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) key = knn_cas(key, o, (lane & o) == 0);
    } else {
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1u;
        const unsigned long long x = __shfl_sync(0xffffffffu, c, src);
        const int pos = __popc(__ballot_sync(0xffffffffu, key < x) & 0xffffu);
        const unsigned long long up = __shfl_up_sync(0xffffffffu, key, 1);
        key = lane < pos ? key : (lane == pos ? x : up);
      }
    }
    const unsigned long long x = __shfl_sync(0xffffffffu, key, k - 1);
    if (x < kth) kth = x;
  }
};

// ascending order of floats as unsigned words
__device__ __forceinline__ unsigned knn_order(float x) {
  const unsigned u = __float_as_uint(x);
  return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float knn_unorder(unsigned u) {
  return __uint_as_float(u ^ ((u >> 31) ? 0x80000000u : 0xffffffffu));
}

// Exact scores read the nodes from a second image: per group of 32 nodes
// [7][32] float2, joint by joint (position, velocity), so that a warp's seven
// loads of a group are contiguous (from the 64-byte rows of the tree a load
// touches sixteen lines).
constexpr int KT_SOA = 7 * KT_GROUP;   // float2 per group
__device__ __forceinline__ void knn_store_soa(float2* soa, long node, const float* x) {
  float2* p = soa + node / KT_GROUP * KT_SOA + node % KT_GROUP;
#pragma unroll
  for (int c = 0; c < 7; ++c) p[KT_GROUP * c] = make_float2(x[c], x[7 + c]);
}
__device__ __forceinline__ float knn_dist(const float* qv, const float2 (&x)[7], float w) {
  float dq = 0.f, dv = 0.f;
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    const float t = qv[c] - x[c].x, u = qv[7 + c] - x[c].y;
    dq = fmaf(t, t, dq);
    dv = fmaf(u, u, dv);
  }
  return fmaf(w, dv, dq);
}
// the same with the two sums as the halves of paired operations, from the negated
// query ((x - q)^2 is (q - x)^2): half the instructions, for a loop they bound
__device__ __forceinline__ float knn_dist2(const float2 (&nq)[7], const float2 (&x)[7], float w) {
  float2 d = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < 7; ++c) {
    const float2 t = __fadd2_rn(x[c], nq[c]);
    d = __ffma2_rn(t, t, d);
  }
  return fmaf(w, d.y, d.x);
}

// The k nearest of n nodes (their image soa, ids from id0 on) to a query
// from its row g of group minima over ntiles node tiles: lanes 0 .. k - 1 of
// the returned list hold the keys.  all: the scores are not to be used.
// list: KT_LIST words of the warp's own.  Groups in reach are collected
// first and scored nearest first, the reach shrinking with the k-th distance
// found so far (about k + 2 groups are scored).  A group at a time in 64
// registers: the loads' latency is hidden by 32 warps an SM rather than by
// several groups in flight (8192 queries, 65536 nodes, k = 16: 50 us; two
// groups at a time with 16 warps an SM 69 us).
// kWide: *wide is set when the scores do not tell the nodes apart, which is looked
// at once when KT_TRIAL groups have been gone through: a quarter of all groups are in
// reach still.  The list is then empty but for its bound, and knn_wide does the
// search.  (A query that stays here may still score up to that quarter.)  Without
// kWide such a query scores the groups one by one, a warp for itself.
constexpr int KT_LIST = 160, KT_TRIAL = 64;
template <bool kWide>
__device__ __forceinline__ KeyList knn_select(const float2* __restrict__ soa, int n, int id0,
                                              const float4* __restrict__ query, int k, float w,
                                              float2 sc, const float* __restrict__ g, int ntiles,
                                              bool all, unsigned long long* list,
                                              bool* wide = nullptr) {
  const int lane = threadIdx.x & 31;
  float qv[14], q2;
  load_query(query, qv);
  {
    float sq[14];
    all |= !knn_scaled(qv, sc, sq, q2);
  }
  KeyList best;
  if (kWide && all) {
    *wide = true;
    return best;
  }
  const float4* g4 = reinterpret_cast<const float4*>(g);
  const int n4 = kt_row_f4(ntiles);
  // the four groups of the tile of float4 j; whether there is one
  auto load4 = [&](int j, float (&x)[4]) {
    const bool have = j < n4 && kt_f4_tile(j) < ntiles;
    float4 v = make_float4(NAN, NAN, NAN, NAN);
    if (have) v = __ldcg(g4 + j);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    return have;
  };
  // tau: the k-th least of the lanes' least group minima (each a node of its own)
  float m = INFINITY;
#pragma unroll 4
  for (int b = 0; b < n4; b += 32) {
    float x[4];
    load4(b + lane, x);
#pragma unroll
    for (int c = 0; c < 4; ++c) m = fminf(m, x[c] > KT_FORCED ? x[c] : INFINITY);
  }
#pragma unroll
  for (int s = 2; s <= 32; s <<= 1)
#pragma unroll
    for (int o = s >> 1; o > 0; o >>= 1) {
      const float y = __shfl_xor_sync(0xffffffffu, m, o);
      m = ((lane & o) == 0) == ((lane & s) == 0) ? fminf(m, y) : fmaxf(m, y);
    }
  const float tau = __shfl_sync(0xffffffffu, m, k - 1);
  const float slack = fmaf(8.f * KT_C, q2, KT_ABS);
  const float c2 = sc.x * sc.x;   // of a scaled squared distance
  // largest score of a node at (scaled) distance at most D
  auto reach = [&](float D) { return fmaf(D, 1.f + 2.f * KT_C, slack - q2) + 1e-6f * q2; };
  float lim = INFINITY;
  if (!all && tau < KT_EMPTY) {
    // (rounded up by the last factor) at least k nodes are this near
    const float dmax = (fmaxf(tau + q2, 0.f) + slack) / (1.f - 2.f * KT_C) * (1.f + 1e-6f);
    lim = reach(dmax);
    best.kth = knn_key(dmax / c2, 0x7fffffff);   // farther nodes need not enter the list
  }
  int cnt = 0, scored = 0;   // groups collected, gone through
  bool tried = false, give_up = false;
  auto useless = [&]() {     // do the scores leave a quarter of the groups in reach?
    int in = 0;
#pragma unroll 1
    for (int b = 0; b < n4; b += 32) {
      float x[4];
      load4(b + lane, x);
#pragma unroll
      for (int c = 0; c < 4; ++c) in += __popc(__ballot_sync(0xffffffffu, x[c] <= lim));
    }
    return in > ntiles;
  };
  auto flush = [&]() {
    __syncwarp();
    if (kWide && scored >= KT_TRIAL && !tried) {
      tried = true;
      give_up = useless();
      if (give_up) {
        lim = -INFINITY;     // nothing more is collected
        cnt = 0;
      }
    }
    scored += cnt;
    for (int f = 0; f < cnt; f += 32) {
      const int ne = min(32, cnt - f);
      unsigned long long e = lane < ne ? list[f + lane] : ~0ull;
      if (ne > 1)
#pragma unroll
        for (int s = 2; s <= 32; s <<= 1)
#pragma unroll
          for (int o = s >> 1; o > 0; o >>= 1)
            e = knn_cas(e, o, ((lane & o) == 0) == ((lane & s) == 0));
      for (int j = 0; j < ne; ++j) {
        // sorted scores: nothing further is in reach once one is not (scores
        // that force a group are below any reach)
        const unsigned long long ej = __shfl_sync(0xffffffffu, e, j);
        if (!all && knn_unorder((unsigned)(ej >> 32)) > lim) break;
        const unsigned gr = (unsigned)ej;
        const int node = (int)gr * KT_GROUP + lane;
        unsigned long long key = KT_NONE;
        if (node < n) {
          float2 x[7];
#pragma unroll
          for (int v = 0; v < 7; ++v) x[v] = __ldg(soa + (long)gr * KT_SOA + KT_GROUP * v + lane);
          const float d = knn_dist(qv, x, w);
          if (d <= INFINITY) key = knn_key(d, id0 + node);   // a NaN distance never enters
        }
        best.offer(key, k);
        if (!all) lim = fminf(lim, reach(c2 * __uint_as_float((unsigned)(best.kth >> 32))));
      }
    }
    cnt = 0;
    __syncwarp();
  };
#pragma unroll 2
  for (int b = 0; b < n4; b += 32) {
    float x[4];
    const bool have = load4(b + lane, x);
    bool in[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) in[c] = all ? have : x[c] <= lim;
    if (__any_sync(0xffffffffu, in[0] || in[1] || in[2] || in[3])) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const unsigned m = __ballot_sync(0xffffffffu, in[c]);
        if (in[c])
          list[cnt + __popc(m & ((1u << lane) - 1u))] =
              ((unsigned long long)knn_order(x[c]) << 32) |
              (unsigned)(4 * kt_f4_tile(b + lane) + c);
        cnt += __popc(m);
      }
      if (cnt >= 32) flush();
    }
  }
  if (cnt) flush();
  if (kWide) *wide = give_up;
  if (give_up) {       // start again; the k-th key so far is one of those to find
    best.key = KT_NONE;
    best.kth += best.kth < KT_NONE;
  }
  return best;
}

// The exact scan of all nodes, for the queries whose scores are of no use: node
// states that nearly coincide, states outside the filter's range.  Every warp of a
// block of NW calls this (it synchronises) and gets its list, best unless wide is set.
// The block copies kGroups groups at a time into shared memory (cp.async, a ring of
// kStages) and each of its wide queries scores them from there; `team`
// neighbouring warps share a query (the first one's wide and best count), a group
// in turn each.  The loop is bound by issue, hence the paired distance.  A warp
// reading every group for itself took, 8192 queries of a tree of 65536 equal nodes,
// 2780 us (L2 bandwidth), one such query 1280 us (latency); now 1441 and 199 (the
// scan of fn_knn.cu, without the filter before it, 1145 and 130).
// kStages, kGroups: for a query to a warp two stages of four groups, 15 KB a block
// that leave ordinary searches of small trees their L1 (three of eight, 44 KB: 20000
// queries on 2000 nodes 89 us, so 86); three of eight for shared queries, whose scan
// is bound by latency (one query on 65536 nodes 257 -> 150 us).
template <int NW, int kGroups, int kStages>
struct KnnWide {
  union {
    unsigned long long list[NW][KT_LIST];            // knn_select's
    float4 stage[kStages][kGroups * KT_SOA / 2];
    unsigned long long key[NW][16];
  };
  int wide[NW];
};
template <int NW, int kGroups, int kStages>
__device__ __forceinline__ KeyList knn_wide(KnnWide<NW, kGroups, kStages>& sh, KeyList best,
                                            bool wide, int team, const float2* soa, int n, int id0,
                                            const float4* query, int k, float w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rank = warp % team;
  if (!__syncthreads_or(rank == 0 && wide)) return best;
  if (lane == 0 && rank == 0) sh.wide[warp] = wide;
  if (rank != 0) best = KeyList{};
  __syncthreads();
  const bool mine = sh.wide[warp - rank] != 0;
  float2 nq[7];
  if (mine) {
    float qv[14];
    load_query(query, qv);
#pragma unroll
    for (int c = 0; c < 7; ++c) nq[c] = make_float2(-qv[c], -qv[7 + c]);
  }
  constexpr int kF4 = KT_SOA / 2;              // of a group
  const int groups = (n + KT_GROUP - 1) / KT_GROUP, chunks = (groups + kGroups - 1) / kGroups;
  auto copy = [&](int c) {                     // one commit group, empty past the end
    if (c < chunks) {
      const int have = min(kGroups, groups - c * kGroups) * kF4;
      const float4* src = reinterpret_cast<const float4*>(soa) + (long)c * kGroups * kF4;
      const uint32_t dst = su32(sh.stage[c % kStages]);
      for (int i = threadIdx.x; i < have; i += 32 * NW)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16 * i),
                     "l"(src + i)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  for (int c = 0; c < kStages - 1; ++c) copy(c);
  for (int c = 0; c < chunks; ++c) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kStages - 2) : "memory");
    __syncthreads();                           // chunk c is there, c - 1 is scored
    copy(c + kStages - 1);
    if (!mine) continue;
    const float2* st = reinterpret_cast<const float2*>(sh.stage[c % kStages]) + lane;
    const int have = min(kGroups, groups - c * kGroups);
    for (int i = rank; i < have; i += team) {
      const int node = (c * kGroups + i) * KT_GROUP + lane;
      float2 x[7];
#pragma unroll
      for (int j = 0; j < 7; ++j) x[j] = st[i * KT_SOA + KT_GROUP * j];
      const float d = knn_dist2(nq, x, w);
      const unsigned long long key =
          node < n && d <= INFINITY ? knn_key(d, id0 + node) : KT_NONE;
      if (__any_sync(0xffffffffu, key < best.kth)) best.offer(key, k);
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  if (team > 1) {
    __syncthreads();                           // the last chunk is scored
    if (lane < 16) sh.key[warp][lane] = best.key;
    __syncthreads();
    if (rank == 0 && mine)
      for (int r = 1; r < team; ++r) best.offer(lane < 16 ? sh.key[warp + r][lane] : KT_NONE, k);
  }
  return best;
}

}  // namespace fn
