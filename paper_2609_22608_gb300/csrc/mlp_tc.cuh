// What the surrogate's tcgen05 kernels (inference and training) share: the
// shared-memory map of a 128-edge tile, its feature rows and the ring that
// streams the packed weights.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "fn_mlp_tc.h"
#include "fn_umma.cuh"

namespace fn {

typedef __nv_bfloat16 bf16;

// shared memory map (bytes)
constexpr int kSA = 0;                          // A operand: 128 x 256 bf16 (64 KB)
constexpr int kSB = 65536;                      // weight ring: 4 x 32 KB
constexpr int kSW1 = kSB + 4 * kTcChunkBytes;   // packed W1 (16 KB)
constexpr int kSBias = kSW1 + kTcW1Bytes;       // b1, b2, b3 (3 x 256 f32)
constexpr int kSW4 = kSBias + 3 * 256 * 4;      // W4 [256][2] f32
constexpr int kSBar = kSW4 + 512 * 4;           // mbarriers + TMEM address
constexpr int kSY = kSBar + 128;                // layer-4 partial sums [4][128][2] f32
constexpr int kTcSmem = kSY + 4 * kTcM * 2 * 4;

// 16 warps: warp w reads TMEM lane quarter w % 4 (the tcgen05 access rule)
// and column group w / 4 (64 of the 256 accumulator columns) in the
// epilogues, so that four warps share each scheduler.
constexpr int kTcThreads = 512;

constexpr int kRing = 4;
constexpr int kTmemCols = 256;
// instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator,
// bf16 A and B, both K-major, N = 256, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                            ((uint32_t)(kTcM >> 4) << 24);

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const bf16 a = __float2bfloat16_rn(lo), b = __float2bfloat16_rn(hi);
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// The 28 scaled boundary-state values of one edge and four zeros (an absent
// edge: zeros) as row r of the K = 32 A operand at sA (4 core matrices per
// 8-row group).
__device__ __forceinline__ void tc_features(const ArmK& A, const float* p0, const float* p1,
                                            bool on, uint8_t* sA, int r) {
  float f[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) f[j] = 0.f;
  if (on) {
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      const float c = 0.5f * (A.q_lo[j] + A.q_hi[j]);
      const float h = 0.5f * (A.q_hi[j] - A.q_lo[j]);
      f[j] = (p0[j] - c) / h;
      f[7 + j] = p0[8 + j] / A.qd_max[j];
      f[14 + j] = (p1[j] - c) / h;
      f[21 + j] = p1[8 + j] / A.qd_max[j];
    }
  }
#pragma unroll
  for (int kb = 0; kb < 4; ++kb) {
    uint4 v;
    v.x = pack_bf16x2(f[8 * kb + 0], f[8 * kb + 1]);
    v.y = pack_bf16x2(f[8 * kb + 2], f[8 * kb + 3]);
    v.z = pack_bf16x2(f[8 * kb + 4], f[8 * kb + 5]);
    v.w = pack_bf16x2(f[8 * kb + 6], f[8 * kb + 7]);
    *reinterpret_cast<uint4*>(sA + ((r >> 3) * 4 + kb) * 128 + (r & 7) * 16) = v;
  }
}

// The weight ring of one thread: chunks of 64 K columns (32 KB) copied kRing - 1
// ahead of the MMAs that read them, four to a layer, so that chunk c of a layer
// always lies in slot c; `period` chunks are a tile's, then they repeat.
// Barriers at bar: slot arrived (4), slot consumed (4).
struct TcRing {
  uint32_t bar, b_base;
  const bf16* W;
  int period;
  long total, g;                        // chunks to multiply, the next one
  long long limit;                      // of a wait
  uint32_t in_flight, ph_w, ph_free;    // a bit per slot

  __device__ TcRing(uint32_t bar_, uint32_t b_, const bf16* W_, int period_, int tiles,
                    long long limit_)
      : bar(bar_), b_base(b_), W(W_), period(period_), total((long)tiles * period_), g(0),
        limit(limit_), in_flight(0), ph_w(0), ph_free(0) {}
  __device__ void fill(int b, long chunk) {
    mbar_expect_tx(bar + 8u * b, kTcChunkBytes);
    bulk_g2s(b_base + b * kTcChunkBytes, W + (chunk % period) * (kTcChunkBytes / 2),
             kTcChunkBytes, bar + 8u * b);
    in_flight |= 1u << b;
  }
  __device__ void start() {
    for (int c = 0; c < kRing && c < total; ++c) fill(c, c);
  }
  // accumulator = A (K = 256 layout at a_base) times the next four chunks;
  // false when a wait ran out
  __device__ bool layer(uint32_t tmem, uint32_t a_base) {
#pragma unroll
    for (int c = 0; c < 4; ++c, ++g) {
      if (!mbar_wait(bar + 8u * c, ph_w >> c & 1u, limit)) return false;
      ph_w ^= 1u << c;
      in_flight &= ~(1u << c);
      const uint32_t bb = b_base + c * kTcChunkBytes;
#pragma unroll
      for (int s = 0; s < kTcKc / 16; ++s)
        umma_f16(tmem, sdesc(a_base + (4 * c + s) * 256, 128, 256 * 16),
                 sdesc(bb + s * 256, 128, kTcKc * 16), kIdesc, (c | s) != 0);
      umma_commit(bar + 8u * (4 + c));
      // refill the slot of the previous chunk (its MMAs are queued before
      // this chunk's) with the chunk kRing - 1 ahead of this one
      if (g >= 1 && g + kRing - 1 < total) {
        const int pb = (c + kRing - 1) % kRing;
        if (!mbar_wait(bar + 8u * (4 + pb), ph_free >> pb & 1u, limit)) return false;
        ph_free ^= 1u << pb;
        fill(pb, g + kRing - 1);
      }
    }
    return true;
  }
  // after a failure: wait (bounded) for the copies still in flight
  __device__ void drain() {
    for (int b = 0; b < kRing; ++b)
      if (in_flight >> b & 1u) mbar_wait(bar + 8u * b, ph_w >> b & 1u);
  }
};

}  // namespace fn
