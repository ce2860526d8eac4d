// Block layout of the paired edge scan with its per-link records in tensor
// memory (PairCore<TmemStash>), shared by the standalone edge-timing kernels
// and the planner's warp-per-edge edge body.
//
// One CTA of NW = 12 or 16 warps per SM holds all 512 tensor-memory columns;
// warp w uses lane quarter w % 4 and the 128-column block 128 (w / 4).  A warp
// works on runs of up to TM_GROUP edges: it stages a run, computes the
// end-sample splits of the whole run in one pass (split_group) and then scans
// the edges one by one.  The coefficients, staged edges, splits, the paired
// link table and the duration grid sit in dynamic shared memory, sized above
// half of the SM's so that no second CTA (which would wait for the columns) is
// placed on the SM.
// Sixteen warps (128 registers) hide more of the recursion's latency: 65536
// edges at K = 128, S = 64 711 -> 684 us in full mode, 193 -> 177 us at fixed
// durations.  The planner's kernels keep twelve: they run beside others that
// need the shared memory (an anytime toss 18.2 ms with sixteen, 18.1 with
// twelve).
#pragma once

#include <stdint.h>

#include <algorithm>

#include "edge_core.cuh"
#include "fn_internal.h"
#include "fn_tmem.cuh"

namespace fn {

#define TM_GROUP 10
constexpr int kTmCols = 512;
static_assert(FN_SPLIT_WORDS * sizeof(float) % 16 == 0, "16-byte split slots");
static_assert(TM_GROUP <= 10, "split_group takes at most ten edges");

// The CTA's carve of its dynamic shared memory and the calling warp's slots.
template <int NW>
struct TmBlock {
  static constexpr int kWarps = NW;
  static constexpr size_t kCoef = (size_t)NW * FN_CUBIC_WORDS * 32 * sizeof(float2);
  static constexpr size_t kEdge = (size_t)NW * TM_GROUP * 32 * sizeof(float);
  static constexpr size_t kSplit = (size_t)NW * TM_GROUP * FN_SPLIT_WORDS * sizeof(float);
  static constexpr size_t kLink = 7 * FN_LINK2_F4 * sizeof(float4);
  static constexpr size_t kGrid = FN_MAX_GRID * sizeof(float);
  static constexpr size_t kUsed = kCoef + kEdge + kSplit + kLink + kGrid + 16;   // + 4 words
  static constexpr size_t kSmem = (NW == 16 ? 180 : 140) * 1024;
  static_assert(kUsed <= kSmem, "tensor-memory scan: shared-memory layout");
  static_assert(2 * (kSmem + 1024) > 233472, "one CTA per SM");
  static_assert(kCoef % 16 == 0 && kEdge % 16 == 0 && kSplit % 16 == 0, "16-byte carve");
  static_assert((NW + 3) / 4 * FN_TM_COLS_PER_WARP <= kTmCols, "the warps of a lane quarter");
  float2* coef;     // [NW][FN_CUBIC_WORDS][32] paired coefficients
  float* edge;      // [NW][TM_GROUP][32] staged edges
  float* split;     // [NW][TM_GROUP][FN_SPLIT_WORDS] end-sample splits
  float4* link;     // [7][FN_LINK2_F4] paired link table
  float* grid;      // [FN_MAX_GRID] durations
  uint32_t* tmem;   // the allocation's base address
  int* next;        // the CTA's run counter
  int* aux;         // two words free for the kernel
  __device__ explicit TmBlock(void* smem) {
    char* b = reinterpret_cast<char*>(smem);
    coef = reinterpret_cast<float2*>(b);
    edge = reinterpret_cast<float*>(b + kCoef);
    split = reinterpret_cast<float*>(b + kCoef + kEdge);
    link = reinterpret_cast<float4*>(b + kCoef + kEdge + kSplit);
    grid = reinterpret_cast<float*>(b + kCoef + kEdge + kSplit + kLink);
    tmem = reinterpret_cast<uint32_t*>(b + kCoef + kEdge + kSplit + kLink + kGrid);
    next = reinterpret_cast<int*>(tmem + 1);
    aux = reinterpret_cast<int*>(tmem + 2);
  }
  __device__ float* edges_of(int w) const { return edge + TM_GROUP * 32 * w; }
  __device__ float* splits_of(int w) const { return split + TM_GROUP * FN_SPLIT_WORDS * w; }
  // warp w's core: its coefficient column and its tensor-memory block
  __device__ PairCore<TmemStash> core(uint32_t taddr, int w, int lane) const {
    return PairCore<TmemStash>{
        LinkTab2{link}, CubicLane2{coef + w * FN_CUBIC_WORDS * 32 + lane},
        TmemStash{taddr + ((uint32_t)((w & 3) * 32) << 16) +
                  FN_TM_COLS_PER_WARP * (uint32_t)(w >> 2)}};
  }
};

// CTAs for E items: one per SM, fewer only when there are fewer items.  A
// range with a warp for each item then costs its slowest one alone (tm_claim):
// 256 edges at K = 64 take 23 us on 152 SMs, and took 36 as pairs on the six
// warps of 22.
inline int tm_blocks(long E) { return (int)std::max<long>(1, std::min<long>(E, num_sms())); }

// Claim of a run by a warp of the CTA whose range holds `len` items: about
// (range left) / (2 NW) items, at least two (one where there is a warp
// for every item) and at most TM_GROUP, so that runs shrink towards the end of
// the range and the warps finish together.  Returns the run's first item (relative to the range) and its
// length n (0: the range is done), the same on every lane.
template <int NW>
__device__ __forceinline__ int tm_claim(int* next, int len, int& n) {
  const int lane = threadIdx.x & 31;
  int first = 0;
  n = 0;
  if (lane == 0) {
    const int seen = atomicAdd(next, 0);
    const int want = min(TM_GROUP, max(len <= NW ? 1 : 2, (len - seen) / (2 * NW)));
    first = atomicAdd(next, want);
    n = max(0, min(want, len - first));
  }
  first = __shfl_sync(0xffffffffu, first, 0);
  n = __shfl_sync(0xffffffffu, n, 0);
  return first;
}

}  // namespace fn
