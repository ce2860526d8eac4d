// Parents of Algorithm 1 (Sec. IV-E): brute-force parallel scan of the tree
// for each query's k nearest nodes under the velocity-weighted squared joint
// distance, ties broken by the lower node index.
//
// Layout: one thread per query, 128 queries per block; the block streams its
// slice of the tree through shared memory in tiles of 128 nodes (8 KB), so
// every node is read from L2 once per block and then broadcast from shared
// memory to all 128 queries.  Each thread keeps a sorted top-KM list
// (KM = 8 or 16) in registers.  The node range is split over `nsplit` blocks
// per query tile to fill the GPU; partial lists go to the caller's workspace
// and a second kernel merges them.
//
// Searches of 256 nodes and more (knn_tc_wanted) filter with the tensor
// cores instead (knn_tc.cuh): same lists.
#include <cuda_runtime.h>

#include <mutex>

#include "fn_internal.h"
#include "fn_pdl.cuh"
#include "knn_core.cuh"
#include "knn_tc.cuh"

namespace fn {

template <int KM>
__global__ void __launch_bounds__(128) k_knn_partial(const float4* __restrict__ tree, int N,
                                                     int first, const float4* __restrict__ queries,
                                                     int B, float w_vel, int nsplit, int k,
                                                     float* __restrict__ part_d,
                                                     int32_t* __restrict__ part_i,
                                                     float* __restrict__ out_d,
                                                     int32_t* __restrict__ out_i) {
  __shared__ float4 tile[KNN_TILE * 4];
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  const int split = blockIdx.y;
  const int span = N - first;
  const int per = (span + nsplit - 1) / nsplit;
  const int lo = first + split * per;
  const int hi = min(N, lo + per);
  TopK<KM> top;
  top.init();
  float qv[14];
  const bool active = b < B;
  if (active) load_query(queries + 4 * (long)b, qv);
  else
    for (int j = 0; j < 14; ++j) qv[j] = 0.f;
  knn_scan_range<KM>(tree, lo, hi, qv, w_vel, top, tile);
  if (!active) return;
  if (nsplit == 1) {
    top.store(out_d + (long)b * k, out_i + (long)b * k, k);
  } else {
    const long off = ((long)split * B + b) * KM;
    top.store(part_d + off, part_i + off, KM);
  }
}

// Merge of the split lists with one warp per query: lane l holds split l's
// sorted list; k rounds of a warp-wide (d, index) argmin over the list heads,
// the winning lane drops its head.
template <int KM>
__global__ void __launch_bounds__(256) k_knn_merge(int B, int nsplit, int k,
                                                   const float* __restrict__ part_d,
                                                   const int32_t* __restrict__ part_i,
                                                   float* __restrict__ out_d,
                                                   int32_t* __restrict__ out_i) {
  const int lane = threadIdx.x & 31;
  const long b = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= B) return;
  float d[KM];
  int id[KM];
#pragma unroll
  for (int j = 0; j < KM; ++j) {
    d[j] = INFINITY;
    id[j] = 0x7fffffff;
  }
  if (lane < nsplit) {
    const long off = ((long)lane * B + b) * KM;
#pragma unroll
    for (int j = 0; j < KM; ++j) {
      d[j] = part_d[off + j];
      id[j] = part_i[off + j];
    }
  }
  for (int r = 0; r < k; ++r) {
    float md = d[0];
    int mi = id[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float od = __shfl_xor_sync(0xffffffffu, md, o);
      const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
      if (knn_less(od, oi, md, mi)) { md = od; mi = oi; }
    }
    if (lane == 0) {
      const bool empty = (mi == 0x7fffffff);
      out_d[b * k + r] = empty ? INFINITY : md;
      out_i[b * k + r] = empty ? -1 : mi;
    }
    if (id[0] == mi && mi != 0x7fffffff) {  // the winner drops its head
#pragma unroll
      for (int j = 0; j + 1 < KM; ++j) {
        d[j] = d[j + 1];
        id[j] = id[j + 1];
      }
      d[KM - 1] = INFINITY;
      id[KM - 1] = 0x7fffffff;
    }
  }
}

// ---------------------------------------------------------------------------
// tensor-core filter (knn_tc.cuh)
// ---------------------------------------------------------------------------
// a thread per operand row: nodes [first, N) in ntiles tiles, then (queries
// of one batch) in tiles of 128
__global__ void __launch_bounds__(128) k_knn_tc_pack(const float4* __restrict__ tree, int N,
                                                     int first, int node_rows,
                                                     const float4* __restrict__ queries, int B,
                                                     float2 sc, uint8_t* __restrict__ nimg,
                                                     float2* __restrict__ soa,
                                                     uint8_t* __restrict__ qimg,
                                                     int* __restrict__ err) {
  pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *err = 0;
  float x[14];
  if (i < node_rows) {
    const bool have = i < N - first;
    if (have) {
      load_query(tree + 4 * (long)(first + i), x);
      knn_store_soa(soa, i, x);
    }
    knn_pack_node(nimg + (long)(i / KT_ROWS) * KT_TILE, i % KT_ROWS, x, sc, have);
  } else {
    const int b = i - node_rows;   // the grid ends with the last query tile
    const bool have = b < B;
    if (have) load_query(queries + 4 * (long)b, x);
    knn_pack_query(qimg + (long)(b / KT_ROWS) * KT_TILE, b % KT_ROWS, x, sc, have);
  }
}

struct KnnTcWork {
  const uint8_t* qimg;
  const uint8_t* nimg;
  float* gmin;
  int ntiles, B;
  __device__ __forceinline__ KtUnit operator()(long u) const {
    const long qt = u / ntiles, stride = 4 * kt_row_f4(ntiles);
    const int nt = (int)(u - qt * ntiles);
    return KtUnit{qimg + qt * 2 * KT_TILE, nimg + (long)nt * KT_TILE, gmin + qt * KT_QT * stride,
                  stride, (int)min((long)KT_QT, B - qt * KT_QT), nt, ntiles - 1 - nt};
  }
};

__global__ void __launch_bounds__(KT_THREADS, 1) k_knn_tc_mins(KnnTcWork W, long units, int* err) {
  extern __shared__ __align__(1024) uint8_t kt_smem[];
  pdl_begin();
  const long G = gridDim.x, b = blockIdx.x;
  knn_mins(kt_smem, W, units * b / G, units * (b + 1) / G, err);
}

// team warps to a query, of which the first searches alone and all share an
// exact scan (knn_wide)
template <int kGroups, int kStages>
__global__ void __launch_bounds__(256, 4)
    k_knn_tc_select(const float2* __restrict__ soa, int n, int first,
                    const float4* __restrict__ queries, int B, int k, float w, float2 sc,
                    const float* __restrict__ gmin, int ntiles, const int* __restrict__ err,
                    int team, float* __restrict__ out_d, int32_t* __restrict__ out_i) {
  __shared__ KnnWide<8, kGroups, kStages> sh;
  pdl_begin();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long b = ((long)blockIdx.x * 8 + warp) / team;
  const bool mine = warp % team == 0 && b < B;
  KeyList r;
  bool wide = false;
  if (mine)
    r = knn_select<true>(soa, n, first, queries + 4 * b, k, w, sc, gmin + b * 4 * kt_row_f4(ntiles),
                   ntiles, *err != 0, sh.list[warp], &wide);
  r = knn_wide(sh, r, wide, team, soa, n, first, queries + 4 * b, k, w);
  if (mine && lane < k) {
    out_d[b * k + lane] = __uint_as_float((unsigned)(r.key >> 32));
    out_i[b * k + lane] = r.key >= KT_NONE ? -1 : (int)(unsigned)r.key;
  }
}

// images and group minima of one batch of queries, at most (one tile of 256 queries
// if that is more): 64 MiB of minima and their queries' images at every tree size
constexpr size_t kKtBatchBytes = (size_t)88 << 20;
// Three overlapping launches cost about 11 us whatever they search (one after the
// other 17); the scan in one or two takes as long at 128 nodes (k = 8: 25 us for 32
// queries or more, 15 us for one) and 42 us at 256.  From 256 nodes on the
// filter is the faster one at every batch up to 16384 queries and every k measured
// (8192 queries: 44 -> 25 us at 256 nodes and k = 8, 1906 -> 123 at 65536 and
// k = 16).  Larger batches on a few hundred nodes are bound by the selection, whose
// time goes with k: with k = 1 the filter stays ahead (a million queries, 256 nodes
// 986 -> 820 us), with k = 8 the scan is ahead from 24576 queries at 256 nodes (52
// against 54 us, 269 against 459 for 262144), 65536 at 384 (121, 131) and 262144 at 576
// (496, 525), with k = 16 from 131072 at 256 only (275, 288): left with the filter, as a
// planning batch is far smaller and the line would run through B, N and k.  States closer to one another than
// the score's error, or outside its range, leave every group in reach; the
// exact scan of all nodes in the select step (knn_wide) then takes about the
// scan's time and the filter's.  8192 queries, 65536 nodes, k = 16: equal nodes
// 1145 -> 1441 us, four clusters 1902 -> 1437, states in degrees 1913 -> 1405;
// 2048 queries, 4096 nodes, k = 8: 45 -> 80, 80 -> 70, 82 -> 98; one query,
// 65536 nodes: 130 -> 199, 140 -> 220, 140 -> 128.
static bool knn_tc_wanted(int N) { return N >= 256; }

struct KnnTcPlan {
  int ntiles, batch;                     // batch 0: not even one tile of queries fits
  size_t nimg, soa, qimg, gmin, total;   // offsets into the workspace
};
// as many queries to a batch as `bytes` hold: the workspace of a larger tree or of
// fewer queries still serves, in more batches
static KnnTcPlan knn_tc_plan(int B, int N, size_t bytes = SIZE_MAX) {
  KnnTcPlan p;
  p.ntiles = (N + KT_ROWS - 1) / KT_ROWS;
  const size_t row = (size_t)kt_row_f4(p.ntiles) * sizeof(float4);
  const size_t tile = row * KT_QT + 2 * KT_TILE;   // of KT_QT queries
  p.nimg = 256;
  p.soa = p.nimg + (size_t)p.ntiles * KT_TILE;
  p.qimg = p.soa + (size_t)p.ntiles * (KT_ROWS / KT_GROUP) * KT_SOA * sizeof(float2);
  const size_t room = bytes > p.qimg ? (bytes - p.qimg) / tile : 0;
  const size_t fit = std::min(room, std::max<size_t>(1, kKtBatchBytes / tile)) * KT_QT;
  p.batch = (int)std::min<size_t>(fit, ((size_t)B + KT_QT - 1) / KT_QT * KT_QT);
  p.gmin = p.qimg + (size_t)(p.batch / KT_ROWS) * KT_TILE;
  p.total = p.gmin + (size_t)p.batch * row;
  return p;
}

// Whether the filter still pays in the batches of a workspace that does not hold
// the plan: a batch takes about 15 us whatever it searches, the scan, split or not,
// 15 us and as much again for 2^22 pairs (more where its threads are few).  16384 nodes
// and 8192 queries in 32 batches 526 us, the scan 1096; past the line 256 nodes, 8192
// queries in 32 batches 460, the scan 44.
static bool knn_tc_batches_pay(int B, int n, int batch) {
  return ((long)B + batch - 1) / batch <= 1 + ((long)B * n >> 22);
}

static fn_status knn_tc_launch(const float* tree, int N, int first, const float* queries, int B,
                               int k, float w_vel, int32_t* idx, float* d2, void* workspace,
                               const KnnTcPlan& p, cudaStream_t st) {
  static std::once_flag once[64];
  static bool attr_ok[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::call_once(once[dev & 63], [&] {
    attr_ok[dev & 63] = cudaFuncSetAttribute(k_knn_tc_mins,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kKtSmem) == cudaSuccess;
  });
  if (!attr_ok[dev & 63]) return FN_ECUDA;
  uint8_t* ws = (uint8_t*)workspace;
  int* err = (int*)ws;
  float2* soa = (float2*)(ws + p.soa);
  float* gmin = (float*)(ws + p.gmin);
  const float2 sc = knn_scales(w_vel, 7 * 16.0 * (1.0 + w_vel));   // of joints up to 4 rad, 4 rad/s
  // tiles of the nodes actually searched (the plan holds room for all N)
  const int ntiles = (N - first + KT_ROWS - 1) / KT_ROWS;
  for (int b0 = 0; b0 < B; b0 += p.batch) {
    const int nb = std::min(p.batch, B - b0);
    const int qtiles = (nb + KT_QT - 1) / KT_QT;
    const int nrows = b0 == 0 ? ntiles * KT_ROWS : 0;   // the node image serves every batch
    const float4* q = (const float4*)queries + 4 * (long)b0;
    k_knn_tc_pack<<<nrows / 128 + 2 * qtiles, 128, 0, st>>>((const float4*)tree, N, first, nrows, q,
                                                            nb, sc, ws + p.nimg, soa, ws + p.qimg, err);
    const long units = (long)qtiles * ntiles;
    const KnnTcWork W{ws + p.qimg, ws + p.nimg, gmin, ntiles, nb};
    // (launched while the step before drains: 100 queries on 600 nodes 10.9 us, with
    // plain launches 16.8)
    pl_launch(k_knn_tc_mins, (unsigned)std::min<long>(units, num_sms()), KT_THREADS, kKtSmem, st, W,
              units, err);
    int team = 8;   // warps to a query, up to what the chip holds
    while (team > 1 && (long)nb * team > 32L * num_sms()) team /= 2;
    const auto select = team > 1 ? k_knn_tc_select<8, 3> : k_knn_tc_select<4, 2>;
    pl_launch(select, (unsigned)(((long)nb * team + 7) / 8), 256, 0, st, soa, N - first, first, q, nb,
              k, w_vel, sc, gmin, ntiles, err, team, d2 + (long)b0 * k, idx + (long)b0 * k);
  }
  return launch_status();
}

int knn_km(int k) { return k <= 8 ? 8 : 16; }

// split count: about two blocks per SM, each split at least 4 tiles of
// nodes, at most 32 (one merge lane per split)
int knn_nsplit(int B, int N) {
  const int qblocks = (B + 127) / 128;
  const int want = (2 * num_sms() + qblocks - 1) / std::max(qblocks, 1);
  const int chunks = std::max(1, N / (4 * KNN_TILE));
  return std::max(1, std::min(std::min(want, chunks), 32));
}

// workspace of the split pass
static size_t knn_split_bytes(int B, int N, int k) {
  if (B <= 0 || N <= 0 || k < 1 || k > FN_MAX_KNN) return 0;
  const int ns = knn_nsplit(B, N);
  if (ns <= 1) return 0;
  const size_t per = (size_t)ns * B * knn_km(k);
  const size_t a = (per * sizeof(float) + 255) & ~(size_t)255;
  return a + per * sizeof(int32_t);
}

fn_status knn_launch(const float* tree, int N, int first, const float* queries, int B, int k,
                     float w_vel, int32_t* idx, float* d2, int nsplit, float* part_d,
                     int32_t* part_i, cudaStream_t st) {
  dim3 grid((B + 127) / 128, nsplit);
  if (knn_km(k) == 8) {
    k_knn_partial<8><<<grid, 128, 0, st>>>((const float4*)tree, N, first, (const float4*)queries,
                                           B, w_vel, nsplit, k, part_d, part_i, d2, idx);
    if (nsplit > 1)
      k_knn_merge<8><<<(B + 7) / 8, 256, 0, st>>>(B, nsplit, k, part_d, part_i, d2, idx);
  } else {
    k_knn_partial<16><<<grid, 128, 0, st>>>((const float4*)tree, N, first, (const float4*)queries,
                                            B, w_vel, nsplit, k, part_d, part_i, d2, idx);
    if (nsplit > 1)
      k_knn_merge<16><<<(B + 7) / 8, 256, 0, st>>>(B, nsplit, k, part_d, part_i, d2, idx);
  }
  return launch_status();
}

}  // namespace fn

using namespace fn;

extern "C" size_t fn_knn_workspace_bytes(int B, int N, int k) {
  const size_t split = knn_split_bytes(B, N, k);
  if (B <= 0 || N <= 0 || k < 1 || k > FN_MAX_KNN || !knn_tc_wanted(N)) return split;
  return std::max(split, knn_tc_plan(B, N).total);
}

extern "C" fn_status fn_knn_tree(const float* tree, int N, int first, const float* queries, int B,
                                 int k, float w_vel, int32_t* idx, float* d2, void* workspace,
                                 size_t workspace_bytes, void* stream) {
  if (N < 0 || first < 0 || first > N || B < 0 || k < 1 || k > FN_MAX_KNN) return FN_EINVAL;
  if (!(w_vel >= 0.f) || !std::isfinite(w_vel)) return FN_EINVAL;
  if (B == 0) return FN_OK;
  if (!queries || !idx || !d2 || !aligned16(queries)) return FN_EINVAL;
  if (N > first && (!tree || !aligned16(tree))) return FN_EINVAL;
  int nsplit = 1;
  float* part_d = nullptr;
  int32_t* part_i = nullptr;
  const size_t need = knn_split_bytes(B, N, k);
  // the tensor-core filter where the workspace holds its plan, or so many queries
  // beside the nodes that the batches are few; one that does not still gets the
  // split pass
  if (workspace && aligned256(workspace) && N > first && knn_tc_wanted(N - first)) {
    const KnnTcPlan p = knn_tc_plan(B, N, workspace_bytes);
    if (workspace_bytes >= knn_tc_plan(B, N).total ||
        (workspace_bytes >= need && p.batch > 0 && knn_tc_batches_pay(B, N - first, p.batch)))
      return knn_tc_launch(tree, N, first, queries, B, k, w_vel, idx, d2, workspace, p,
                           (cudaStream_t)stream);
  }
  if (workspace && need > 0) {
    if (workspace_bytes < need || !aligned256(workspace)) return FN_EINVAL;
    nsplit = knn_nsplit(B, N);
    const size_t per = (size_t)nsplit * B * knn_km(k);
    part_d = (float*)workspace;
    part_i = (int32_t*)((char*)workspace + ((per * sizeof(float) + 255) & ~(size_t)255));
  }
  return knn_launch(tree, N, first, queries, B, k, w_vel, idx, d2, nsplit, part_d, part_i,
                    (cudaStream_t)stream);
}
