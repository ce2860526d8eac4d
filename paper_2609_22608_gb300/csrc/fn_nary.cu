// Minimum feasible time refined by the N-ary search (Sec. IV-D, the search
// after Def. "Minimum feasible time"): the grid scan finds the first
// feasible grid index k*, then the bracket (T_{k*-1}, T_{k*}] (T_{-1} = 0)
// is split into N = 32 equal slots per round; the 31 interior slot
// boundaries are checked and the slot where the check first passes is
// kept, until the bracket is no wider than eps.  rho_v is checked once, at
// the refined duration.
//
// One warp per edge, on the paired core with its records in tensor memory
// (tm_scan.cuh) unless a scalar variant of the grid scan was chosen.  A round is the grid scan's own probe/verify machinery
// (edge_core.cuh) run over a 31-entry duration list in the warp's shared
// slot, so the kernel keeps a single torque-evaluation call site: the grid
// pass and every round go through the same edge_scan call in one loop.  The
// rounds use witness probing: the 31 points are so close together that the
// points below T* usually violate at the sample that proved the bracket's
// lower end infeasible, so a round starts by probing that sample at every
// point, and a failed verify passes its violating sample on the same way.
#include <cuda_runtime.h>

#include "fn_internal.h"
#include <mutex>

#include "fn_tune.h"
#include "nary_core.cuh"
#include "tm_scan.cuh"

namespace fn {

using Tm = TmBlock<16>;

struct NaryGrid {
  float T[FN_MAX_GRID];
};

#define NARY_WARPS 3   // as the grid scan: static shared memory within 48 KB
#define NARY_MAX_ROUNDS 16

struct NaryOut {
  int32_t* k_star;
  float *T_star, *T_lo, *rho3;
  uint8_t* ok;
  int32_t* rounds;
};

// edge e's results (the warp's staged edge es; o.k = -2: invalid states)
__device__ __forceinline__ void nary_write(const ArmK& A, const float* es, long e,
                                           const NaryEdge& o, const NaryOut& out) {
  const bool found = o.k >= 0;
  const float rv = found ? warp_rho_v(A, es, o.b) : NAN;
  if ((threadIdx.x & 31) == 0) {
    out.k_star[e] = o.k;
    out.T_star[e] = found ? o.b : (o.k == -1 ? INFINITY : NAN);   // -2 invalid, -3 aborted
    if (out.T_lo) out.T_lo[e] = found ? o.a : NAN;
    out.rho3[3 * e + 0] = found ? o.rt : NAN;
    out.rho3[3 * e + 1] = found ? o.rp : NAN;
    out.rho3[3 * e + 2] = rv;
    out.ok[e] = (found && rv <= 1.f) ? 1 : 0;
    if (out.rounds) out.rounds[e] = o.r;
  }
}

// Persistent: warp w takes edges w, w + W, ...  MINB sets the register
// budget, as for the grid scan's kernel, whose tuned variant it follows.
template <int MINB>
__global__ void __launch_bounds__(32 * NARY_WARPS, MINB)
    k_time_edges_nary(ArmK A, NaryGrid G, int K, int S, const float* __restrict__ s0,
                      const float* __restrict__ s1, int E, const float* __restrict__ T_cap,
                      float eps, int max_rounds, NaryOut out,
                      unsigned long long* __restrict__ counter) {
  __shared__ float sT[FN_MAX_GRID];
  __shared__ float sSub[NARY_WARPS][32];
  __shared__ float sEdge[NARY_WARPS][32];
  __shared__ float sCoef[NARY_WARPS][FN_CUBIC_WORDS * 32];
  __shared__ float sWr[NARY_WARPS][FN_LINK_WORDS * 32];
  __shared__ __align__(16) float sSplit[NARY_WARPS][FN_SPLIT_WORDS];
  __shared__ float4 sLink[7 * FN_LINK_F4];
  fill_links(A, sLink);
  for (int i = threadIdx.x; i < K; i += blockDim.x) sT[i] = G.T[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* es = sEdge[w];
  float* sub = sSub[w];
  const CubicLane cb{&sCoef[w][lane]};
  const LaneLink wr{&sWr[w][lane]};
  const LinkTab L{sLink};
  const long W = (long)gridDim.x * NARY_WARPS;
  unsigned nsamp = 0;
  for (long e = (long)blockIdx.x * NARY_WARPS + w; e < E; e += W) {
    const bool finite = stage_rows(s0 + 16 * e, s1 + 16 * e, es);
    const float Tp = T_cap ? __ldg(T_cap + e) : INFINITY;
    NaryEdge o{-2, 0, NAN, NAN, NAN, NAN};
    if (finite)
      o = nary_edge(A, ScalarCore{L, cb, wr}, es, sSplit[w], sub, sT, grid_prefix(sT, K, Tp), S,
                    eps, max_rounds, nsamp);
    nary_write(A, es, e, o, out);
  }
  if (counter && lane == 0 && nsamp) atomicAdd(counter, (unsigned long long)nsamp);
}

// The same on tm_scan.cuh's block layout: runs of edges claimed by the CTA's
// warps, the splits of a run in one pass, then an edge at a time.  A pass
// checks 64 samples of a duration (two of the four interior probes of 32) where
// the scalar core checks 32 (one), and finds the same first violating sample,
// so the rounds are the scalar core's bit for bit.  The paired passes and the
// shared splits bound it as the grid scan: 65536 edges at K = 128, S = 64, eps =
// 1e-4 take 2.08 ms, the scalar variant 2.99.
constexpr size_t kNarySub = Tm::kWarps * 32 * sizeof(float);
static_assert(Tm::kUsed + kNarySub <= Tm::kSmem, "the warps' points beside the scan's layout");
__global__ void __launch_bounds__(32 * Tm::kWarps, 1)
    k_time_nary_tm(ArmK A, NaryGrid G, int K, int S, const float* __restrict__ s0,
                   const float* __restrict__ s1, int E, const float* __restrict__ T_cap,
                   float eps, int max_rounds, NaryOut out,
                   unsigned long long* __restrict__ counter) {
  extern __shared__ float4 tm_smem[];
  const Tm blk(tm_smem);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* sT = blk.grid;
  float* sub = reinterpret_cast<float*>(reinterpret_cast<char*>(tm_smem) + Tm::kUsed) + 32 * w;
  fill_links2(A, blk.link);
  const long per = ((long)E + gridDim.x - 1) / gridDim.x;
  const long r_lo = std::min<long>((long)blockIdx.x * per, E), r_hi = std::min<long>(r_lo + per, E);
  if (threadIdx.x == 0) *blk.next = 0;
  for (int i = threadIdx.x; i < K; i += blockDim.x) sT[i] = G.T[i];
  if (w == 0) tmem_alloc(blk.tmem, kTmCols);
  tmem_sync_block();
  const uint32_t tmem = *blk.tmem;
  const PairCore<TmemStash> core = blk.core(tmem, w, lane);
  float* es_g = blk.edges_of(w);
  float* split_g = blk.splits_of(w);
  unsigned nsamp = 0;
  for (;;) {
    int n;
    const int first = tm_claim<Tm::kWarps>(blk.next, (int)(r_hi - r_lo), n);
    if (n == 0) break;                               // warp-uniform
    const long e0 = r_lo + first;
    unsigned fin = 0u;
    for (int i = 0; i < n; ++i)
      if (stage_rows(s0 + 16 * (e0 + i), s1 + 16 * (e0 + i), es_g + 32 * i)) fin |= 1u << i;
    split_group(A, core, es_g, split_g, n, nsamp);
    for (int i = 0; i < n; ++i) {
      float* es = es_g + 32 * i;
      const float Tp = T_cap ? __ldg(T_cap + e0 + i) : INFINITY;
      NaryEdge o{-2, 0, NAN, NAN, NAN, NAN};
      if ((fin >> i) & 1u)
        o = nary_edge(A, core, es, split_g + FN_SPLIT_WORDS * i, sub, sT, grid_prefix(sT, K, Tp),
                      S, eps, max_rounds, nsamp);
      nary_write(A, es, e0 + i, o, out);
    }
  }
  if (counter && lane == 0 && nsamp) atomicAdd(counter, (unsigned long long)nsamp);
  tmem_sync_block();   // every warp's tensor-memory accesses precede the release
  if (w == 0) tmem_dealloc(tmem, kTmCols);
}

static fn_status launch_nary_tm(const ArmK& A, const NaryGrid& G, int K, int S, const float* s0,
                                const float* s1, int E, const float* T_cap, float eps,
                                int max_rounds, const NaryOut& out, unsigned long long* counter,
                                cudaStream_t st) {
  static std::once_flag once[64];
  static bool attr_ok[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::call_once(once[dev & 63], [&] {
    attr_ok[dev & 63] = cudaFuncSetAttribute(k_time_nary_tm,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Tm::kSmem) == cudaSuccess;
  });
  if (!attr_ok[dev & 63]) return FN_ECUDA;
  k_time_nary_tm<<<tm_blocks(E), 32 * Tm::kWarps, Tm::kSmem, st>>>(A, G, K, S, s0, s1, E, T_cap, eps,
                                                               max_rounds, out, counter);
  return launch_status();
}

}  // namespace fn

using namespace fn;

extern "C" fn_status fn_time_edges_nary(const fn_arm_t* arm, const float* s0, const float* s1,
                                        int E, const float* T_grid, int K, int S,
                                        const float* T_cap, float eps, int max_rounds,
                                        int32_t* k_star, float* T_star, float* T_lo, float* rho3,
                                        uint8_t* ok, int32_t* rounds,
                                        unsigned long long* sample_count, void* stream) {
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  if (E < 0 || S < 2 || S > FN_MAX_S) return FN_EINVAL;
  if (!(eps > 0.f) || !std::isfinite(eps)) return FN_EINVAL;
  if (max_rounds < 0 || max_rounds > NARY_MAX_ROUNDS) return FN_EINVAL;
  if (!T_grid || K < 1 || K > FN_MAX_GRID) return FN_EINVAL;
  NaryGrid G;
  for (int k = 0; k < K; ++k) {
    if (!(T_grid[k] > 0.f) || !std::isfinite(T_grid[k])) return FN_EINVAL;
    if (k > 0 && !(T_grid[k] > T_grid[k - 1])) return FN_EINVAL;
    G.T[k] = T_grid[k];
  }
  if (E == 0) return FN_OK;
  if (!s0 || !s1 || !k_star || !T_star || !rho3 || !ok) return FN_EINVAL;
  if (!aligned16(s0) || !aligned16(s1)) return FN_EINVAL;
  typedef void (*Kern)(ArmK, NaryGrid, int, int, const float*, const float*, int, const float*,
                       float, int, NaryOut, unsigned long long*);
  const NaryOut out{k_star, T_star, T_lo, rho3, ok, rounds};
  const int v = tuned_variant(TUNE_EDGES_FULL, E, K, S);    // the grid scan's core and budget
  if (v == kPairEdgeVariant)
    return launch_nary_tm(A, G, K, S, s0, s1, E, T_cap, eps, max_rounds, out, sample_count,
                          (cudaStream_t)stream);
  Kern kern = v == 0 ? k_time_edges_nary<2> : (v == 1 ? k_time_edges_nary<3> : k_time_edges_nary<4>);
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * NARY_WARPS, 0) !=
          cudaSuccess || per_sm < 1)
    per_sm = 1;
  const long want = ((long)E + NARY_WARPS - 1) / NARY_WARPS;
  const int blocks = (int)std::max<long>(1, std::min<long>(want, (long)per_sm * num_sms()));
  kern<<<blocks, 32 * NARY_WARPS, 0, (cudaStream_t)stream>>>(A, G, K, S, s0, s1, E, T_cap, eps,
                                                             max_rounds, out, sample_count);
  return launch_status();
}
