// Control-side entry points of Sec. IV-F and Sec. IV-E:
//   fn_controller_torque  the tracking controller of Eq. (controller): the
//                         cubic refitted from the measured state to the
//                         rendezvous, its initial acceleration clipped to the
//                         taper box, Eq. (torque), then the torque, power and
//                         slew clips; one thread per controller instance;
//   fn_check_edges_full   the full-resolution recheck of a plan's edges at
//                         their own durations: all three ratios of Def.
//                         "Feasibility Check" over S samples and the
//                         clearance over S_clear points; one to eight warps
//                         per edge.
#include <cuda_runtime.h>

#include <mutex>

#include "edge_core.cuh"
#include "fn_internal.h"
#include "fn_kin.cuh"

namespace fn {

// the limits the controller clips to, exactly as given (ArmK keeps only
// their reciprocals)
struct CtrlK {
  float tau_max[7];
  float w_max;
  float dslew[7];   // rate_j * dt
  float dt;
};

#define CTRL_ACC 1
#define CTRL_TORQUE 2
#define CTRL_POWER 4
#define CTRL_SLEW 8
#define CTRL_INVALID 0x80

__global__ void __launch_bounds__(128) k_controller(ArmK A, CtrlK L, int B,
                                                    const float* __restrict__ state,
                                                    const float* __restrict__ goal,
                                                    const float* __restrict__ Th,
                                                    const float* __restrict__ tau_prev,
                                                    float* __restrict__ tau,
                                                    float* __restrict__ qdd_out,
                                                    uint8_t* __restrict__ flags) {
  for (long b = (long)blockIdx.x * blockDim.x + threadIdx.x; b < B;
       b += (long)gridDim.x * blockDim.x) {
    EdgeStates es;
    bool fin = true;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      es.q0[j] = state[16 * b + j];
      es.qd0[j] = state[16 * b + 8 + j];
      es.q1[j] = goal[16 * b + j];
      es.qd1[j] = goal[16 * b + 8 + j];
      fin = fin && isfinite(es.q0[j]) && isfinite(es.qd0[j]) && isfinite(es.q1[j]) &&
            isfinite(es.qd1[j]);
    }
    const float T = Th[b];
    if (!fin || !(isfinite(T) && T > 0.f)) {
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        tau[7 * b + j] = NAN;
        if (qdd_out) qdd_out[7 * b + j] = NAN;
      }
      if (flags) flags[b] = CTRL_INVALID;
      continue;
    }
    unsigned f = 0;
    // Eq. (controller): the refitted cubic's acceleration at t = 0,
    // 2 b2 / T^2 = 6 (q_g - q) / T^2 - (4 qd + 2 qd_g) / T, from the
    // compensated coefficients (the two terms cancel on short horizons)
    Cubic cu;
    cubic_coef<true>(es, T, cu);
    PointCoef pc;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      float q, v, a;
      cubic_eval(cu, j, 0.f, q, v, a);
      // the box keeping the velocity after one period inside the taper
      const float bound = taper(A, j, es.q0[j]);
      const float lo = (-bound - es.qd0[j]) / L.dt, hi = (bound - es.qd0[j]) / L.dt;
      const float c = fminf(fmaxf(a, lo), hi);
      if (c != a) f |= CTRL_ACC;
      pc.q[j] = es.q0[j];
      pc.qd[j] = es.qd0[j];
      pc.qdd[j] = c;
      if (qdd_out) qdd_out[7 * b + j] = c;
    }
    float t7[7];
    torque_at(A, pc, 0.f, [&](int j, float tq, float) { t7[j] = tq; });
    float pw = 0.f;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      const float m = L.tau_max[j];
      const float c = fminf(fmaxf(t7[j], -m), m);
      if (c != t7[j]) f |= CTRL_TORQUE;
      t7[j] = c;
      pw = fmaf(c, es.qd0[j], pw);
    }
    if (fabsf(pw) > L.w_max) {
      const float sc = L.w_max / fabsf(pw);
#pragma unroll
      for (int j = 0; j < 7; ++j) t7[j] *= sc;
      f |= CTRL_POWER;
    }
    if (tau_prev) {
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        const float p = tau_prev[7 * b + j];
        const float c = fminf(fmaxf(t7[j], p - L.dslew[j]), p + L.dslew[j]);
        if (c != t7[j]) f |= CTRL_SLEW;
        t7[j] = c;
      }
    }
#pragma unroll
    for (int j = 0; j < 7; ++j) tau[7 * b + j] = t7[j];
    if (flags) flags[b] = (uint8_t)f;
  }
}

// The exact fixed-duration check (all S samples), rho_v, then the clearance
// (lane = point), by `group` warps of the CTA to an edge: warp r of a group
// takes the batches of 32 samples r, r + group, ... and of points likewise from
// the other end, and the maxima meet in shared memory.  A recheck is a few
// edges at a high resolution, so the chain of an edge's passes sets its time: 16
// edges at S = 256 with five obstacles take 13 us with eight warps each, and
// took 26 with one.
#define CHECK_WARPS 8
#define CHECK_BLOCKS 2   // of an SM
constexpr size_t kCheckWarp = (FN_CUBIC_WORDS + FN_LINK_WORDS + 1) * 32 * sizeof(float);
constexpr size_t kCheckSmem = CHECK_WARPS * (kCheckWarp + 4 * sizeof(float)) +
                              7 * FN_LINK_F4 * sizeof(float4);
// Warps to an edge, `warps` being what the chip holds at once: as many as it has
// batches of 32 samples and as keep all edges on the chip together.  With more
// edges than that warps that share one wait for one another: then one, or two
// where they end the last wave earlier (a wave of pairs takes 0.55 of a wave of
// single warps: S = 256, five obstacles 23.1 us against 43.8; S = 64 12.8
// against 23.0).  At S = 256 with five obstacles 608, 1216 and 3500 edges take 20.6,
// 28.7 and 75.8 us with four, two and two warps; 26.8, 49.2 and 135 with eight;
// 32.8, 33.0 and 92.2 with one.  65536 edges take 1180 us with one, 2352 with eight
// (and took 1758 with one in smaller blocks).
__host__ __device__ __forceinline__ int check_group(long E, int S, int warps) {
  int group = 1;
  while (group < CHECK_WARPS && 32 * group < S && E * 2 * group <= warps) group *= 2;
  const long waves1 = (E + warps - 1) / warps, waves2 = (2 * E + warps - 1) / warps;
  if (E > warps && S > 32 && 11 * waves2 < 20 * waves1) group = 2;
  return group;
}

__global__ void __launch_bounds__(32 * CHECK_WARPS, CHECK_BLOCKS)
    k_check_edges(ArmK A, fn_problem_t P, int E, const int* __restrict__ E_dev, int S,
                  int S_clear, float margin, int warps, const float* __restrict__ s0,
                  const float* __restrict__ s1, const float* __restrict__ Tv,
                  float* __restrict__ rho3, float* __restrict__ clearance,
                  uint8_t* __restrict__ ok) {
  extern __shared__ float4 check_smem[];
  float4* sLink = check_smem;
  float* sPart = reinterpret_cast<float*>(sLink + 7 * FN_LINK_F4);   // [CHECK_WARPS][4]
  fill_links(A, sLink);
  __syncthreads();
  if (E_dev) E = min(E, max(*E_dev, 0));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int group = check_group(E, S, warps);   // of the edges there are
  const int r = w % group, g = w / group, ng = CHECK_WARPS / group;
  float* mine = sPart + 4 * CHECK_WARPS + (kCheckWarp / sizeof(float)) * w;
  float* es = mine + (FN_CUBIC_WORDS + FN_LINK_WORDS) * 32;
  const CubicLane cb{mine + lane};
  const ScalarCore core{LinkTab{sLink}, cb, LaneLink{mine + FN_CUBIC_WORDS * 32 + lane}};
  auto group_sync = [&] {
    if (group == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + g), "r"(32 * group) : "memory");
  };
  for (long e = (long)blockIdx.x * ng + g; e < E; e += (long)gridDim.x * ng) {   // group-uniform
    const bool finite = stage_rows(s0 + 16 * e, s1 + 16 * e, es);
    const float T = Tv[e];
    if (!finite || !(isfinite(T) && T > 0.f)) {
      if (r == 0 && lane == 0) {
        rho3[3 * e] = rho3[3 * e + 1] = rho3[3 * e + 2] = NAN;
        clearance[e] = NAN;
        ok[e] = 0;
      }
      continue;
    }
    float mt = 0.f, mp = 0.f, mc = INFINITY;
    cubic_store_shared<true>(cb, es, T, 32);
#pragma unroll 1
    for (int b = r; 32 * b < S; b += group) {
      const int s = 32 * b + lane;
      float rx = 0.f, px = 0.f;
      core.eval(A, dup2(sample_u(s, S)), dup2(1.f), dup2(1.f),
                [&](int, float2 tau, float2 v, float inv_tau) {
                  rx = fmaxf(rx, fabsf(tau.x) * inv_tau);
                  px = fmaf(tau.x, v.x, px);
                }, lane);
      if (s < S) {
        mt = fmaxf(mt, rx);
        mp = fmaxf(mp, fabsf(px) * A.inv_w);
      }
    }
    if (P.n_obs > 0) {
      Cubic c;
      cubic_coef_sh<true>(es, T, c);
#pragma unroll 1
      for (int s = 32 * (group - 1 - r) + lane; s < S_clear; s += 32 * group) {
        const float u = sample_u(s, S_clear);
        float q[7];
#pragma unroll
        for (int j = 0; j < 7; ++j) {
          float v, a;
          cubic_eval(c, j, u, q[j], v, a);
        }
        mc = fminf(mc, config_clearance(A, q, P));
      }
    }
    mt = warp_max(mt);
    mp = warp_max(mp);
    mc = -warp_max(-mc);
    if (lane == 0) {
      sPart[4 * w] = mt;
      sPart[4 * w + 1] = mp;
      sPart[4 * w + 2] = mc;
    }
    group_sync();
    if (r == 0) {
      float rt = 0.f, rp = 0.f, cl = INFINITY;
      for (int i = 0; i < group; ++i) {
        rt = fmaxf(rt, sPart[4 * (w + i)]);
        rp = fmaxf(rp, sPart[4 * (w + i) + 1]);
        cl = fminf(cl, sPart[4 * (w + i) + 2]);
      }
      const float rv = warp_rho_v(A, es, T);
      if (lane == 0) {
        rho3[3 * e] = rt;
        rho3[3 * e + 1] = rp;
        rho3[3 * e + 2] = rv;
        clearance[e] = cl;
        ok[e] = (rt <= 1.f && rp <= 1.f && rv <= 1.f && (P.n_obs == 0 || cl >= margin)) ? 1 : 0;
      }
    }
    group_sync();   // the partial maxima are read
  }
}

}  // namespace fn

using namespace fn;

extern "C" fn_status fn_controller_torque(const fn_arm_t* arm, int B, const float* state,
                                          const float* goal, const float* T,
                                          const float* tau_prev, float dt,
                                          const float* tau_rate_max, float* tau, float* qdd_des,
                                          uint8_t* flags, void* stream) {
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  if (B < 0 || !(dt > 0.f) || !std::isfinite(dt)) return FN_EINVAL;
  if (tau_prev && !tau_rate_max) return FN_EINVAL;
  CtrlK L;
  for (int j = 0; j < 7; ++j) {
    L.tau_max[j] = arm->tau_max[j];
    L.dslew[j] = 0.f;
    if (tau_prev) {
      if (!(tau_rate_max[j] >= 0.f) || !std::isfinite(tau_rate_max[j])) return FN_EINVAL;
      L.dslew[j] = tau_rate_max[j] * dt;
    }
  }
  L.w_max = arm->w_max;
  L.dt = dt;
  if (B == 0) return FN_OK;
  if (!state || !goal || !T || !tau) return FN_EINVAL;
  const int blocks = (int)std::min<long>(((long)B + 127) / 128, 8L * num_sms());
  k_controller<<<blocks, 128, 0, (cudaStream_t)stream>>>(A, L, B, state, goal, T, tau_prev, tau,
                                                         qdd_des, flags);
  return launch_status();
}

extern "C" fn_status fn_check_edges_full(const fn_arm_t* arm, const float* s0, const float* s1,
                                         const float* T, int E, const int* E_dev, int S,
                                         int S_clear, int n_obs, const float* obs, float margin,
                                         float* rho3, float* clearance, uint8_t* ok,
                                         void* stream) {
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  if (E < 0 || S < 2 || S > FN_MAX_S) return FN_EINVAL;
  if (n_obs < 0 || n_obs > FN_MAX_OBS || (n_obs > 0 && (!obs || S_clear < 2))) return FN_EINVAL;
  if (!std::isfinite(margin)) return FN_EINVAL;
  fn_problem_t P;
  memset(&P, 0, sizeof(P));
  P.n_obs = n_obs;
  for (int b = 0; b < n_obs; ++b)
    for (int c = 0; c < 4; ++c) P.obs[b][c] = obs[4 * b + c];
  if (E == 0) return FN_OK;
  if (!s0 || !s1 || !T || !rho3 || !clearance || !ok) return FN_EINVAL;
  if (!aligned16(s0) || !aligned16(s1)) return FN_EINVAL;
  static std::once_flag once[64];
  static bool attr_ok[64];
  int dev = 0;
  cudaGetDevice(&dev);
  std::call_once(once[dev & 63], [&] {
    attr_ok[dev & 63] = cudaFuncSetAttribute(k_check_edges,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kCheckSmem) == cudaSuccess;
  });
  if (!attr_ok[dev & 63]) return FN_ECUDA;
  const int fit = CHECK_BLOCKS * num_sms(), warps = fit * CHECK_WARPS;
  // an edge count on the device may be any up to E: a block for each of the first
  const long want = E_dev ? E : ((long)E * check_group(E, S, warps) + CHECK_WARPS - 1) / CHECK_WARPS;
  const int blocks = (int)std::max<long>(1, std::min<long>(want, fit));
  k_check_edges<<<blocks, 32 * CHECK_WARPS, kCheckSmem, (cudaStream_t)stream>>>(
      A, P, E, E_dev, S, S_clear, margin, warps, s0, s1, T, rho3, clearance, ok);
  return launch_status();
}
