// Duration surrogate: an MLP 28 -> 256 -> 256 -> 256 -> 2 (ReLU) predicting
// (log T*, feasibility logit) of an edge from its boundary states, trained
// on labels produced by the exact duration scan (the windowed scan that uses
// it is fn_edges.cu's k_time_window_tm).  The paper has no learned
// component; this is the project's addition on top of Sec. IV-D's search.
//
// Precision (identical in the FP64 test oracle): inputs, weights and hidden
// activations are rounded to bf16 and contracted on the tensor cores with
// FP32 accumulation; biases, losses and gradients of the outputs are FP32;
// Adam keeps FP32 master weights and refreshes the bf16 copies after every
// step.
//
// Inference and training are fused tcgen05 kernels (fn_mlp_tc.cu,
// fn_mlp_train.cu); this file holds the reference forward, layer by layer
// through memory, with the two-column layer 4 on mma.sync.m16n8k16, and the
// model's state.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "edge_core.cuh"
#include "fn_internal.h"
#include "fn_mlp_tc.h"
#include "fn_umma.cuh"

namespace fn {

typedef __nv_bfloat16 bf16;

static const int kDims[5] = {32, 256, 256, 256, 2};  // input padded from 28 to 32
#define MLP_LAYERS 4
#define MLP_H 256

// ---------------------------------------------------------------------------
// features: q scaled by the joint box to [-1, 1], qd by qd_max, both states
// ---------------------------------------------------------------------------
__global__ void k_mlp_features(ArmK A, const float* __restrict__ s0, const float* __restrict__ s1,
                               int E, bf16* __restrict__ X) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long)E * 32) return;
  const long e = i >> 5;
  const int f = (int)(i & 31);
  float v = 0.f;
  if (f < 28) {
    const int j = f % 7, part = f / 7;
    const float* s = (part < 2 ? s0 : s1) + 16 * e;
    const float c = 0.5f * (A.q_lo[j] + A.q_hi[j]);
    const float h = 0.5f * (A.q_hi[j] - A.q_lo[j]);
    v = (part & 1) ? s[8 + j] / A.qd_max[j] : (s[j] - c) / h;
  }
  X[i] = __float2bfloat16_rn(v);
}

// ---------------------------------------------------------------------------
// C (M x N, f32) = A (M x K) B (K x N) + bias, bf16 operands, f32 accumulate.
// Tiles: 64 x 64 per block, 32 along K; 4 warps of 32 x 32.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(128) k_gemm_bf16(int M, int N, int K,
                                                   const bf16* __restrict__ A, int lda,
                                                   const bf16* __restrict__ B, int ldb,
                                                   const float* __restrict__ bias,
                                                   float* __restrict__ C, int ldc) {
  __shared__ __align__(16) bf16 As[64][40];  // [m][k]
  __shared__ __align__(16) bf16 Bs[64][40];  // [n][k]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = warp >> 1, wn = warp & 1;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  const bf16 zero = __float2bfloat16_rn(0.f);
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
  for (int k0 = 0; k0 < K; k0 += 32) {
    for (int t = tid; t < 64 * 32; t += 128) {
      const int r = t >> 5, c = t & 31;   // (m, k)
      const int gm = m0 + r, gk = k0 + c;
      bf16 v = zero;
      if (gm < M && gk < K) v = A[(long)gm * lda + gk];
      As[r][c] = v;
    }
    for (int t = tid; t < 64 * 32; t += 128) {
      const int r = t & 63, c = t >> 6;   // (n, k)
      const int gn = n0 + r, gk = k0 + c;
      bf16 v = zero;
      if (gn < N && gk < K) v = B[(long)gk * ldb + gn];
      Bs[r][c] = v;
    }
    __syncthreads();
    const int g = lane >> 2, tg = lane & 3;
#pragma unroll
    for (int ks = 0; ks < 32; ks += 16) {
      uint32_t a[2][4], b[4][2];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        const int r0 = wm * 32 + mi * 16 + g, c0 = ks + 2 * tg;
        a[mi][0] = *reinterpret_cast<const uint32_t*>(&As[r0][c0]);
        a[mi][1] = *reinterpret_cast<const uint32_t*>(&As[r0 + 8][c0]);
        a[mi][2] = *reinterpret_cast<const uint32_t*>(&As[r0][c0 + 8]);
        a[mi][3] = *reinterpret_cast<const uint32_t*>(&As[r0 + 8][c0 + 8]);
      }
#pragma unroll
      for (int ni = 0; ni < 4; ++ni) {
        const int n = wn * 32 + ni * 8 + g;
        b[ni][0] = *reinterpret_cast<const uint32_t*>(&Bs[n][ks + 2 * tg]);
        b[ni][1] = *reinterpret_cast<const uint32_t*>(&Bs[n][ks + 2 * tg + 8]);
      }
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni) mma_bf16(acc[mi][ni], a[mi], b[ni]);
    }
    __syncthreads();
  }
  const int g = lane >> 2, tg = lane & 3;
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          const int row = m0 + wm * 32 + mi * 16 + g + 8 * h;
          const int col = n0 + wn * 32 + ni * 8 + 2 * tg + cc;
          if (row >= M || col >= N) continue;
          C[(long)row * ldc + col] = acc[mi][ni][2 * h + cc] + bias[col];
        }
}

// Adam on FP32 master weights; bf16 copy refreshed.  *fail: the gradient was
// given up halfway, nothing is changed.
__global__ void k_mlp_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ g, const int* __restrict__ fail,
                           bf16* __restrict__ pb, long n, float lr, float b1, float b2, float eps,
                           float c1, float c2) {
  if (*fail) return;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float upd = (mi / c1) / (sqrtf(vi / c2) + eps);
    const float pn = p[i] - lr * upd;
    p[i] = pn;
    if (pb) pb[i] = __float2bfloat16_rn(pn);
  }
}

__global__ void k_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, long n) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

}  // namespace fn

using namespace fn;

struct fn_mlp {
  int max_batch;
  float* W[MLP_LAYERS];   // master [in][out]
  float* b[MLP_LAYERS];
  bf16* Wb[MLP_LAYERS];
  float* mW[MLP_LAYERS]; float* vW[MLP_LAYERS]; float* mb[MLP_LAYERS]; float* vb[MLP_LAYERS];
  float* gW[MLP_LAYERS]; float* gb[MLP_LAYERS];
  int step;
  // workspace for one batch
  bf16* X;        // [n][32]: features, row by row (reference forward) or as an image (training)
  bf16* Hb[3];    // [n][256]: activations, likewise
  bf16* dZ[3];    // [n][256]: the images of dz3, dz2, dz1
  bf16* dYb;      // [2][n]: dL/dy
  size_t rows;    // max_batch up to whole tiles, which the workspace holds
  float* Y;       // [n][2]
  float* grads;   // gW, gb and the loss in one piece
  size_t n_grads;
  float* loss;    // [1]
  int* fail;      // [1] the last gradient was given up (with the gradients: zeroed before one)
  // the weights packed for tcgen05 (with every change of the weights, on its
  // stream) and the kernels' error flag
  bf16* W1p;      // [16 KB]
  bf16* Wp;       // [512 KB]
  int* tc_err;    // [1]
  long long wait; // limit of their waits, clock cycles
  std::vector<void*> allocs;
};

static fn_status mlp_alloc(fn_mlp* m, void** p, size_t bytes) {
  if (cudaMalloc(p, bytes ? bytes : 16) != cudaSuccess) return FN_ENOMEM;
  m->allocs.push_back(*p);
  return FN_OK;
}

extern "C" fn_status fn_mlp_destroy(fn_mlp_t* m) {
  if (!m) return FN_EINVAL;
  for (void* p : m->allocs) cudaFree(p);
  delete m;
  return FN_OK;
}

// The packed copies of the weights, after every change of these on the stream
// of the change: whoever may use the new weights may use them packed, on any
// stream.  (Packed at their first use instead, they were written on that
// call's stream, of which a use on another one knew nothing.)
static void mlp_pack(fn_mlp* m, cudaStream_t st) {
  mlp_tc_pack(m->Wb[0], m->Wb[1], m->Wb[2], m->W1p, m->Wp, st);
}

extern "C" fn_status fn_mlp_create(int max_batch, unsigned long long seed, fn_mlp_t** out) {
  if (!out || max_batch < 1 || max_batch > (1 << 22)) return FN_EINVAL;
  fn_mlp* m = new fn_mlp();
  m->max_batch = max_batch;
  m->wait = kWaitCycles;
  m->step = 0;
  fn_status rc = FN_OK;
  auto A = [&](void** p, size_t bytes) {
    if (rc == FN_OK) rc = mlp_alloc(m, p, bytes);
  };
  for (int l = 0; l < MLP_LAYERS; ++l) {
    const size_t nw = (size_t)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
    A((void**)&m->W[l], nw * 4); A((void**)&m->b[l], nb * 4); A((void**)&m->Wb[l], nw * 2);
    A((void**)&m->mW[l], nw * 4); A((void**)&m->vW[l], nw * 4);
    A((void**)&m->mb[l], nb * 4); A((void**)&m->vb[l], nb * 4);
  }
  // every gradient tensor a multiple of 16 bytes into the piece
  m->n_grads = 4;
  for (int l = 0; l < MLP_LAYERS; ++l)
    m->n_grads += (size_t)kDims[l] * kDims[l + 1] + (kDims[l + 1] + 3) / 4 * 4;
  A((void**)&m->grads, m->n_grads * 4);
  if (rc == FN_OK) {
    float* g = m->grads;
    for (int l = 0; l < MLP_LAYERS; ++l) {
      m->gW[l] = g;
      g += (size_t)kDims[l] * kDims[l + 1];
      m->gb[l] = g;
      g += (kDims[l + 1] + 3) / 4 * 4;
    }
    m->loss = g;
    m->fail = reinterpret_cast<int*>(g + 1);
  }
  const size_t n = ((size_t)max_batch + kTcM - 1) / kTcM * kTcM;
  m->rows = n;
  A((void**)&m->X, n * 32 * 2);
  for (int l = 0; l < 3; ++l) A((void**)&m->Hb[l], n * MLP_H * 2);
  for (int l = 0; l < 3; ++l) A((void**)&m->dZ[l], n * MLP_H * 2);
  A((void**)&m->dYb, n * 2 * 2);
  A((void**)&m->Y, n * 2 * 4);
  A((void**)&m->W1p, kTcW1Bytes); A((void**)&m->Wp, kTcWpBytes); A((void**)&m->tc_err, 4);
  if (rc != FN_OK) {
    fn_mlp_destroy(m);
    return rc;
  }
  cudaMemset(m->tc_err, 0, 4);
  cudaMemset(m->fail, 0, 4);
  // He-uniform initial weights (inputs 28 of 32 used), zero biases, zero moments
  std::mt19937_64 rng(seed);
  for (int l = 0; l < MLP_LAYERS; ++l) {
    const int fin = l == 0 ? 28 : kDims[l], nin = kDims[l], nout = kDims[l + 1];
    const double lim = std::sqrt(6.0 / fin);
    std::uniform_real_distribution<double> U(-lim, lim);
    std::vector<float> w((size_t)nin * nout);
    for (int i = 0; i < nin; ++i)
      for (int o = 0; o < nout; ++o) w[(size_t)i * nout + o] = (l == 0 && i >= 28) ? 0.f : (float)U(rng);
    if (cudaMemcpy(m->W[l], w.data(), w.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess)
      rc = FN_ECUDA;
    const size_t nw = w.size();
    cudaMemset(m->b[l], 0, nout * 4);
    cudaMemset(m->mW[l], 0, nw * 4); cudaMemset(m->vW[l], 0, nw * 4);
    cudaMemset(m->mb[l], 0, nout * 4); cudaMemset(m->vb[l], 0, nout * 4);
    k_to_bf16<<<(unsigned)((nw + 255) / 256), 256>>>(m->W[l], m->Wb[l], (long)nw);
  }
  mlp_pack(m, nullptr);
  if (rc != FN_OK || cudaDeviceSynchronize() != cudaSuccess) {
    fn_mlp_destroy(m);
    return FN_ECUDA;
  }
  *out = m;
  return FN_OK;
}

// forward pass of n rows whose features are in m->X; Y = output
static void mlp_forward(fn_mlp* m, int n, cudaStream_t st) {
  for (int l = 0; l < 3; ++l)
    gemm_tc(n, 256, kDims[l], l ? m->Hb[l - 1] : m->X, kDims[l], m->Wb[l], 256, m->b[l], true,
            m->Hb[l], 256, m->tc_err, st);
  k_gemm_bf16<<<dim3(1, (n + 63) / 64), 128, 0, st>>>(n, 2, 256, m->Hb[2], 256, m->Wb[3], 2,
                                                      m->b[3], m->Y, 2);
}

static fn_status mlp_features(fn_mlp* m, const fn_arm_t* arm, const float* s0, const float* s1,
                              int n, cudaStream_t st) {
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  const long tot = (long)n * 32;
  k_mlp_features<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(A, s0, s1, n, m->X);
  return FN_OK;
}

// inference on the tcgen05 path (fused, no workspace, any E)
extern "C" fn_status fn_mlp_predict(fn_mlp_t* m, const fn_arm_t* arm, const float* s0,
                                    const float* s1, int E, float* Y, void* stream) {
  if (!m || E < 0 || !Y || (E > 0 && (!s0 || !s1))) return FN_EINVAL;
  if (E == 0) return FN_OK;
  if (!aligned16(s0) || !aligned16(s1)) return FN_EINVAL;
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  return mlp_tc_forward(A, s0, s1, E, m->W1p, m->Wp, m->b[0], m->b[1], m->b[2], m->Wb[3],
                        m->b[3], Y, m->tc_err, m->wait, st);
}

namespace fn {
fn_status mlp_forward_rows(fn_mlp* m, const ArmK& A, const float* s0, const float* s1, int E_max,
                           const int* E_dev, float* Y, cudaStream_t st) {
  if (!m || E_max < 0) return FN_EINVAL;
  if (E_max == 0) return FN_OK;
  return mlp_tc_forward(A, s0, s1, E_max, m->W1p, m->Wp, m->b[0], m->b[1], m->b[2], m->Wb[3],
                        m->b[3], Y, m->tc_err, m->wait, st, E_dev);
}
}  // namespace fn

extern "C" fn_status fn_mlp_set_wait(fn_mlp_t* m, long long cycles) {
  if (!m) return FN_EINVAL;
  m->wait = cycles;
  return FN_OK;
}

// the same forward layer by layer, E <= max_batch per internal batch
extern "C" fn_status fn_mlp_predict_ref(fn_mlp_t* m, const fn_arm_t* arm, const float* s0,
                                        const float* s1, int E, float* Y, void* stream) {
  if (!m || E < 0 || !Y || (E > 0 && (!s0 || !s1))) return FN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  for (int e0 = 0; e0 < E; e0 += m->max_batch) {
    const int n = std::min(m->max_batch, E - e0);
    fn_status rc = mlp_features(m, arm, s0 + 16L * e0, s1 + 16L * e0, n, st);
    if (rc != FN_OK) return rc;
    mlp_forward(m, n, st);
    if (cudaMemcpyAsync(Y + 2L * e0, m->Y, (size_t)n * 8, cudaMemcpyDeviceToDevice, st) !=
        cudaSuccess)
      return FN_ECUDA;
  }
  return launch_status();
}

extern "C" fn_status fn_mlp_error(fn_mlp_t* m, int* flag, int reset) {
  if (!m || !flag) return FN_EINVAL;
  if (cudaMemcpy(flag, m->tc_err, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return FN_ECUDA;
  if (reset && cudaMemset(m->tc_err, 0, 4) != cudaSuccess) return FN_ECUDA;
  return FN_OK;
}

// the loss of the gradient enqueued on st, and whether it was given up
static fn_status mlp_read_loss(fn_mlp* m, float* loss, cudaStream_t st) {
  float h[2];   // loss, fail
  if (cudaMemcpyAsync(h, m->loss, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return FN_ECUDA;
  int fail;
  std::memcpy(&fail, h + 1, sizeof(fail));
  *loss = h[0];
  return fail ? FN_ECUDA : FN_OK;
}

extern "C" fn_status fn_mlp_backward(fn_mlp_t* m, const fn_arm_t* arm, const float* s0,
                                     const float* s1, const int32_t* k_star, const float* T_grid,
                                     int K, int E, float* loss, void* stream) {
  if (!m || E < 1 || E > m->max_batch || !s0 || !s1 || !k_star) return FN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (!T_grid || K < 1 || K > FN_MAX_GRID) return FN_EINVAL;
  MlpLogT logT = {};
  for (int k = 0; k < K; ++k) {
    if (!(T_grid[k] > 0.f)) return FN_EINVAL;
    logT.v[k] = std::log(T_grid[k]);
  }
  ArmK A;
  if (!make_armk(arm, &A)) return FN_EINVAL;
  // not part of a graph: a replay would not count Adam's steps
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
    return FN_ECUDA;
  if (cudaMemsetAsync(m->grads, 0, m->n_grads * 4, st) != cudaSuccess) return FN_ECUDA;
  MlpTrain p;
  p.s0 = s0; p.s1 = s1; p.kstar = k_star; p.E = E;
  p.W1p = m->W1p; p.Wp = m->Wp; p.W4b = m->Wb[3];
  for (int l = 0; l < MLP_LAYERS; ++l) {
    p.b[l] = m->b[l]; p.gW[l] = m->gW[l]; p.gb[l] = m->gb[l];
  }
  p.img[0] = m->X;
  for (int l = 0; l < 3; ++l) {
    p.img[1 + l] = m->Hb[l];
    p.img[4 + l] = m->dZ[l];
  }
  p.dy = m->dYb; p.dy_pitch = (long)m->rows;
  p.loss = m->loss; p.err = m->tc_err; p.fail = m->fail; p.wait = m->wait;
  const fn_status rc = mlp_tc_train(A, logT, p, st);
  if (rc != FN_OK) return rc;
  return loss ? mlp_read_loss(m, loss, st) : FN_OK;
}

extern "C" fn_status fn_mlp_adam_step(fn_mlp_t* m, float lr, void* stream) {
  if (!m || !(lr >= 0.f)) return FN_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  m->step += 1;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = (float)(1.0 - std::pow(0.9, m->step));
  const float c2 = (float)(1.0 - std::pow(0.999, m->step));
  for (int l = 0; l < MLP_LAYERS; ++l) {
    const long nw = (long)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
    k_mlp_adam<<<(unsigned)((nw + 255) / 256), 256, 0, st>>>(m->W[l], m->mW[l], m->vW[l], m->gW[l], m->fail,
                                                            m->Wb[l], nw, lr, b1, b2, eps, c1, c2);
    k_mlp_adam<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(m->b[l], m->mb[l], m->vb[l], m->gb[l], m->fail,
                                                            nullptr, nb, lr, b1, b2, eps, c1, c2);
  }
  mlp_pack(m, st);
  return launch_status();
}

extern "C" fn_status fn_mlp_train_step(fn_mlp_t* m, const fn_arm_t* arm, const float* s0,
                                       const float* s1, const int32_t* k_star,
                                       const float* T_grid, int K, int E, float lr, float* loss,
                                       void* stream) {
  fn_status rc = fn_mlp_backward(m, arm, s0, s1, k_star, T_grid, K, E, nullptr, stream);
  if (rc != FN_OK) return rc;
  if ((rc = fn_mlp_adam_step(m, lr, stream)) != FN_OK) return rc;
  if (!loss) return FN_OK;
  rc = mlp_read_loss(m, loss, (cudaStream_t)stream);
  if (rc != FN_OK) m->step -= 1;   // the step was left out
  return rc;
}

// parameter / gradient / moment access (host arrays, layer l, W [in][out])
extern "C" fn_status fn_mlp_get_params(fn_mlp_t* m, int l, float* W, float* b) {
  if (!m || l < 0 || l >= MLP_LAYERS) return FN_EINVAL;
  const size_t nw = (size_t)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
  if (cudaDeviceSynchronize() != cudaSuccess) return FN_ECUDA;
  if (W && cudaMemcpy(W, m->W[l], nw * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return FN_ECUDA;
  if (b && cudaMemcpy(b, m->b[l], nb * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return FN_ECUDA;
  return FN_OK;
}

extern "C" fn_status fn_mlp_set_params(fn_mlp_t* m, int l, const float* W, const float* b) {
  if (!m || l < 0 || l >= MLP_LAYERS) return FN_EINVAL;
  const size_t nw = (size_t)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
  if (W && cudaMemcpy(m->W[l], W, nw * 4, cudaMemcpyHostToDevice) != cudaSuccess) return FN_ECUDA;
  if (b && cudaMemcpy(m->b[l], b, nb * 4, cudaMemcpyHostToDevice) != cudaSuccess) return FN_ECUDA;
  k_to_bf16<<<(unsigned)((nw + 255) / 256), 256>>>(m->W[l], m->Wb[l], (long)nw);
  mlp_pack(m, nullptr);
  return cudaDeviceSynchronize() == cudaSuccess ? FN_OK : FN_ECUDA;
}

extern "C" fn_status fn_mlp_get_grads(fn_mlp_t* m, int l, float* gW, float* gb) {
  if (!m || l < 0 || l >= MLP_LAYERS) return FN_EINVAL;
  const size_t nw = (size_t)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
  if (cudaDeviceSynchronize() != cudaSuccess) return FN_ECUDA;
  if (gW && cudaMemcpy(gW, m->gW[l], nw * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return FN_ECUDA;
  if (gb && cudaMemcpy(gb, m->gb[l], nb * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return FN_ECUDA;
  return FN_OK;
}

extern "C" fn_status fn_mlp_set_grads(fn_mlp_t* m, int l, const float* gW, const float* gb) {
  if (!m || l < 0 || l >= MLP_LAYERS) return FN_EINVAL;
  const size_t nw = (size_t)kDims[l] * kDims[l + 1], nb = kDims[l + 1];
  if (gW && cudaMemcpy(m->gW[l], gW, nw * 4, cudaMemcpyHostToDevice) != cudaSuccess) return FN_ECUDA;
  if (gb && cudaMemcpy(m->gb[l], gb, nb * 4, cudaMemcpyHostToDevice) != cudaSuccess) return FN_ECUDA;
  // the caller's gradient, in place before any stream's next step
  if (cudaMemset(m->fail, 0, 4) != cudaSuccess) return FN_ECUDA;
  return cudaDeviceSynchronize() == cudaSuccess ? FN_OK : FN_ECUDA;
}

// binary file: "FNMLP1\0\0", step, then per layer W (f32 [in][out]) and b
extern "C" fn_status fn_mlp_save(fn_mlp_t* m, const char* path) {
  if (!m || !path) return FN_EINVAL;
  FILE* f = std::fopen(path, "wb");
  if (!f) return FN_EINVAL;
  const char magic[8] = {'F', 'N', 'M', 'L', 'P', '1', 0, 0};
  bool ok = std::fwrite(magic, 1, 8, f) == 8 && std::fwrite(&m->step, 4, 1, f) == 1;
  for (int l = 0; l < MLP_LAYERS && ok; ++l) {
    std::vector<float> W((size_t)kDims[l] * kDims[l + 1]), b(kDims[l + 1]);
    ok = fn_mlp_get_params(m, l, W.data(), b.data()) == FN_OK &&
         std::fwrite(W.data(), 4, W.size(), f) == W.size() &&
         std::fwrite(b.data(), 4, b.size(), f) == b.size();
  }
  std::fclose(f);
  return ok ? FN_OK : FN_ECUDA;
}

extern "C" fn_status fn_mlp_load(fn_mlp_t* m, const char* path) {
  if (!m || !path) return FN_EINVAL;
  FILE* f = std::fopen(path, "rb");
  if (!f) return FN_EINVAL;
  char magic[8];
  int step = 0;
  bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "FNMLP1", 6) == 0 &&
            std::fread(&step, 4, 1, f) == 1;
  for (int l = 0; l < MLP_LAYERS && ok; ++l) {
    std::vector<float> W((size_t)kDims[l] * kDims[l + 1]), b(kDims[l + 1]);
    ok = std::fread(W.data(), 4, W.size(), f) == W.size() &&
         std::fread(b.data(), 4, b.size(), f) == b.size() &&
         fn_mlp_set_params(m, l, W.data(), b.data()) == FN_OK;
  }
  std::fclose(f);
  if (ok) m->step = step;
  return ok ? FN_OK : FN_EINVAL;
}

