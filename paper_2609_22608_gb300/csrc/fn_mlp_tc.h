// Tensor-core (tcgen05 / TMEM) inference of the duration surrogate.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fn_api.h"
#include "fn_arm.cuh"

namespace fn {

// Packed weight layout (the UMMA canonical K-major layout without swizzle):
// a chunk holds N = 256 output rows x Kt input columns; element (n, k) of a
// chunk sits at byte ((n / 8) * (Kt / 8) + k / 8) * 128 + (n % 8) * 16 +
// (k % 8) * 2, i.e. 8 x 8 "core matrices" of 128 contiguous bytes, adjacent
// along K 128 B apart and along N Kt * 16 B apart.
constexpr int kTcN = 256;              // hidden width (MMA N)
constexpr int kTcM = 128;              // edges per tile (MMA M, one TMEM lane each)
constexpr int kTcK1 = 32;              // layer-1 inputs (28 features + 4 zeros)
constexpr int kTcKc = 64;              // K columns per streamed weight chunk
constexpr int kTcChunkBytes = kTcN * kTcKc * 2;         // 32 KB
constexpr int kTcW1Bytes = kTcN * kTcK1 * 2;            // 16 KB
constexpr int kTcWpBytes = 4 * 4 * kTcChunkBytes;       // W2, W3, W3^T, W2^T: 16 chunks

// Pack the bf16 weights W [K][256] (row-major over the outputs): layer 1 as
// one chunk of 32 columns, layers 2 and 3, W3^T and W2^T (the backward pass)
// as chunks of kTcKc columns.
void mlp_tc_pack(const __nv_bfloat16* W1, const __nv_bfloat16* W2, const __nv_bfloat16* W3,
                 __nv_bfloat16* W1p, __nv_bfloat16* Wp, cudaStream_t st);

// Y[e] = MLP(features(s0[e], s1[e])) for e < E with the packed layers 1-3,
// the bf16 layer-4 weights W4b [256][2] and the FP32 biases.  *err is set
// to 1 if a wait on the tensor core or a copy took more than `wait` cycles.
// Y: device [E][2].
// E_dev (device, may be NULL): the rows actually present, at most E.
fn_status mlp_tc_forward(const ArmK& A, const float* s0, const float* s1, int E,
                         const __nv_bfloat16* W1p, const __nv_bfloat16* W23p, const float* b1,
                         const float* b2, const float* b3, const __nv_bfloat16* W4b,
                         const float* b4, float* Y, int* err, long long wait, cudaStream_t st,
                         const int* E_dev = nullptr);

// C = A B (+ bias, ReLU) in BF16 with FP32 accumulation on the tensor cores
// (fn_mlp_tc.cu): A [M][K], B [K][N], C [M][N] rounded to BF16.  *err is set
// to 1 if a wait on the tensor core timed out.
void gemm_tc(int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb,
             const float* bias, bool relu, __nv_bfloat16* C, int ldc, int* err, cudaStream_t st);

// One gradient (fn_mlp_train.cu).  img: the operand images of ceil(E / 128)
// tiles, X (8 KB a tile), h1, h2, h3, dz3, dz2, dz1 (64 KB a tile); row r, column
// c of a tile of width w at byte ((r / 8) * (w / 8) + c / 8) * 128 +
// (r % 8) * 16 + (c % 8) * 2.  loss, gW and gb are added
// to (zero before a gradient).  A wait that ran out sets *err, which stays, and
// *fail (zero before a gradient): the gradient is not one then.
struct MlpTrain {
  const float *s0, *s1;                       // [E][16]
  const int32_t* kstar;                       // [E]
  int E;
  const __nv_bfloat16 *W1p, *Wp, *W4b;
  const float* b[4];
  __nv_bfloat16* img[7];
  __nv_bfloat16* dy;                          // dL/dy by columns, dy_pitch (whole tiles) apart
  long dy_pitch;
  float *gW[4], *gb[4], *loss;
  int *err, *fail;
  long long wait;                             // limit of a wait in cycles
};
struct MlpLogT { float v[FN_MAX_GRID]; };     // log of the grid's durations
fn_status mlp_tc_train(const ArmK& A, const MlpLogT& logT, const MlpTrain& p, cudaStream_t st);

}  // namespace fn

struct fn_mlp;

namespace fn {

// The model's tensor-core forward over rows counted on the device (for a
// caller inside a captured sequence).  Stream-ordered, no host synchronisation.
fn_status mlp_forward_rows(fn_mlp* m, const ArmK& A, const float* s0, const float* s1, int E_max,
                           const int* E_dev, float* Y, cudaStream_t st);

}  // namespace fn
