// One gradient of the duration surrogate on the 5th-generation tensor cores,
// in two launches.
//
// k_mlp_train: one CTA walks tiles of 128 edges through forward and backward
// without leaving the SM.  Per tile: features; layers 1-3 as in inference
// (mlp_tc.cuh), the signs of the activations kept in two registers a layer;
// y = h3 W4 + b4 on mma.sync (two columns: nothing for tcgen05), the loss and
// dL/dy; dz3 = (dy W4^T) [h3 > 0]; then dz2 and dz1 through the packed W3^T and
// W2^T, masked by the kept signs.  X, h1, h2, h3, dz3, dz2, dz1 go to global
// memory with one bulk copy each, as they lie in shared memory ("images" of
// 8 x 8 core matrices); the bias gradients are summed from the registers, each
// warp over its 32 rows with a transposing butterfly, FP32.
//
// k_mlp_dw: dW_l = h_{l-1}^T dz_l over all edges.  The images read as MN-major
// operands are the transposes, so nothing is transposed or converted: a CTA
// takes a slice of the rows, 64 at a time (one bulk copy per operand, three
// stages), into the whole 256 x 256 FP32 accumulator (all 512 columns of tensor
// memory), and adds it to the gradient in 16-byte reductions.  dW1 is summed as
// dz1^T X (256 x 32), because the tensor core's M is 128; its few CTAs take the
// blocks in turn into kDw1Sets accumulators, so that a chain of additions on the
// tensor core (which does not round to nearest) is no longer than dW2's.  dW4 (two columns) is
// a chain of mma.sync over all rows in order, 16 of h3's columns to a CTA
// beside the others: one sum per element, whatever the batch and the grid.
//
// What bounds it: a gradient of 8192 edges is 64 tiles, one to a CTA, so the
// chain of a tile's five accumulators (31 us: MMAs, epilogue and one image
// copy after the other) and then dW4's chain and the flush of the
// accumulators (15 us).  Passing every layer through memory as FP32 in 17
// launches, with dW4 summed over all rows by four CTAs, took 1180 us for 8192
// edges against 106 with the loss read back, 500 against 99 for 1024 and
// 3790 against 163 for 32768.  dW4's one chain truncates (1.5e-5 off FP64 at 8192
// rows, 1.1e-4 at 32768); FP32 sums of stages of 512 rows measured 2.8e-6 and 9e-7
// at the same speed, but move the gradients of large batches by the 1e-4 that they
// repair, and with them every training run that is to be repeated.
//
// Waits are bounded as in inference: on a timeout the kernel raises the error
// flag, waits for its own copies in flight, frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fn_internal.h"
#include "mlp_tc.cuh"

namespace fn {

// shared memory beyond inference's map (kSY holds the column sums per lane
// quarter, [4][256]): the tile's y and its sums of the loss and dL/dy
constexpr int kSYv = kTcSmem;                       // [128][2] f32
constexpr int kSL = kSYv + kTcM * 2 * 4;            // [4][3] f32
constexpr int kTrainSmem = kSL + 64;

// lane j returns the sum over the warp's lanes of their v[j] (v is used up)
__device__ __forceinline__ float warp_colsum(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float keep = up ? v[i + o] : v[i], give = up ? v[i] : v[i + o];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 8 values of row `row`, columns 8 kb .., rounded to bf16 into the K = 256 A operand
__device__ __forceinline__ void store_row8(uint8_t* sA, int row, int kb, const float* x) {
  uint4 o;
  o.x = pack_bf16x2(x[0], x[1]);
  o.y = pack_bf16x2(x[2], x[3]);
  o.z = pack_bf16x2(x[4], x[5]);
  o.w = pack_bf16x2(x[6], x[7]);
  *reinterpret_cast<uint4*>(sA + ((row >> 3) * 32 + kb) * 128 + (row & 7) * 16) = o;
}

// D += A B, 16 x 8 x 16; ld_a: the 16 x 16 operand A from four core matrices at
// the lanes' addresses, transposed when they hold A^T
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
template <bool TRANS>
__device__ __forceinline__ void ld_a(uint32_t (&a)[4], uint32_t addr) {
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr)
                 : "memory");
}

__global__ void __launch_bounds__(kTcThreads, 1)
    k_mlp_train(ArmK A, MlpLogT logT, MlpTrain p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lq = warp & 3, cg = warp >> 2;          // TMEM lane quarter, column group
  const int trow = lq * 32 + lane;                  // this thread's row of the tile
  const int ntiles = (p.E + kTcM - 1) / kTcM;
  if ((int)blockIdx.x >= ntiles) return;   // block-uniform, before any barrier
  const int my_tiles = (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  uint8_t* sA = smem + kSA;
  float* sBias = reinterpret_cast<float*>(smem + kSBias);
  float* sW4 = reinterpret_cast<float*>(smem + kSW4);
  float* sY = reinterpret_cast<float*>(smem + kSY);
  float* sYv = reinterpret_cast<float*>(smem + kSYv);
  float* sL = reinterpret_cast<float*>(smem + kSL);
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(smem + kSBar + 80);
  volatile int* s_fail = reinterpret_cast<volatile int*>(smem + kSBar + 84);
  const uint32_t a_base = su32(sA), b_base = su32(smem + kSB), w1_base = su32(smem + kSW1);
  const uint32_t bar_base = su32(smem + kSBar);   // the ring's 8, layer done, W1 arrived
  const uint32_t bar_layer = bar_base + 64u, bar_w1 = bar_base + 72u, bar_drain = bar_base + 88u;

  for (int i = tid; i < 768; i += blockDim.x)
    sBias[i] = i < 256 ? p.b[0][i] : (i < 512 ? p.b[1][i - 256] : p.b[2][i - 512]);
  for (int i = tid; i < 512; i += blockDim.x) sW4[i] = __bfloat162float(p.W4b[i]);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32((const void*)s_tmem)),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < 10; ++b) mbar_init(bar_base + 8u * b, 1);
    mbar_init(bar_drain, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const uint32_t tmem_lane = tmem + ((uint32_t)(lq * 32) << 16);   // this warp's 32 lanes

  TcRing ring(bar_base, b_base, p.Wp, 16, my_tiles, p.wait);   // thread 0: W2, W3, W3^T, W2^T
  uint32_t ph_layer = 0;
  bool fail = false;
  if (tid == 0) {
    mbar_expect_tx(bar_w1, kTcW1Bytes);
    bulk_g2s(w1_base, p.W1p, kTcW1Bytes, bar_w1);
    ring.start();
  }
  const float b40 = p.b[3][0], b41 = p.b[3][1];

  for (int it = 0; it < my_tiles; ++it) {
    const long tile = (long)blockIdx.x + (long)it * gridDim.x;
    const long row = tile * kTcM + trow;
    const bool on = row < p.E;   // the rows past the batch are zeros in every image
    // ---- features -> A (K = 32 layout) and its image
    if (tid == 0) bulk_read_wait();   // the last image of the tile before
    __syncthreads();
    if (tid < kTcM) tc_features(A, p.s0 + 16 * row, p.s1 + 16 * row, on, sA, tid);
    proxy_fence();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      if (it == 0 && !mbar_wait(bar_w1, 0, p.wait)) fail = true;
      if (!fail) {
        bulk_s2g(p.img[0] + tile * (kTcM * kTcK1), a_base, kTcM * kTcK1 * 2);
#pragma unroll
        for (int s = 0; s < kTcK1 / 16; ++s)
          umma_f16(tmem, sdesc(a_base + s * 256, 128, kTcK1 * 16),
                   sdesc(w1_base + s * 256, 128, kTcK1 * 16), kIdesc, s > 0);
        umma_commit(bar_layer);
      }
    }
    // h > 0 of the thread's 64 columns: of the layer last masked with, the first, the third
    uint32_t pos[2] = {0u, 0u}, pos1[2] = {0u, 0u}, pos3[2] = {0u, 0u};
    // accumulators in turn: h1, h2, h3, dh2, dh1
#pragma unroll 1
    for (int phase = 0; phase < 5; ++phase) {
      if (tid == 0) {
        if (fail) *s_fail = 1;
        bulk_read_wait();   // A is free once its image has been read (and its MMAs are done)
      }
      __syncthreads();
      const bool lf = *s_fail || !mbar_wait(bar_layer, ph_layer, p.wait);
      ph_layer ^= 1;
      tc_fence_after();
      if (__syncthreads_or(lf)) {
        *s_fail = 1;
        break;
      }
      if (phase < 3) {
        const float* bias = sBias + 256 * phase;
        if (phase == 1) {
          pos1[0] = pos[0];
          pos1[1] = pos[1];
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int cb = 2 * cg + i;
          uint32_t v[32], m = 0u;
          tmem_ld32(tmem_lane + cb * 32, v);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float r = fmaxf(__uint_as_float(v[8 * q + j]) + bias[cb * 32 + 8 * q + j], 0.f);
              x[j] = on ? r : 0.f;
              if (__bfloat162float(__float2bfloat16_rn(x[j])) > 0.f) m |= 1u << (8 * q + j);
            }
            store_row8(sA, trow, cb * 4 + q, x);
          }
          if (phase < 2) pos[i] = m;
          else pos3[i] = m;
        }
      } else {
        // dz = dh [h > 0]: dz2 by the second layer's signs, then dz1 by the first's
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int cb = 2 * cg + i;
          uint32_t v[32];
          tmem_ld32(tmem_lane + cb * 32, v);
          float t[32];
#pragma unroll
          for (int j = 0; j < 32; ++j)
            t[j] = pos[i] >> j & 1u ? __uint_as_float(v[j]) : 0.f;
#pragma unroll
          for (int q = 0; q < 4; ++q) store_row8(sA, trow, cb * 4 + q, t + 8 * q);
          sY[256 * lq + cb * 32 + lane] = warp_colsum(t, lane);
          pos[i] = pos1[i];
        }
      }
      if (phase == 2) {
        // y = h3 W4 + b4: 16 rows to a warp, K in ascending steps of 16
        tc_fence_before();
        proxy_fence();
        __syncthreads();
        if (tid == 0) bulk_s2g(p.img[3] + tile * (kTcM * 256), a_base, kTcM * 256 * 2);
        if (warp < 8) {
          const int g = lane >> 2, tg = lane & 3;
          const uint32_t a0 = a_base +
                              ((2 * warp + (lane >> 3 & 1)) * 32 + (lane >> 4)) * 128 +
                              (lane & 7) * 16;
          float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int ks = 0; ks < 16; ++ks) {
            uint32_t a[4], b0 = 0u, b1 = 0u;
            ld_a<false>(a, a0 + ks * 256);
            if (g < 2) {
              const float* w = sW4 + 2 * (16 * ks + 2 * tg) + g;
              b0 = pack_bf16x2(w[0], w[2]);
              b1 = pack_bf16x2(w[16], w[18]);
            }
            mma_bf16(y, a, b0, b1);
          }
          if (tg == 0) {
            float* o = sYv + 2 * (16 * warp + g);
            o[0] = y[0] + b40;
            o[1] = y[1] + b41;
            o[16] = y[2] + b40;
            o[17] = y[3] + b41;
          }
        }
        if (tid == 0) bulk_read_wait();   // dz3 takes h3's place
        __syncthreads();
        // loss L = (1/n) sum_i [ f_i (y_i0 - log T*_i)^2 + BCE(y_i1, f_i) ] and dL/dy
        float g0 = 0.f, g1 = 0.f, L = 0.f;
        if (on) {
          const float y0 = sYv[2 * trow], y1 = sYv[2 * trow + 1];
          const int k = p.kstar[row];
          const float f = k >= 0 ? 1.f : 0.f;
          const float d = k >= 0 ? y0 - logT.v[min(k, FN_MAX_GRID - 1)] : 0.f;
          const float s = 1.f / (1.f + expf(-y1));
          L = f * d * d + fmaxf(y1, 0.f) - y1 * f + log1pf(expf(-fabsf(y1)));
          g0 = 2.f * f * d / (float)p.E;
          g1 = (s - f) / (float)p.E;
        }
        const bf16 d0 = __float2bfloat16_rn(g0), d1 = __float2bfloat16_rn(g1);
        if (cg == 0) {
          p.dy[row] = d0;
          p.dy[p.dy_pitch + row] = d1;
          const float sl = warp_sum(L), s0 = warp_sum(g0), s1 = warp_sum(g1);
          if (lane == 0) {
            sL[3 * lq] = s0;
            sL[3 * lq + 1] = s1;
            sL[3 * lq + 2] = sl;
          }
        }
        // dz3 = (dy W4^T) [h3 > 0], dy rounded to bf16
        const float e0 = __bfloat162float(d0), e1 = __bfloat162float(d1);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int cb = 2 * cg + i;
          float t[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float* w = sW4 + 2 * (cb * 32 + j);
            t[j] = pos3[i] >> j & 1u ? fmaf(e1, w[1], e0 * w[0]) : 0.f;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) store_row8(sA, trow, cb * 4 + q, t + 8 * q);
          sY[256 * lq + cb * 32 + lane] = warp_colsum(t, lane);
        }
      }
      tc_fence_before();
      proxy_fence();
      __syncthreads();
      if (tid == 0 && !fail) {
        tc_fence_after();
        bulk_s2g(p.img[phase < 2 ? 1 + phase : 2 + phase] + tile * (kTcM * 256), a_base, kTcM * 256 * 2);
        if (phase < 4) {
          fail = !ring.layer(tmem, a_base);
          if (!fail) umma_commit(bar_layer);
          else *s_fail = 1;
        }
      }
      // the tile's column sums into the gradients: 128 rows to an addition
      if (phase >= 2) {
        auto sum4 = [](const float* v, int pitch) {
          return (v[0] + v[pitch]) + (v[2 * pitch] + v[3 * pitch]);
        };
        if (tid >= 256) {
          const int k = tid - 256;
          atomicAdd((phase == 2 ? p.gb[2] : (phase == 3 ? p.gb[1] : p.gb[0])) + k,
                    sum4(sY + k, 256));
          if (phase == 2) {
            if (k < 2) atomicAdd(p.gb[3] + k, sum4(sL + k, 3));
            if (k == 2) atomicAdd(p.loss, sum4(sL + 2, 3) / (float)p.E);
          }
        }
      }
    }
    if (*s_fail) break;   // written before the phases' last barrier, or by every thread
  }
  // ---- exit: the images are complete; on failure, wait (bounded) for this
  // CTA's copies and MMAs still in flight
  if (tid == 0) bulk_wait();
  __syncthreads();
  if (*s_fail || fail) {
    if (tid == 0) {
      atomicExch(p.err, 1);
      atomicExch(p.fail, 1);
      mbar_wait(bar_w1, 0);
      ring.drain();
      umma_drain(bar_drain);
    }
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
}

// ---------------------------------------------------------------------------
// weight gradients from the images
// ---------------------------------------------------------------------------
constexpr int kDwRows = 64, kDwStages = 3, kDwThreads = 256;
constexpr int kDwA = kDwRows * 256 * 2;             // 32 KB: 64 rows of a 256-wide image
constexpr int kDwStage = 2 * kDwA;
constexpr int kDwBar = kDwStages * kDwStage;
constexpr int kDwSmem = kDwBar + 128;
constexpr int kDw1Sets = 4;                         // accumulators of dW1, 32 columns each
// dW4: CTAs of 16 columns of h3, 512 rows to a stage (16 KB of h3, 2 KB of dy)
constexpr int kDw4Ctas = 16, kDw4Rows = 512, kDw4Stages = 4;
constexpr int kDw4H = kDw4Rows * 16 * 2, kDw4Stage = kDw4H + kDw4Rows * 2 * 2;
static_assert(kDw4Stages * kDw4Stage <= kDwSmem, "dW4's stages fit the kernel's shared memory");

// gW4 columns 16 c .. of h3: warp 0 multiplies, every warp copies
__device__ __forceinline__ void dw4(const MlpTrain& p, int c, uint8_t* smem) {
  const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, tg = lane & 3;
  const int rows = (p.E + kTcM - 1) / kTcM * kTcM, n = (rows + kDw4Rows - 1) / kDw4Rows;
  const uint32_t base = su32(smem);
  auto cp16 = [](uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  };
  auto load = [&](int i) {   // one commit group per stage, empty past the end
    const int r0 = i * kDw4Rows, r = min(kDw4Rows, rows - r0);
    const uint32_t s = base + (i % kDw4Stages) * kDw4Stage;
    const char* src = reinterpret_cast<const char*>(p.img[3]) + (long)r0 * 512 + c * 256;
    for (int t = tid; t < 2 * r; t += kDwThreads)      // 16 pieces of each 8-row group
      cp16(s + t * 16, src + (long)(t >> 4) * 4096 + (t & 15) * 16);
    for (int t = tid; t < r / 4; t += kDwThreads) {    // r / 8 pieces of each of dy's columns
      const int col = t >= r / 8, q = t - col * (r / 8);
      cp16(s + kDw4H + col * kDw4Rows * 2 + q * 16, p.dy + (long)col * p.dy_pitch + r0 + 8 * q);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  for (int i = 0; i < kDw4Stages - 1; ++i) {
    if (i < n) load(i);
    else asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  for (int i = 0; i < n; ++i) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kDw4Stages - 2) : "memory");
    __syncthreads();   // stage i has arrived, stage i - 1 is used up
    if (i + kDw4Stages - 1 < n) load(i + kDw4Stages - 1);
    else asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (tid < 32) {
      const uint8_t* st = smem + (i % kDw4Stages) * kDw4Stage;
      const uint8_t* dy = st + kDw4H + (g & 1) * kDw4Rows * 2 + tg * 4;
      const int steps = min(kDw4Rows, rows - i * kDw4Rows) / 16;   // a multiple of 8
      for (int k = 0; k < steps; k += 8) {
        uint32_t a[8][4], b[8][2];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          ld_a<true>(a[j], su32(st) + (k + j) * 512 + lane * 16);
          b[j][0] = g < 2 ? *reinterpret_cast<const uint32_t*>(dy + (k + j) * 32) : 0u;
          b[j][1] = g < 2 ? *reinterpret_cast<const uint32_t*>(dy + (k + j) * 32 + 16) : 0u;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) mma_bf16(d, a[j], b[j][0], b[j][1]);
      }
    }
  }
  if (tid < 32 && tg == 0) {
    float* o = p.gW[3] + 2 * (16 * c + g);
    o[0] = d[0];
    o[1] = d[1];
    o[16] = d[2];
    o[17] = d[3];
  }
}

// as kIdesc with both operands MN-major; N = 256 or 32
constexpr uint32_t kDwIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                              ((uint32_t)(kTcM >> 4) << 24);

// blocks [0, 16): dW4, the longest chain; then the CTAs of one layer's dW split
// the 64-row blocks of the batch evenly: S for dW3, S for dW2, the rest dW1
__global__ void __launch_bounds__(kDwThreads, 1) k_mlp_dw(MlpTrain p, int S) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (blockIdx.x < kDw4Ctas) {
    dw4(p, blockIdx.x, smem);
    return;
  }
  const int bx = (int)blockIdx.x - kDw4Ctas;
  const int layer = bx < S ? 2 : (bx < 2 * S ? 1 : 0);
  const int s = layer ? bx % S : bx - 2 * S;
  const int ns = layer ? S : (int)gridDim.x - kDw4Ctas - 2 * S;
  const int nb = (p.E + kDwRows - 1) / kDwRows;
  const int r0 = (int)((long)s * nb / ns), n = (int)((long)(s + 1) * nb / ns) - r0;
  if (n <= 0) return;                                // block-uniform, before any barrier
  // A: the image whose columns are the accumulator's rows, B: its columns
  const bf16* gA = layer ? p.img[layer] : p.img[6];
  const bf16* gB = layer ? p.img[6 - layer] : p.img[0];
  const int wB = layer ? 256 : kTcK1;                // B's width
  const uint32_t bytesB = kDwRows * wB * 2;
  const int sets = layer ? 1 : kDw1Sets;
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(smem + kDwBar + 64);
  volatile int* s_fail = reinterpret_cast<volatile int*>(smem + kDwBar + 68);
  const uint32_t base = su32(smem), bar = base + kDwBar;   // arrived (3), consumed (3), done, drain
  const uint32_t bar_done = bar + 8u * (2 * kDwStages), bar_drain = bar_done + 8u;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32((const void*)s_tmem)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < 2 * kDwStages + 2; ++b) mbar_init(bar + 8u * b, 1);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  if (tid == 0) {
    const uint32_t idesc = kDwIdesc | (uint32_t)(wB >> 3) << 17;
    const uint32_t kB = wB * 16;                     // B's 8-row groups, bytes apart
    auto fill = [&](int st, int i) {
      mbar_expect_tx(bar + 8u * st, kDwA + bytesB);
      bulk_g2s(base + st * kDwStage, gA + (long)(r0 + i) * (kDwRows * 256), kDwA, bar + 8u * st);
      bulk_g2s(base + st * kDwStage + kDwA, gB + (long)(r0 + i) * (kDwRows * wB), bytesB,
               bar + 8u * st);
    };
    int filled = min(n, kDwStages), done = 0;
    for (int i = 0; i < filled; ++i) fill(i, i);
    for (; done < n; ++done) {
      const int st = done % kDwStages;
      if (!mbar_wait(bar + 8u * st, (done / kDwStages) & 1, p.wait)) break;
      const uint32_t a = base + st * kDwStage, b = a + kDwA;
#pragma unroll
      for (int j = 0; j < kDwRows / 16; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          umma_f16(tmem + 256 * h + 32 * (done % sets), sdesc(a + j * 8192 + h * 2048, 4096, 128),
                   sdesc(b + j * 2 * kB, kB, 128), idesc, done >= sets || j != 0);
      umma_commit(bar + 8u * (kDwStages + st));
      // refill the stage of the block before (its MMAs are queued before these)
      if (done >= 1 && done - 1 + kDwStages < n) {
        const int pb = (done - 1) % kDwStages;
        if (!mbar_wait(bar + 8u * (kDwStages + pb), ((done - 1) / kDwStages) & 1, p.wait)) break;
        fill(pb, filled);
        ++filled;
      }
    }
    if (done == n) {
      umma_commit(bar_done);
    } else {
      *s_fail = 1;
      for (int i = done; i < filled; ++i)
        mbar_wait(bar + 8u * (i % kDwStages), (i / kDwStages) & 1);
    }
  }
  __syncthreads();
  const bool bad = *s_fail || !mbar_wait(bar_done, 0, p.wait);
  if (__syncthreads_or(bad)) {
    if (tid == 0) {
      atomicExch(p.err, 1);
      atomicExch(p.fail, 1);
      umma_drain(bar_drain);
    }
  } else {
    tc_fence_after();
    // warp w: lanes of quarter w % 4, accumulator half w / 4
    const int h = warp >> 2, m = h * 128 + (warp & 3) * 32 + lane;
    const uint32_t src = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 256 * h;
    if (layer) {
      float* out = p.gW[layer] + 256 * m;
#pragma unroll 1
      for (int cb = 0; cb < 8; ++cb) {
        uint32_t v[32];
        tmem_ld32(src + cb * 32, v);
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          atomicAdd(reinterpret_cast<float4*>(out + cb * 32 + j),
                    make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3])));
      }
    } else {
      float t[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) t[j] = 0.f;
#pragma unroll 1
      for (int i = 0; i < min(n, sets); ++i) {
        uint32_t v[32];
        tmem_ld32(src + 32 * i, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) t[j] += __uint_as_float(v[j]);
      }
#pragma unroll
      for (int j = 0; j < 32; ++j) atomicAdd(p.gW[0] + 256 * j + m, t[j]);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u)
                 : "memory");
}

fn_status mlp_tc_train(const ArmK& A, const MlpLogT& logT, const MlpTrain& p, cudaStream_t st) {
  static bool attr[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr[dev]) {
    if (cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem) !=
            cudaSuccess)
      return FN_ECUDA;
    attr[dev] = true;
  }
  const int ntiles = (p.E + kTcM - 1) / kTcM;
  k_mlp_train<<<std::min(ntiles, num_sms()), kTcThreads, kTrainSmem, st>>>(A, logT, p);
  // four 64-row blocks to a CTA, so that its loads and MMAs (~2 us) outweigh
  // the flush of its accumulator, as long as the grid is one wave
  const int nb = (p.E + kDwRows - 1) / kDwRows;
  const int S = std::max(1, std::min((nb + 3) / 4, (num_sms() - kDw4Ctas) * 2 / 5));
  k_mlp_dw<<<kDw4Ctas + 2 * S + (S + 1) / 2, kDwThreads, kDwSmem, st>>>(p, S);
  return launch_status();
}

}  // namespace fn
