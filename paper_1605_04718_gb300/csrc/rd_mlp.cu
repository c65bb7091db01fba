// rd_mlp.cu -- the surrogate network of delayed-acceptance sampling (not in
// the paper; Christen & Fox 2005): an MLP
//   x -> SiLU(W1 x + b1) -> SiLU(W2 . + b2) -> SiLU(W3 . + b3) -> W4 . + b4
// with x_i = (log theta_i - mu_i) / s_i (padded to 16 inputs), width 256,
// BF16 weights and activations into FP32-accumulating tcgen05 GEMMs, FP32
// master weights, Adam with decoupled weight decay, and the output mapped to
// a log-likelihood by Phi~ = floor + exp(shift + scale * net(x)).
//
// Forward and backward are row-local, so one kernel (k_mlp) takes a tile of 32 or
// 128 rows through all layers: weights stream into shared memory (128B-swizzled,
// cp.async) as operand A, the rows' activations are operand B, so the units lie
// on the TMEM lanes and a small tile still keeps 16 warps busy.  Each layer is
// two M = 128 kind::f16 MMA sequences (BF16 inputs, FP32 accumulators in TMEM)
// issued by one thread; the bias + SiLU (or SiLU') epilogue goes from TMEM
// straight into the next layer's operand tile.  Only the weight gradients sum
// over rows: k_mlp_wgrad forms them per layer, half of the outputs and a share
// of the row tiles, k_mlp_reduce adds the shares in a fixed order.
// Measured (GB300): Phi~ of 4096 rows 375 us with a kernel per layer, 36 us in
// one kernel with rows on the lanes (128-row tiles only), 20 us as it is; loss
// and gradients of 1024 rows 1017, 118 and 63 us.  What is left is latency: the
// weights' way from L2 (264 KB per tile), the layers' chain of MMAs, barrier
// and epilogue (16 instructions per value) and launches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "rd_common.cuh"
#include "rd_internal.h"
#include "rd_tc_ptx.cuh"

namespace rd {
namespace mlp {

using namespace tc;

constexpr int kIn = 16;        // padded input features
constexpr int kW = RD_SURROGATE_WIDTH;  // 256
constexpr int kMlpThreads = 512;
constexpr int kMaxSplits = 16;  // row shares of the weight gradients

// Instruction descriptor of kind::f16 with BF16 A and B, FP32 D.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float silu(float z) { return z / (1.f + __expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
  const float s = 1.f / (1.f + __expf(-z));
  return s * (1.f + z * (1.f - s));
}

struct Norm {
  double in_mu[RD_NPARAM], in_sd[RD_NPARAM];
  double floor, shift, scale;
};

// FP32 parameter layout: W1 [W][16], b1 [W], W2 [W][W], b2, W3 [W][W], b3, W4 [W], b4 [1].
struct Layout {
  int W;
  size_t oW1, ob1, oW2, ob2, oW3, ob3, oW4, ob4, total;
  __host__ __device__ constexpr explicit Layout(int w)
      : W(w),
        oW1(0),
        ob1((size_t)w * kIn),
        oW2(ob1 + w),
        ob2(oW2 + (size_t)w * w),
        oW3(ob2 + w),
        ob3(oW3 + (size_t)w * w),
        oW4(ob3 + w),
        ob4(oW4 + w),
        total(ob4 + 1) {}
  __host__ __device__ constexpr size_t stride() const { return (total + 3) / 4 * 4; }
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Copies rows x cols of a row-major BF16 matrix (16-byte aligned rows) into a
// 128B-swizzled tile, asynchronously; rows from rows_valid on become zero.
template <int COLS>
__device__ __forceinline__ void load_tile(uint8_t* tile, const __nv_bfloat16* g, int ld, int rows,
                                          int rows_valid) {
  constexpr int PER = COLS / 8;
  const uint32_t base = smem_u32(tile);
  for (int i = threadIdx.x; i < rows * PER; i += kMlpThreads) {
    const int r = i / PER, c = (i % PER) * 8;
    const uint32_t off = sw128_offset(rows, r, c);
    if (r < rows_valid)
      cp_async16(base + off, g + (size_t)r * ld + c);
    else
      *reinterpret_cast<uint4*>(tile + off) = make_uint4(0, 0, 0, 0);
  }
}

struct MlpArgs {
  int B, P;
  const double* theta;      // [B][P]
  const __nv_bfloat16* Wb;  // BF16 weights in the parameter layout
  const float* params;
  Norm nm;
  double* phit;             // MLP_PREDICT: [B]
  const float* target;      // else: [B]
  float* out;               // else: [B]
  double* sq_err;           // else: summed
  // MLP_GRAD: the features [B][16]; the rest with the units along the rows
  __nv_bfloat16* X;
  __nv_bfloat16 *H1, *H2, *dZ1, *dZ2, *dZ3;  // [W][B]
  float* Z1;                                 // [W][B]
  float* part4;             // [tile][W + 1]: shares of dW4, db4
  int* err;
  unsigned long long wait_ns;  // limit of the bounded waits
  int stall;                // failure-path test aid: layer 1's MMAs are never committed
};

enum { MLP_PREDICT = 0, MLP_LOSS = 1, MLP_GRAD = 2 };

struct MlpCtrl {
  uint64_t bar, fin;
  uint32_t tmem_base;
  int abort;
  float w4[kW];
  float out[128];
  alignas(16) float dout[128];
  float acc4[2][kW];
};
constexpr uint32_t kMlpTileW = kW * kW * 2;  // 128 KB: one layer's weights, rows = outputs
constexpr uint32_t act_bytes(int nr) { return (uint32_t)(nr > 64 ? 2 : 1) * kW * 128u; }
constexpr uint32_t mlp_smem_bytes(int nr) {
  // at least 150 KB, so that no other CTA with a TMEM allocation shares the SM
  return 1024 + kMlpTileW + act_bytes(nr) + (uint32_t)sizeof(MlpCtrl);
}

// After a wait that gave up: waits (again bounded) until every MMA that thread 0
// issued has finished, so that no tensor memory is freed under one.  By warp 0.
__device__ __forceinline__ void drain(uint64_t* fin) {
  if (threadIdx.x == 0) mma_commit(fin);
  __syncwarp();
  volatile int never = 0;
  mbar_wait_bounded(fin, 0, &never);
}

// One layer, D[unit][row] for both halves of the units: A = the weights' tile
// (K-major: its rows are the units; MN-major: its columns), B = the rows'
// activations ([K][NR], MN-major) or features (K-major).
template <int KK, int NR, int A_MN, int B_MN>
__device__ __forceinline__ void issue_layer(uint32_t d, uint32_t tw, uint32_t tx) {
  const uint32_t idesc = idesc_bf16(128, NR, A_MN, B_MN);
  const uint64_t bd = sdesc_sw128(tx, B_MN ? (uint32_t)kW * 128u : 16u, 1024u);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint64_t ad = sdesc_sw128(tw + (A_MN ? h * 2u * kW * 128u : h * 128u * 128u),
                                    A_MN ? (uint32_t)kW * 128u : 16u, 1024u);
#pragma unroll
    for (int kk = 0; kk < KK; ++kk) {
      const uint32_t oa = A_MN ? kk * 2048u : (uint32_t)(kk >> 2) * kW * 128u + (kk & 3) * 32u;
      const uint32_t ob = kk * 2048u;  // K-major B has KK = 1
      mma_f16(d + (uint32_t)(h * NR), ad + (oa >> 4), bd + (ob >> 4), idesc, kk > 0 ? 1u : 0u);
    }
  }
}

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// f(first row, 16 accumulator values, 16 results) over this thread's rows of one
// unit; results as BF16 into the activation tile and, if g is not null, g[row].
template <int NR, class F>
__device__ __forceinline__ void epilogue(uint32_t t, uint8_t* tile, int unit, int r0,
                                         __nv_bfloat16* g, F&& f) {
#pragma unroll 1
  for (int r = r0; r < r0 + NR / 2; r += 16) {
    float v[16];
    __nv_bfloat16 h[16];
    __syncwarp();
    tmem_ld16(t + (uint32_t)r, v);
    tmem_wait_ld();
    f(r, v, h);
#pragma unroll
    for (int k = 0; k < 16; k += 8) {
      const uint4 q = make_uint4(pack_bf16(h[k], h[k + 1]), pack_bf16(h[k + 2], h[k + 3]),
                                 pack_bf16(h[k + 4], h[k + 5]), pack_bf16(h[k + 6], h[k + 7]));
      *reinterpret_cast<uint4*>(tile + sw128_offset(kW, unit, r + k)) = q;
      if (g) *reinterpret_cast<uint4*>(g + r + k) = q;
    }
  }
}

// NR rows per CTA, units on the TMEM lanes (two accumulators of 128), rows on
// the columns: a tile of 32 rows still keeps every warp busy, so a batch of a
// few thousand rows spreads over all SMs.
template <int MODE, int NR>
__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp(const __grid_constant__ MlpArgs a) {
  extern __shared__ uint8_t mlp_smem[];
  uint8_t* const base = mlp_smem + ((1024u - (smem_u32(mlp_smem) & 1023u)) & 1023u);
  uint8_t* const tw = base;
  uint8_t* const ta = base + kMlpTileW;
  MlpCtrl* const ctl = reinterpret_cast<MlpCtrl*>(base + kMlpTileW + act_bytes(NR));
  constexpr Layout L(kW);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row0 = blockIdx.x * NR, valid = min(NR, a.B - row0);
  const int half = (warp >> 2) & 1;
  const int unit = 128 * half + 32 * (warp & 3) + lane, r0 = (NR / 2) * (warp >> 3);
  // layer 1's operands; its weights sit where W2's last 64 columns go later
  uint8_t* const tw1 = tw + kMlpTileW - 32768;
  load_tile<kIn>(tw1, a.Wb + L.oW1, kIn, kW, kW);
  cp_async_commit();
  auto load_w_cols = [&](const __nv_bfloat16* w, int b0, int b1) {  // 64-column blocks
    const uint32_t tb = smem_u32(tw);
    const int per = 8 * (b1 - b0);
    for (int i = tid; i < kW * per; i += kMlpThreads) {
      const int r = i / per, c = (i - r * per + 8 * b0) * 8;
      cp_async16(tb + sw128_offset(kW, r, c), w + (size_t)r * kW + c);
    }
    cp_async_commit();
  };
  load_w_cols(a.Wb + L.oW2, 0, 3);
  // features x_j = (log theta_j - mu_j) / s_j as BF16, zero-padded to 16, while
  // the weights are on their way; a thread each, since FP64 logarithms are what
  // they cost (a kernel of its own took 5 us for 4096 rows)
  for (int i = tid; i < NR * a.P; i += kMlpThreads) {
    const int r = i / a.P, j = i - r * a.P;
    float v = 0.f;
    if (r < valid) {
      const double t = a.theta[(size_t)(row0 + r) * a.P + j];
      v = (float)((log(t > 0.0 ? t : 1e-300) - a.nm.in_mu[j]) / a.nm.in_sd[j]);
    }
    for (int k = j; k < kIn; k += a.P) {
      const __nv_bfloat16 x = __float2bfloat16_rn(k == j ? v : 0.f);
      *reinterpret_cast<__nv_bfloat16*>(ta + sw128_offset(NR, r, k)) = x;
      if (MODE == MLP_GRAD) a.X[(size_t)(row0 + r) * kIn + k] = x;
    }
  }
  for (int i = tid; i < kW; i += kMlpThreads) ctl->w4[i] = a.params[L.oW4 + i];
  const float bias1 = a.params[L.ob1 + unit], bias2 = a.params[L.ob2 + unit],
              bias3 = a.params[L.ob3 + unit];
  if (warp == 0) {
    tmem_alloc(&ctl->tmem_base, 4 * NR);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&ctl->bar, 1);
    mbar_init(&ctl->fin, 1);
    ctl->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cp_async_wait<1>();
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_base;
  const uint32_t d0 = tmem, d1 = tmem + 2u * NR;  // a layer's accumulators
  const uint32_t t_off = ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(half * NR);
  const uint32_t sa = smem_u32(ta), sw = smem_u32(tw);
  uint32_t phase = 0;
  // waits for the MMAs issued since the last wait (a wait that gives up leaves
  // wrong values and raises the error flag at the end; later ones give up at once)
  auto done = [&]() {
    mbar_wait_bounded(&ctl->bar, phase & 1u, &ctl->abort, a.wait_ns);
    ++phase;
    tc_fence_after();
  };
  auto operands_ready = [&]() {
    cp_async_wait<0>();
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  };
  auto silu_epilogue = [&](uint32_t d, float bias, __nv_bfloat16* h_out, float* z_out) {
    epilogue<NR>(d + t_off, ta, unit, r0, h_out ? h_out + (size_t)unit * a.B + row0 : nullptr,
                 [&](int r, float (&v)[16], __nv_bfloat16 (&h)[16]) {
#pragma unroll
                   for (int j = 0; j < 16; ++j) {
                     v[j] += bias;
                     h[j] = __float2bfloat16_rn(silu(v[j]));
                   }
                   if (z_out) {
                     float4* z = reinterpret_cast<float4*>(z_out + (size_t)unit * a.B + row0 + r);
#pragma unroll
                     for (int j = 0; j < 4; ++j)
                       z[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                   }
                 });
  };
  // ---- layer 1 -> d0
  if (tid == 0) {
    issue_layer<1, NR, 0, 0>(d0, smem_u32(tw1), sa);
    if (!a.stall) mma_commit(&ctl->bar);
  }
  __syncwarp();
  done();
  load_w_cols(a.Wb + L.oW2, 3, 4);
  silu_epilogue(d0, bias1, MODE == MLP_GRAD ? a.H1 : nullptr, MODE == MLP_GRAD ? a.Z1 : nullptr);
  operands_ready();
  // ---- layer 2 -> d1
  if (tid == 0) {
    issue_layer<16, NR, 0, 1>(d1, sw, sa);
    mma_commit(&ctl->bar);
  }
  __syncwarp();
  done();
  load_w_cols(a.Wb + L.oW3, 0, 4);
  silu_epilogue(d1, bias2, MODE == MLP_GRAD ? a.H2 : nullptr, nullptr);
  operands_ready();
  // ---- layer 3 -> d0
  if (tid == 0) {
    issue_layer<16, NR, 0, 1>(d0, sw, sa);
    mma_commit(&ctl->bar);
  }
  __syncwarp();
  done();
  silu_epilogue(d0, bias3, nullptr, nullptr);
  __syncthreads();
  // ---- head: out[b] = sum_j H3[j][b] W4[j] + b4, one warp per row
#pragma unroll 1
  for (int r = warp; r < valid; r += kMlpThreads / 32) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kW / 32; ++i) {
      const int j = lane + 32 * i;
      const __nv_bfloat16 h =
          *reinterpret_cast<const __nv_bfloat16*>(ta + sw128_offset(kW, j, r));
      s += __bfloat162float(h) * ctl->w4[j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ctl->out[r] = s + a.params[L.ob4];
  }
  __syncthreads();
  if (MODE == MLP_PREDICT) {
    if (tid < valid)
      a.phit[row0 + tid] = a.nm.floor + exp(a.nm.shift + a.nm.scale * (double)ctl->out[tid]);
  } else {
    if (tid < NR) {
      double e2 = 0.0;
      if (tid < valid) {
        const float y = ctl->out[tid];
        const float e = y - a.target[row0 + tid];
        a.out[row0 + tid] = y;
        ctl->dout[tid] = 2.f * e / (float)a.B;
        e2 = (double)e * (double)e;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
      if (lane == 0) atomicAdd(a.sq_err, e2);
    }
    __syncthreads();
  }
  if (MODE == MLP_GRAD) {  // every tile is full: the batch is a multiple of 128
    // shares of dW4 and db4 over the tile's rows
    {
      const int j = tid & (kW - 1), hlf = tid / kW;
      float s = 0.f;
      for (int r = (NR / 2) * hlf; r < (NR / 2) * (hlf + 1); r += 8) {
        const uint4 q = *reinterpret_cast<const uint4*>(ta + sw128_offset(kW, j, r));
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 8; ++k)
          s += ctl->dout[r + k] * __bfloat162float(__ushort_as_bfloat16(
                                      (unsigned short)(w[k >> 1] >> (16 * (k & 1)))));
      }
      ctl->acc4[hlf][j] = s;
      __syncthreads();
      float* p4 = a.part4 + (size_t)blockIdx.x * (kW + 1);
      if (tid < kW) p4[tid] = ctl->acc4[0][tid] + ctl->acc4[1][tid];
      if (tid == 0) {
        float t = 0.f;
        for (int r = 0; r < NR; ++r) t += ctl->dout[r];
        p4[kW] = t;
      }
    }
    const size_t g0 = (size_t)unit * a.B + row0;
    // ---- dZ3 = dout W4 o SiLU'(Z3), Z3 still in d0
    const float w4 = ctl->w4[unit];
    epilogue<NR>(d0 + t_off, ta, unit, r0, a.dZ3 + g0,
                 [&](int r, float (&v)[16], __nv_bfloat16 (&h)[16]) {
#pragma unroll
                   for (int j = 0; j < 16; ++j)
                     h[j] = __float2bfloat16_rn(ctl->dout[r + j] * w4 * silu_grad(v[j] + bias3));
                 });
    operands_ready();
    // ---- dH2 = W3^T dZ3 -> d0; dZ2 = dH2 o SiLU'(Z2), Z2 in d1
    if (tid == 0) {
      issue_layer<16, NR, 1, 1>(d0, sw, sa);
      mma_commit(&ctl->bar);
    }
    __syncwarp();
    done();
    load_w_cols(a.Wb + L.oW2, 0, 4);
    epilogue<NR>(d0 + t_off, ta, unit, r0, a.dZ2 + g0,
                 [&](int r, float (&v)[16], __nv_bfloat16 (&h)[16]) {
                   float z[16];
                   tmem_ld16(d1 + t_off + (uint32_t)r, z);
                   tmem_wait_ld();
#pragma unroll
                   for (int j = 0; j < 16; ++j)
                     h[j] = __float2bfloat16_rn(v[j] * silu_grad(z[j] + bias2));
                 });
    operands_ready();
    // ---- dH1 = W2^T dZ2 -> d0; dZ1 = dH1 o SiLU'(Z1)
    if (tid == 0) {
      issue_layer<16, NR, 1, 1>(d0, sw, sa);
      mma_commit(&ctl->bar);
    }
    __syncwarp();
    done();
    epilogue<NR>(d0 + t_off, ta, unit, r0, a.dZ1 + g0,
                 [&](int r, float (&v)[16], __nv_bfloat16 (&h)[16]) {
                   const float4* z4 = reinterpret_cast<const float4*>(a.Z1 + g0 + r);
#pragma unroll
                   for (int j = 0; j < 4; ++j) {
                     const float4 z = z4[j];
                     h[4 * j] = __float2bfloat16_rn(v[4 * j] * silu_grad(z.x));
                     h[4 * j + 1] = __float2bfloat16_rn(v[4 * j + 1] * silu_grad(z.y));
                     h[4 * j + 2] = __float2bfloat16_rn(v[4 * j + 2] * silu_grad(z.z));
                     h[4 * j + 3] = __float2bfloat16_rn(v[4 * j + 3] * silu_grad(z.w));
                   }
                 });
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    if (ctl->abort) drain(&ctl->fin);
    tc_fence_after();
    tmem_dealloc(tmem, 4 * NR);
  }
  if (tid == 0 && ctl->abort) atomicOr(a.err, 1);
}

// Weight and bias gradients dW_l = dZ_l H_{l-1}^T, db_l = row sums of dZ_l
// (units along the rows): block (x = outputs 128 x .. 128 x + 127, y = layer,
// z = share of the 128-row tiles), into that share's copy of the parameter
// layout.
struct WgradArgs {
  int B, tiles, splits;
  const __nv_bfloat16* dZ[3];  // [W][B]
  const __nv_bfloat16* H[3];   // [0]: the features [B][16]; else [W][B]
  float* part;  // [splits][stride()]
  int* err;
  unsigned long long wait_ns;
  int stall;
};
constexpr uint32_t kWgTileA = 128 * 128 * 2, kWgTileB = 128 * kW * 2;
constexpr uint32_t kWgSmem = 1024 + 2 * (kWgTileA + kWgTileB) + 4 * 128 * 4;

__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp_wgrad(const __grid_constant__ WgradArgs a) {
  extern __shared__ uint8_t wg_smem[];
  uint8_t* const base = wg_smem + ((1024u - (smem_u32(wg_smem) & 1023u)) & 1023u);
  float* const sums = reinterpret_cast<float*>(base + 2 * (kWgTileA + kWgTileB));  // [4][128]
  __shared__ uint64_t bar, fin;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  constexpr Layout L(kW);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int layer = blockIdx.y, m0 = 128 * blockIdx.x, share = blockIdx.z;
  const int n = layer == 0 ? kIn : kW;
  const __nv_bfloat16* dz = a.dZ[layer] + (size_t)m0 * a.B;
  const __nv_bfloat16* hh = a.H[layer];
  const int t0 = (int)((long long)a.tiles * share / a.splits);
  const int t1 = (int)((long long)a.tiles * (share + 1) / a.splits);
  if (warp == 0) {
    tmem_alloc(&tmem_base, 256);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&bar, 1);
    mbar_init(&fin, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  auto load = [&](int t) {
    uint8_t* s = base + (uint32_t)(t & 1) * (kWgTileA + kWgTileB);
    load_tile<128>(s, dz + (size_t)t * 128, a.B, 128, 128);
    if (layer == 0)
      load_tile<kIn>(s + kWgTileA, hh + (size_t)t * 128 * kIn, kIn, 128, 128);
    else
      load_tile<128>(s + kWgTileA, hh + (size_t)t * 128, a.B, kW, kW);
    cp_async_commit();
  };
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const uint32_t idesc = idesc_bf16(128, n, 0, layer == 0 ? 1 : 0);
  const int col = tid & 127, quarter = tid >> 7;
  float colsum = 0.f;
  uint32_t phase = 0;
  bool ok = true;
  load(t0);
  for (int t = t0; t < t1; ++t) {
    uint8_t* s = base + (uint32_t)(t & 1) * (kWgTileA + kWgTileB);
    if (t > t0) {  // the other buffer's MMAs are done: it may be refilled
      ok = mbar_wait_bounded(&bar, phase & 1u, &abort_flag, a.wait_ns) && ok;
      ++phase;
      tc_fence_after();
    }
    cp_async_wait<0>();
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0) {
      const uint32_t sb = smem_u32(s + kWgTileA);
      const uint64_t ad = sdesc_sw128(smem_u32(s), 16u, 1024u);
      const uint64_t bd = layer == 0 ? sdesc_sw128(sb, 128u * 128u, 1024u)
                                     : sdesc_sw128(sb, 16u, 1024u);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint32_t oa = (uint32_t)(kk >> 2) * 128u * 128u + (kk & 3) * 32u;
        const uint32_t ob =
            layer == 0 ? kk * 2048u : (uint32_t)(kk >> 2) * kW * 128u + (kk & 3) * 32u;
        mma_f16(tmem, ad + (oa >> 4), bd + (ob >> 4), idesc, (t > t0 || kk > 0) ? 1u : 0u);
      }
      if (!a.stall) mma_commit(&bar);
    }
    __syncwarp();
    if (t + 1 < t1) load(t + 1);
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
      const uint4 q = *reinterpret_cast<const uint4*>(s + sw128_offset(128, col, 32 * quarter + r));
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int k = 0; k < 8; ++k)
        colsum += __bfloat162float(
            __ushort_as_bfloat16((unsigned short)(w[k >> 1] >> (16 * (k & 1)))));
    }
  }
  ok = mbar_wait_bounded(&bar, phase & 1u, &abort_flag, a.wait_ns) && ok;
  tc_fence_after();
  sums[tid] = colsum;
  __syncthreads();
  const size_t oW[3] = {L.oW1, L.oW2, L.oW3}, ob[3] = {L.ob1, L.ob2, L.ob3};
  float* part = a.part + (size_t)share * L.stride();
  if (tid < 128)
    part[ob[layer] + m0 + tid] =
        (sums[tid] + sums[128 + tid]) + (sums[256 + tid] + sums[384 + tid]);
  if (ok) {
    const int m = m0 + 32 * (warp & 3) + lane;  // TMEM lane = output
    const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    float* dst = part + oW[layer] + (size_t)m * n;
    for (int c = 16 * (warp >> 2); c < n; c += 64) {
      float v[16];
      __syncwarp();
      tmem_ld16(trow + (uint32_t)c, v);
      tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; j += 4)
        *reinterpret_cast<float4*>(dst + c + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    if (abort_flag) drain(&fin);
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
  if (tid == 0 && abort_flag) atomicOr(a.err, 1);
}

// grads = the shares' sum, in share (row tile) order.
__global__ void k_mlp_reduce(int splits, int tiles, const float* part, const float* part4,
                             float* grads) {
  constexpr Layout L(kW);
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.total) return;
  float s = 0.f;
  if (i < L.oW4) {
#pragma unroll 4
    for (int k = 0; k < splits; ++k) s += part[(size_t)k * L.stride() + i];
  } else {
#pragma unroll 4
    for (int k = 0; k < tiles; ++k) s += part4[(size_t)k * (kW + 1) + (i - L.oW4)];
  }
  grads[i] = s;
}

// ---------------------------------------------------------------------------
// Small CUDA-core kernels
// ---------------------------------------------------------------------------
// Adam with bias correction and decoupled weight decay on the weights (mask
// = 1) but not the biases; refreshes the BF16 copies of W1..W3.
struct AdamArgs {
  float* p;
  const float* g;
  float* m;
  float* v;
  const uint8_t* decay_mask;
  int n;
  float lr, b1, b2, eps, wd, c1, c2;
};
__global__ void k_adam(AdamArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const float gi = a.g[i];
  const float m = a.m[i] = a.b1 * a.m[i] + (1.f - a.b1) * gi;
  const float v = a.v[i] = a.b2 * a.v[i] + (1.f - a.b2) * gi * gi;
  float p = a.p[i];
  if (a.decay_mask[i]) p -= a.lr * a.wd * p;
  p -= a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
  a.p[i] = p;
}

__global__ void k_to_bf16(int n, const float* src, __nv_bfloat16* dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

}  // namespace mlp
}  // namespace rd

// ---------------------------------------------------------------------------
// Host side: the surrogate object, forward/backward, training, prediction
// ---------------------------------------------------------------------------
struct rd_surrogate {
  rd_problem* pb = nullptr;
  int P = 0;
  int W = 256;
  rd::mlp::Norm norm{};
  float* params = nullptr;
  float* grads = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  uint8_t* decay_mask = nullptr;
  __nv_bfloat16* Wb = nullptr;  // BF16 copies of W1, W2, W3 (packed like params)
  int adam_t = 0;
  // activations for up to `cap` rows
  int cap = 0;
  float* out = nullptr;
  double* sqerr = nullptr;
  // the backward pass's, for up to `grad_cap` rows
  int grad_cap = 0;
  __nv_bfloat16 *X = nullptr, *H1 = nullptr, *H2 = nullptr, *dZ1 = nullptr, *dZ2 = nullptr, *dZ3 = nullptr;
  float *Z1 = nullptr, *part = nullptr, *part4 = nullptr;
};

namespace rd {
namespace mlp {

static void free_acts(rd_surrogate* s) {
  cudaFree(s->out);
  cudaFree(s->sqerr);
  s->out = nullptr;
  s->sqerr = nullptr;
  s->cap = 0;
}

static void free_grad(rd_surrogate* s) {
  void* ptrs[] = {s->X, s->H1, s->H2, s->dZ1, s->dZ2, s->dZ3, s->Z1, s->part, s->part4};
  for (void* p : ptrs) cudaFree(p);
  s->X = s->H1 = s->H2 = s->dZ1 = s->dZ2 = s->dZ3 = nullptr;
  s->Z1 = s->part = s->part4 = nullptr;
  s->grad_cap = 0;
}

#define RD_ALLOC(ptr, bytes) \
  if ((e = cudaMalloc(&(ptr), (bytes))) != cudaSuccess) return e;

// Buffers of a forward pass over `rows` rows.
cudaError_t ensure_rows(rd_surrogate* s, int rows) {
  if (rows <= s->cap) return cudaSuccess;
  cudaStreamSynchronize(s->pb->stream);
  free_acts(s);
  const size_t cap = (size_t)((rows + 127) / 128) * 128;
  cudaError_t e;
  RD_ALLOC(s->out, sizeof(float) * cap);
  RD_ALLOC(s->sqerr, sizeof(double));
  s->cap = (int)cap;
  s->pb->generation++;  // captured graphs may hold the old buffers
  return cudaSuccess;
}

// And of a backward pass (rows a multiple of 128).
static cudaError_t ensure_grad_rows(rd_surrogate* s, int rows) {
  cudaError_t e = ensure_rows(s, rows);
  if (e != cudaSuccess || rows <= s->grad_cap) return e;
  cudaStreamSynchronize(s->pb->stream);
  free_grad(s);
  const size_t cap = (size_t)rows, W = (size_t)s->W;
  const Layout L(s->W);
  RD_ALLOC(s->X, sizeof(__nv_bfloat16) * cap * kIn);
  RD_ALLOC(s->H1, sizeof(__nv_bfloat16) * cap * W);
  RD_ALLOC(s->H2, sizeof(__nv_bfloat16) * cap * W);
  RD_ALLOC(s->dZ1, sizeof(__nv_bfloat16) * cap * W);
  RD_ALLOC(s->dZ2, sizeof(__nv_bfloat16) * cap * W);
  RD_ALLOC(s->dZ3, sizeof(__nv_bfloat16) * cap * W);
  RD_ALLOC(s->Z1, sizeof(float) * cap * W);
  RD_ALLOC(s->part, sizeof(float) * kMaxSplits * L.stride());
  RD_ALLOC(s->part4, sizeof(float) * (cap / 32) * (W + 1));
  s->grad_cap = rows;
  return cudaSuccess;
}
#undef RD_ALLOC

static cudaError_t refresh_bf16(rd_surrogate* s, cudaStream_t st) {
  const Layout L(s->W);
  const int n = (int)L.ob4 + 1;
  k_to_bf16<<<(n + 255) / 256, 256, 0, st>>>(n, s->params, s->Wb);
  return cudaGetLastError();
}

template <int MODE, int NR>
static cudaError_t launch_mlp(const MlpArgs& a, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(k_mlp<MODE, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)mlp_smem_bytes(NR));
  if (e != cudaSuccess) return e;
  k_mlp<MODE, NR><<<(a.B + NR - 1) / NR, kMlpThreads, mlp_smem_bytes(NR), st>>>(a);
  return cudaGetLastError();
}

// Rows per tile: 32 while that fills the SMs at most twice, each tile reading all
// weights anew (forward, calls back to back: 4096 rows 16 us against 34 with 128-row
// tiles, 9728 rows 28 against 34, 12160 rows 40 against 34); the backward pass, whose
// tiles do three times as much, once and a half (loss and gradients: 4864 rows 77 us
// against 112, 8192 rows 111 us both ways, 14592 rows 158 against 124).
static int tile_rows(int mode, int B, int n_sm) {
  const int waves2 = mode == MLP_GRAD ? 3 : 4;  // twice the waves
  return B <= waves2 * 16 * n_sm ? 32 : 128;
}

template <int MODE>
static cudaError_t launch_mlp(const MlpArgs& a, int n_sm, cudaStream_t st) {
  return tile_rows(MODE, a.B, n_sm) == 32 ? launch_mlp<MODE, 32>(a, st) : launch_mlp<MODE, 128>(a, st);
}

// One pass over B rows of theta (device [B][P]): MLP_PREDICT writes Phi~ to
// phit; MLP_LOSS writes s->out and the summed squared error against target;
// MLP_GRAD also leaves what the weight gradients need.
static cudaError_t pass(rd_surrogate* s, int mode, int B, const double* theta, double* phit,
                        const float* target, cudaStream_t st) {
  if (mode != MLP_PREDICT) {
    const cudaError_t e = cudaMemsetAsync(s->sqerr, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
  }
  MlpArgs a{};
  a.B = B;
  a.P = s->P;
  a.theta = theta;
  a.X = s->X;
  a.Wb = s->Wb;
  a.params = s->params;
  a.nm = s->norm;
  a.phit = phit;
  a.target = target;
  a.out = s->out;
  a.sq_err = s->sqerr;
  a.H1 = s->H1;
  a.H2 = s->H2;
  a.dZ1 = s->dZ1;
  a.dZ2 = s->dZ2;
  a.dZ3 = s->dZ3;
  a.Z1 = s->Z1;
  a.part4 = s->part4;
  a.err = s->pb->ws.err;
  a.wait_ns = s->pb->dev.wait_ns;
  a.stall = s->pb->dev.stall_step == RD_STALL_SURROGATE;
  const int n_sm = s->pb->n_sm;
  if (mode == MLP_PREDICT) return launch_mlp<MLP_PREDICT>(a, n_sm, st);
  if (mode == MLP_LOSS) return launch_mlp<MLP_LOSS>(a, n_sm, st);
  return launch_mlp<MLP_GRAD>(a, n_sm, st);
}

// Loss and gradient of the mean-squared error against target for B rows (a
// multiple of 128): the summed squared error into s->sqerr, all parameter
// gradients into grads.
static cudaError_t loss_grad(rd_surrogate* s, int B, const double* theta, const float* target,
                             float* grads, cudaStream_t st) {
  cudaError_t e = pass(s, MLP_GRAD, B, theta, nullptr, target, st);
  if (e != cudaSuccess) return e;
  const Layout L(s->W);
  WgradArgs g{};
  g.B = B;
  g.tiles = B / 128;
  g.splits = std::min(g.tiles, kMaxSplits);
  g.dZ[0] = s->dZ1;
  g.dZ[1] = s->dZ2;
  g.dZ[2] = s->dZ3;
  g.H[0] = s->X;
  g.H[1] = s->H1;
  g.H[2] = s->H2;
  g.part = s->part;
  g.err = s->pb->ws.err;
  g.wait_ns = s->pb->dev.wait_ns;
  g.stall = s->pb->dev.stall_step == RD_STALL_SURROGATE;
  if ((e = cudaFuncSetAttribute(k_mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kWgSmem)) != cudaSuccess)
    return e;
  k_mlp_wgrad<<<dim3(s->W / 128, 3, g.splits), kMlpThreads, kWgSmem, st>>>(g);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_mlp_reduce<<<(unsigned)((L.total + 255) / 256), 256, 0, st>>>(g.splits, B / tile_rows(MLP_GRAD, B, s->pb->n_sm), s->part,
                                                                   s->part4, grads);
  return cudaGetLastError();
}

cudaError_t adam_step(rd_surrogate* s, double lr, double b1, double b2, double eps, double wd,
                      cudaStream_t st) {
  const Layout L(s->W);
  s->adam_t += 1;
  AdamArgs a;
  a.p = s->params;
  a.g = s->grads;
  a.m = s->adam_m;
  a.v = s->adam_v;
  a.decay_mask = s->decay_mask;
  a.n = (int)L.total;
  a.lr = (float)lr;
  a.b1 = (float)b1;
  a.b2 = (float)b2;
  a.eps = (float)eps;
  a.wd = (float)wd;
  a.c1 = (float)(1.0 - pow(b1, s->adam_t));
  a.c2 = (float)(1.0 - pow(b2, s->adam_t));
  k_adam<<<(a.n + 255) / 256, 256, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return refresh_bf16(s, st);
}

cudaError_t predict(rd_surrogate* s, int B, const double* theta, double* phit, cudaStream_t st) {
  return pass(s, MLP_PREDICT, B, theta, phit, nullptr, st);
}

}  // namespace mlp
}  // namespace rd

using namespace rd;

#define RD_SCHECK(cond, code, msg) \
  do {                             \
    if (!(cond)) {                 \
      rd::set_error(msg);          \
      return code;                 \
    }                              \
  } while (0)
#define RD_SCUDA(call)                                                     \
  do {                                                                     \
    cudaError_t e_ = (call);                                               \
    if (e_ != cudaSuccess) {                                               \
      rd::set_error(std::string(#call) + ": " + cudaGetErrorString(e_));   \
      return RD_ECUDA;                                                     \
    }                                                                      \
  } while (0)

extern "C" {

rd_status rd_surrogate_destroy(rd_surrogate* s) {
  if (!s) return RD_OK;
  if (s->pb) cudaStreamSynchronize(s->pb->stream);
  rd::mlp::free_acts(s);
  rd::mlp::free_grad(s);
  cudaFree(s->params);
  cudaFree(s->grads);
  cudaFree(s->adam_m);
  cudaFree(s->adam_v);
  cudaFree(s->decay_mask);
  cudaFree(s->Wb);
  delete s;
  return RD_OK;
}

rd_status rd_surrogate_create(rd_problem* p, uint64_t seed, rd_surrogate** out) {
  RD_SCHECK(p && out, RD_EINVAL, "NULL argument");
  *out = nullptr;
  rd_surrogate* s = new rd_surrogate();
  s->pb = p;
  s->P = p->desc.n_params;
  s->W = RD_SURROGATE_WIDTH;
  const mlp::Layout L(s->W);
  // He-uniform initial weights (bound sqrt(6 / fan_in)); last layer scaled by
  // 0.1; biases zero.  A 64-bit linear congruential stream seeded by `seed`.
  std::vector<float> h(L.total, 0.f);
  std::vector<uint8_t> mask(L.total, 0);
  uint64_t state = seed * 6364136223846793005ull + 1442695040888963407ull;
  auto uni = [&]() {
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return (double)(state >> 11) * (1.0 / 9007199254740992.0);
  };
  auto fill = [&](size_t off, int rows, int cols, int fan_in, double scale) {
    const double bound = sqrt(6.0 / fan_in) * scale;
    for (int r = 0; r < rows; ++r)
      for (int c = 0; c < cols; ++c) {
        h[off + (size_t)r * cols + c] = (float)((2.0 * uni() - 1.0) * bound);
        mask[off + (size_t)r * cols + c] = 1;
      }
  };
  fill(L.oW1, s->W, mlp::kIn, s->P, 1.0);
  for (int r = 0; r < s->W; ++r)  // padded inputs carry no weight
    for (int c = s->P; c < mlp::kIn; ++c) h[L.oW1 + (size_t)r * mlp::kIn + c] = 0.f;
  fill(L.oW2, s->W, s->W, s->W, 1.0);
  fill(L.oW3, s->W, s->W, s->W, 1.0);
  fill(L.oW4, 1, s->W, s->W, 0.1);
  for (int j = 0; j < RD_NPARAM; ++j) {
    s->norm.in_mu[j] = 0.0;
    s->norm.in_sd[j] = 1.0;
  }
  s->norm.floor = 0.0;
  s->norm.shift = 0.0;
  s->norm.scale = 1.0;
  bool ok = cudaMalloc(&s->params, sizeof(float) * L.total) == cudaSuccess &&
            cudaMalloc(&s->grads, sizeof(float) * L.total) == cudaSuccess &&
            cudaMalloc(&s->adam_m, sizeof(float) * L.total) == cudaSuccess &&
            cudaMalloc(&s->adam_v, sizeof(float) * L.total) == cudaSuccess &&
            cudaMalloc(&s->decay_mask, L.total) == cudaSuccess &&
            cudaMalloc(&s->Wb, sizeof(__nv_bfloat16) * (L.ob4 + 1)) == cudaSuccess;
  ok = ok && cudaMemcpy(s->params, h.data(), sizeof(float) * L.total, cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemcpy(s->decay_mask, mask.data(), L.total, cudaMemcpyHostToDevice) == cudaSuccess &&
       cudaMemset(s->grads, 0, sizeof(float) * L.total) == cudaSuccess &&
       cudaMemset(s->adam_m, 0, sizeof(float) * L.total) == cudaSuccess &&
       cudaMemset(s->adam_v, 0, sizeof(float) * L.total) == cudaSuccess &&
       mlp::refresh_bf16(s, p->stream) == cudaSuccess &&
       cudaStreamSynchronize(p->stream) == cudaSuccess;
  if (!ok) {
    rd_surrogate_destroy(s);
    set_error("surrogate allocation failed");
    return RD_ENOMEM;
  }
  *out = s;
  return RD_OK;
}

rd_status rd_surrogate_get_params(rd_surrogate* s, float* host, size_t cap, size_t* n,
                                  double* norm) {
  RD_SCHECK(s && n, RD_EINVAL, "NULL argument");
  const mlp::Layout L(s->W);
  *n = L.total;
  if (host) {
    RD_SCHECK(cap >= L.total, RD_EINVAL, "parameter buffer too small");
    RD_SCUDA(cudaStreamSynchronize(s->pb->stream));
    RD_SCUDA(cudaMemcpy(host, s->params, sizeof(float) * L.total, cudaMemcpyDeviceToHost));
  }
  if (norm) {
    for (int j = 0; j < RD_NPARAM; ++j) {
      norm[j] = s->norm.in_mu[j];
      norm[RD_NPARAM + j] = s->norm.in_sd[j];
    }
    norm[2 * RD_NPARAM] = s->norm.floor;
    norm[2 * RD_NPARAM + 1] = s->norm.shift;
    norm[2 * RD_NPARAM + 2] = s->norm.scale;
  }
  return RD_OK;
}

rd_status rd_surrogate_set_params(rd_surrogate* s, const float* host, size_t n,
                                  const double* norm) {
  RD_SCHECK(s, RD_EINVAL, "NULL argument");
  const mlp::Layout L(s->W);
  if (host) {
    RD_SCHECK(n == L.total, RD_EINVAL, "parameter count mismatch");
    RD_SCUDA(cudaStreamSynchronize(s->pb->stream));
    RD_SCUDA(cudaMemcpy(s->params, host, sizeof(float) * L.total, cudaMemcpyHostToDevice));
    RD_SCUDA(mlp::refresh_bf16(s, s->pb->stream));
    RD_SCUDA(cudaStreamSynchronize(s->pb->stream));
  }
  if (norm) {
    for (int j = 0; j < RD_NPARAM; ++j) {
      RD_SCHECK(norm[RD_NPARAM + j] > 0, RD_EINVAL, "input scales must be positive");
      s->norm.in_mu[j] = norm[j];
      s->norm.in_sd[j] = norm[RD_NPARAM + j];
    }
    s->norm.floor = norm[2 * RD_NPARAM];
    s->norm.shift = norm[2 * RD_NPARAM + 1];
    s->norm.scale = norm[2 * RD_NPARAM + 2];
    s->pb->generation++;  // captured sampler graphs hold the normalisation by value
  }
  return RD_OK;
}

rd_status rd_surrogate_loss_grad(rd_surrogate* s, int B, const double* theta,
                                 const float* target, double* loss, float* grads) {
  RD_SCHECK(s && theta && target && loss, RD_EINVAL, "NULL argument");
  RD_SCHECK(B >= 128 && B % 128 == 0, RD_EINVAL, "B must be a positive multiple of 128");
  cudaStream_t st = s->pb->stream;
  RD_SCUDA(mlp::ensure_grad_rows(s, B));
  RD_SCUDA(mlp::loss_grad(s, B, theta, target, grads ? grads : s->grads, st));
  double se = 0.0;
  RD_SCUDA(cudaMemcpyAsync(&se, s->sqerr, sizeof(double), cudaMemcpyDeviceToHost, st));
  RD_SCUDA(cudaStreamSynchronize(st));
  *loss = se / B;
  return RD_OK;
}

rd_status rd_surrogate_predict(rd_surrogate* s, int B, const double* theta, double* phi_tilde) {
  RD_SCHECK(s && theta && phi_tilde, RD_EINVAL, "NULL argument");
  RD_SCHECK(B >= 0, RD_EINVAL, "B must be >= 0");
  if (B == 0) return RD_OK;
  RD_SCUDA(mlp::ensure_rows(s, B));
  RD_SCUDA(mlp::predict(s, B, theta, phi_tilde, s->pb->stream));
  return RD_OK;
}

rd_status rd_surrogate_train(rd_surrogate* s, int n, const double* theta, const double* phi,
                             const rd_train_desc* td, double* report) {
  RD_SCHECK(s && theta && phi && td, RD_EINVAL, "NULL argument");
  RD_SCHECK(td->batch >= 128 && td->batch % 128 == 0, RD_EINVAL,
            "batch must be a positive multiple of 128");
  RD_SCHECK(td->epochs >= 1 && td->lr > 0, RD_EINVAL, "epochs >= 1 and lr > 0 required");
  cudaStream_t st = s->pb->stream;
  const int P = s->P;
  // host copies: normalisation and the shuffled order need them once
  std::vector<double> th((size_t)n * P), ph(n);
  RD_SCUDA(cudaStreamSynchronize(st));
  RD_SCUDA(cudaMemcpy(th.data(), theta, sizeof(double) * th.size(), cudaMemcpyDeviceToHost));
  RD_SCUDA(cudaMemcpy(ph.data(), phi, sizeof(double) * ph.size(), cudaMemcpyDeviceToHost));
  std::vector<int> keep;
  keep.reserve(n);
  double pmin = INFINITY;
  for (int i = 0; i < n; ++i) {
    bool ok = std::isfinite(ph[i]);
    for (int j = 0; j < P && ok; ++j) ok = th[(size_t)i * P + j] > 0;
    if (ok) {
      keep.push_back(i);
      pmin = std::min(pmin, ph[i]);
    }
  }
  RD_SCHECK((int)keep.size() >= 2 * td->batch, RD_EINVAL,
            "too few finite training pairs for two batches");
  // normalisation: inputs by the mean/sd of log theta, targets
  // z = log(phi - floor) standardised, floor = min phi - 1
  mlp::Norm nm{};
  for (int j = 0; j < RD_NPARAM; ++j) {
    nm.in_mu[j] = 0.0;
    nm.in_sd[j] = 1.0;
  }
  for (int j = 0; j < P; ++j) {
    double m = 0, v = 0;
    for (int i : keep) m += log(th[(size_t)i * P + j]);
    m /= keep.size();
    for (int i : keep) {
      const double d = log(th[(size_t)i * P + j]) - m;
      v += d * d;
    }
    nm.in_mu[j] = m;
    nm.in_sd[j] = std::max(sqrt(v / keep.size()), 1e-12);
  }
  nm.floor = pmin - 1.0;
  double zm = 0, zv = 0;
  for (int i : keep) zm += log(ph[i] - nm.floor);
  zm /= keep.size();
  for (int i : keep) {
    const double d = log(ph[i] - nm.floor) - zm;
    zv += d * d;
  }
  nm.shift = zm;
  nm.scale = std::max(sqrt(zv / keep.size()), 1e-12);
  s->norm = nm;
  s->pb->generation++;
  // seeded shuffle, hold-out split
  uint64_t state = td->seed * 2862933555777941757ull + 3037000493ull;
  auto next = [&]() {
    state = state * 6364136223846793005ull + 1442695040888963407ull;
    return state >> 33;
  };
  for (size_t i = keep.size() - 1; i > 0; --i) std::swap(keep[i], keep[next() % (i + 1)]);
  const int n_hold = std::max(td->batch, (int)(td->holdout_frac * keep.size()) / td->batch * td->batch);
  const int n_train = ((int)keep.size() - n_hold) / td->batch * td->batch;
  RD_SCHECK(n_train >= td->batch, RD_EINVAL, "too few training pairs after the hold-out split");
  std::vector<double> th_s((size_t)(n_train + n_hold) * P);
  std::vector<float> z_s(n_train + n_hold);
  for (int r = 0; r < n_train + n_hold; ++r) {
    const int i = keep[r];
    for (int j = 0; j < P; ++j) th_s[(size_t)r * P + j] = th[(size_t)i * P + j];
    z_s[r] = (float)((log(ph[i] - nm.floor) - nm.shift) / nm.scale);
  }
  double* d_th = nullptr;
  float* d_z = nullptr;
  RD_SCUDA(cudaMalloc(&d_th, sizeof(double) * th_s.size()));
  RD_SCUDA(cudaMalloc(&d_z, sizeof(float) * z_s.size()));
  RD_SCUDA(cudaMemcpy(d_th, th_s.data(), sizeof(double) * th_s.size(), cudaMemcpyHostToDevice));
  RD_SCUDA(cudaMemcpy(d_z, z_s.data(), sizeof(float) * z_s.size(), cudaMemcpyHostToDevice));
  RD_SCUDA(mlp::ensure_grad_rows(s, td->batch));
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, st);
  const int nb = n_train / td->batch;
  double train_mse = 0.0;
  std::vector<double> ep_se(nb);
  for (int ep = 0; ep < td->epochs; ++ep) {
    // batches in a seeded order each epoch
    std::vector<int> order(nb);
    for (int b = 0; b < nb; ++b) order[b] = b;
    for (int b = nb - 1; b > 0; --b) std::swap(order[b], order[next() % (b + 1)]);
    double se = 0.0;
    for (int k = 0; k < nb; ++k) {
      const int b = order[k];
      RD_SCUDA(mlp::loss_grad(s, td->batch, d_th + (size_t)b * td->batch * P,
                              d_z + (size_t)b * td->batch, s->grads, st));
      RD_SCUDA(mlp::adam_step(s, td->lr, td->beta1, td->beta2, 1e-8, td->weight_decay, st));
      if (ep == td->epochs - 1) {
        double v = 0.0;
        RD_SCUDA(cudaMemcpyAsync(&v, s->sqerr, sizeof(double), cudaMemcpyDeviceToHost, st));
        RD_SCUDA(cudaStreamSynchronize(st));
        se += v;
      }
    }
    if (ep == td->epochs - 1) train_mse = se / n_train;
  }
  // hold-out error in target units and in Phi units
  double hold_se = 0.0, hold_abs = 0.0;
  std::vector<float> outv(td->batch);
  for (int off = n_train; off + td->batch <= n_train + n_hold; off += td->batch) {
    RD_SCUDA(mlp::pass(s, mlp::MLP_LOSS, td->batch, d_th + (size_t)off * P, nullptr, d_z + off, st));
    double v = 0.0;
    RD_SCUDA(cudaMemcpyAsync(&v, s->sqerr, sizeof(double), cudaMemcpyDeviceToHost, st));
    RD_SCUDA(cudaMemcpyAsync(outv.data(), s->out, sizeof(float) * td->batch, cudaMemcpyDeviceToHost, st));
    RD_SCUDA(cudaStreamSynchronize(st));
    hold_se += v;
    for (int r = 0; r < td->batch; ++r) {
      const double pt = nm.floor + exp(nm.shift + nm.scale * (double)outv[r]);
      const double pe = nm.floor + exp(nm.shift + nm.scale * (double)z_s[off + r]);
      hold_abs += fabs(pt - pe) / pe;
    }
  }
  cudaEventRecord(e1, st);
  cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(d_th);
  cudaFree(d_z);
  int err = 0;
  RD_SCUDA(cudaMemcpy(&err, s->pb->ws.err, sizeof(int), cudaMemcpyDeviceToHost));
  RD_SCHECK(!err, RD_ETIMEOUT, "a training kernel's bounded wait gave up");
  if (report) {
    report[0] = train_mse;
    report[1] = hold_se / std::max(n_hold, 1);
    report[2] = hold_abs / std::max(n_hold, 1);
    report[3] = ms * 1e-3;
  }
  return RD_OK;
}

}  // extern "C"
