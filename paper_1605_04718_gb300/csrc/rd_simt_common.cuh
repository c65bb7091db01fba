// rd_simt_common.cuh -- CUDA-core building blocks of the 2-D FP32 solves
// (rd_solve_simt.cu, rd_solve_cg.cu): the solve of [alpha I - beta Lap_h] by
// shared-memory GEMMs in the cosine basis of one direction and scans along the
// other, and CTA-wide sums.
#pragma once

#include <cuda_runtime.h>

#include "rd_scan.cuh"
#include "rd_tc_ptx.cuh"

namespace rd {

constexpr int kSimtThreads = 256;

template <int N>
constexpr size_t simt_smem_bytes() {
  return (size_t)3 * N * (N + 1) * sizeof(float);
}

// acc[i][j] = sum_k A(ty + 16 i, k) B(k, tx + 16 j), A(m, k) = pa[m*SAM + k*SAK],
// B(k, n) = pb[k*SBK + n*SBN].
template <int N, int SAM, int SAK, int SBK, int SBN>
__device__ __forceinline__ void smem_gemm(const float* __restrict__ pa,
                                          const float* __restrict__ pb,
                                          float (&acc)[N / 16][N / 16], int ty,
                                          int tx) {
  constexpr int TM = N / 16;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = 0.f;
#pragma unroll 4
  for (int k = 0; k < N; ++k) {
    float av[TM], bv[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) av[i] = pa[(ty + 16 * i) * SAM + k * SAK];
#pragma unroll
    for (int j = 0; j < TM; ++j) bv[j] = pb[k * SBK + (tx + 16 * j) * SBN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
}

template <int N>
__device__ __forceinline__ void store_tile(float* W, const float (&acc)[N / 16][N / 16],
                                           int ty, int tx) {
  constexpr int TM = N / 16, NP = N + 1;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) W[(ty + 16 * i) * NP + tx + 16 * j] = acc[i][j];
}

// Segments of a column in the scan: NS of H rows, one thread each.
template <int N>
struct SimtSeg {
  static constexpr int NS = N <= 16 ? 4 : N <= 32 ? 8 : N <= 64 ? 4 : 2;
  static constexpr int H = N / NS;
  static_assert(NS * N <= kSimtThreads && NS * H == N, "");
};

// X <- [(alpha + beta mu_k) I - beta Lap_1D]^-1 X along y for every column k of W
// (rows y, padded to N + 1): the recursions of rd_scan.cuh, N / NS rows a thread.
// sums: [NS][N] scratch.
template <int N>
__device__ __forceinline__ void scan_columns(float* W, float alpha, float beta, const float* mu,
                                             float2* sums) {
  constexpr int NP = N + 1, NS = SimtSeg<N>::NS, H = SimtSeg<N>::H;
  const int k = threadIdx.x % N, seg = threadIdx.x / N;
  const bool on = seg < NS;
  float* const w = W + (on ? seg : 0) * H * NP + k;
  const ScanCoef c = scan_coef<N, H>(alpha, beta, mu[k], 1.f);
  float r[H];
#pragma unroll
  for (int m = 0; m < H; ++m) r[m] = w[m * NP];
  float L, R;
  scan_sums<H>(r, c.a, L, R);
  if (on) sums[seg * N + k] = make_float2(L, R);
  __syncthreads();
  float Lt = sums[(NS - 1) * N + k].x, Rt = sums[k].y;  // of the whole column
#pragma unroll
  for (int i = 1; i < NS; ++i) {
    Lt = fmaf(c.ah, Lt, sums[(NS - 1 - i) * N + k].x);
    Rt = fmaf(c.ah, Rt, sums[i * N + k].y);
  }
  float left = fmaf(c.an, Rt, Lt) * c.inv, right = fmaf(c.an, Lt, Rt) * c.inv;
#pragma unroll
  for (int i = 0; i < NS - 1; ++i) {
    if (i < seg) left = fmaf(c.ah, left, sums[i * N + k].y);
    if (NS - 1 - i > seg) right = fmaf(c.ah, right, sums[(NS - 1 - i) * N + k].x);
  }
#pragma unroll
  for (int m = 0; m < H; ++m) {
    left = fmaf(c.a, left, r[m]);
    r[m] = left;
  }
  float x = fmaf(c.a, right, left) * c.g;
  if (on) w[(H - 1) * NP] = x * c.sc;
#pragma unroll
  for (int m = H - 2; m >= 0; --m) {
    x = fmaf(c.a, x, r[m]);
    if (on) w[m * NP] = x * c.sc;
  }
  __syncthreads();
}

// In place: W <- [alpha I - beta Lap_h]^-1 W.  Two transforms along x and a scan
// along y; outside the scan's range (alpha <= 0, beta < 0 or not finite) four
// transforms and the division by the eigenvalues.  mu: the eigenvalues, sums:
// 256 float2 of scratch.  A step of the CUDA-core kernel, per proposal, four
// transforms -> two and a scan: 64^2 0.251 -> 0.145 us, 128^2 0.899 -> 0.406 us.
template <int N>
__device__ __forceinline__ void implicit_solve_simt(float* W, const float* Cm, float alpha,
                                                    float beta, const float* mu, float2* sums,
                                                    int ty, int tx) {
  constexpr int TM = N / 16, NP = N + 1;
  const bool scan = alpha > 0.f && beta >= 0.f && beta < 1e30f;
  float acc[TM][TM];
  // P[y][k] = sum_x W[y][x] C[k][x]
  smem_gemm<N, NP, 1, 1, NP>(W, Cm, acc, ty, tx);
  __syncthreads();
  store_tile<N>(W, acc, ty, tx);
  __syncthreads();
  if (scan) {
    scan_columns<N>(W, alpha, beta, mu, sums);
  } else {
    // Q[l][k] = sum_y C[l][y] P[y][k];  S = Q / (alpha + beta (mu_l + mu_k))
    smem_gemm<N, NP, 1, NP, 1>(Cm, W, acc, ty, tx);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j)
        acc[i][j] *= tc::recip_nr(fmaf(beta, mu[ty + 16 * i] + mu[tx + 16 * j], alpha));
    __syncthreads();
    store_tile<N>(W, acc, ty, tx);
    __syncthreads();
    // W1[y][k] = sum_l C[l][y] S[l][k]
    smem_gemm<N, 1, NP, NP, 1>(Cm, W, acc, ty, tx);
    __syncthreads();
    store_tile<N>(W, acc, ty, tx);
    __syncthreads();
  }
  // W[y][x] = sum_k W1[y][k] C[k][x]
  smem_gemm<N, NP, 1, NP, 1>(W, Cm, acc, ty, tx);
  __syncthreads();
  store_tile<N>(W, acc, ty, tx);
  __syncthreads();
}

// ------------------------------------------------------------ compensated sums
// A sum of FP32 values or products held as an unevaluated pair s + c: every
// addition's rounding error is recovered exactly (Knuth's two-sum; products by
// FMA) and collected in c, so the sum carries about 46 bits.  The FP64 pipe takes
// 64 cycles per warp instruction and an FP64 dot product needs three of them per
// element (two conversions and an FMA); this needs 11 FP32 instructions.
struct Pair {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x, float low = 0.f) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
    c = __fadd_rn(c, __fadd_rn(e, low));
    s = t;
  }
  __device__ __forceinline__ void add_product(float x, float y) {
    const float p = __fmul_rn(x, y);
    add(p, __fmaf_rn(x, y, -p));
  }
};

// Scratch of cta_reduce.
struct RedScratch {
  float2 part[kSimtThreads / 32];
  double out;
};

// f(sum over the CTA), f evaluated in thread 0 (so that its FP64 operations are
// done once); the result in every thread.
template <class F>
__device__ __forceinline__ double cta_reduce(Pair v, RedScratch* red, F&& f) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v.add(__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red->part[warp] = make_float2(v.s, v.c);
  __syncthreads();
  if (warp == 0) {
    const float2 p = red->part[lane & 7];
    Pair t;
    t.s = p.x;
    t.c = p.y;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
      t.add(__shfl_xor_sync(0xffffffffu, t.s, o), __shfl_xor_sync(0xffffffffu, t.c, o));
    if (lane == 0) red->out = f((double)t.s + (double)t.c);
  }
  __syncthreads();
  return red->out;
}
static_assert(kSimtThreads == 256, "cta_reduce combines 8 warps");

// FP64 sum over the CTA; result valid in thread 0.
__device__ __forceinline__ double cta_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  __syncthreads();
  return s;
}

// FP64 sum over the CTA, returned to every thread.
__device__ __forceinline__ double cta_sum_all(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  __syncthreads();
  return s;
}

}  // namespace rd
