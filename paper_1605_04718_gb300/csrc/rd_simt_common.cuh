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

// Row stride of the arrays in shared memory: rows start on 16-byte boundaries a
// bank group apart, so that four consecutive values load at once without
// conflicts.  96: one more float, two CTAs of three arrays then fit an SM.
__host__ __device__ constexpr int simt_stride(int n) { return n == 96 ? n + 1 : n + 4; }

// Column j of the N / 16 that thread tx owns: in groups of four or two where
// N / 16 allows, for wide loads of row-major B.
template <int N>
__device__ __forceinline__ constexpr int simt_col(int tx, int j) {
  constexpr int TM = N / 16, G = simt_stride(N) % 4 ? 1 : TM % 4 == 0 ? 4 : TM % 2 == 0 ? 2 : 1;
  return (j / G) * 16 * G + tx * G + j % G;
}

template <int M>
__device__ __forceinline__ void load_vec(const float* p, float (&v)[M]) {
  if constexpr (M == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else if constexpr (M == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x, v[1] = x.y;
  } else {
    v[0] = p[0];
  }
}

// acc[i][j] = sum_k A(ty + 16 i, k) B(k, n_j).  A(m, k) = pa[m * NP + k], or
// pa[k * NP + m] if A_T.  BT: B(k, n) = pb[n * NP + k], n_j = tx + 16 j; else
// B(k, n) = pb[k * NP + n], n_j = simt_col(tx, j).  Operands along k are loaded
// four at a time: 8 loads for 64 FMAs at N = 64 instead of 32, which bound it
// (a step of the CUDA-core kernel at 64^2, per proposal, 0.145 -> 0.123 us).
template <int N, bool A_T, bool BT>
__device__ __forceinline__ void smem_gemm(const float* __restrict__ pa,
                                          const float* __restrict__ pb,
                                          float (&acc)[N / 16][N / 16], int ty, int tx) {
  constexpr int TM = N / 16, NP = simt_stride(N);
  constexpr int V = NP % 4 == 0 ? 4 : 1;
  constexpr int G = simt_col<N>(0, 1) == 1 ? (TM > 2 && simt_col<N>(0, 2) == 2 ? 4 : 2) : 1;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = 0.f;
#pragma unroll(V == 4 ? 1 : 4)
  for (int k = 0; k < N; k += V) {
    float av[TM][V];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if constexpr (A_T) {
#pragma unroll
        for (int e = 0; e < V; ++e) av[i][e] = pa[(k + e) * NP + ty + 16 * i];
      } else {
        load_vec<V>(pa + (ty + 16 * i) * NP + k, av[i]);
      }
    }
    if constexpr (BT) {
#pragma unroll
      for (int j = 0; j < TM; ++j) {
        float bv[V];
        load_vec<V>(pb + (tx + 16 * j) * NP + k, bv);
#pragma unroll
        for (int e = 0; e < V; ++e)
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(av[i][e], bv[e], acc[i][j]);
      }
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e)
#pragma unroll
        for (int j = 0; j < TM; j += G) {
          float bv[G];
          load_vec<G>(pb + (k + e) * NP + simt_col<N>(tx, j), bv);
#pragma unroll
          for (int h = 0; h < G; ++h)
#pragma unroll
            for (int i = 0; i < TM; ++i) acc[i][j + h] = fmaf(av[i][e], bv[h], acc[i][j + h]);
        }
    }
  }
}

// The tile of a product whose columns are tx + 16 j (BT) or simt_col(tx, j).
template <int N, bool BT>
__device__ __forceinline__ void store_tile(float* W, const float (&acc)[N / 16][N / 16],
                                           int ty, int tx) {
  constexpr int TM = N / 16, NP = simt_stride(N);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j)
      W[(ty + 16 * i) * NP + (BT ? tx + 16 * j : simt_col<N>(tx, j))] = acc[i][j];
}

// Segments of a column in the scan: NS of H rows, one thread each.
template <int N>
struct SimtSeg {
  static constexpr int NS = N <= 16 ? 4 : N <= 32 ? 8 : N <= 64 ? 4 : 2;
  static constexpr int H = N / NS;
  static_assert(NS * N <= kSimtThreads && NS * H == N, "");
};

// X <- [(alpha + beta mu_k) I - beta Lap_1D]^-1 X along y for every column k of W
// (rows y, stride simt_stride): the recursions of rd_scan.cuh, N / NS rows a thread.
// sums: [NS][N] scratch.
template <int N>
__device__ __forceinline__ void scan_columns(float* W, float alpha, float beta, const float* mu,
                                             float2* sums) {
  constexpr int NP = simt_stride(N), NS = SimtSeg<N>::NS, H = SimtSeg<N>::H;
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
// along y; outside the scan's range (alpha <= 0, beta < 0, beta / alpha above
// kScanMaxRatio or not finite) four transforms and the division by the
// eigenvalues.  mu: the eigenvalues, sums: 256 float2 of scratch.  A step of the
// CUDA-core kernel, per proposal, four transforms -> two and a scan: 64^2 0.251 ->
// 0.145 us, 128^2 0.899 -> 0.406 us.
template <int N>
__device__ __forceinline__ void implicit_solve_simt(float* W, const float* Cm, float alpha,
                                                    float beta, const float* mu, float2* sums,
                                                    int ty, int tx) {
  constexpr int TM = N / 16;
  const bool scan = alpha > 0.f && beta >= 0.f && beta <= kScanMaxRatio * alpha;
  float acc[TM][TM];
  // P[y][k] = sum_x W[y][x] C[k][x]
  smem_gemm<N, false, true>(W, Cm, acc, ty, tx);
  __syncthreads();
  store_tile<N, true>(W, acc, ty, tx);
  __syncthreads();
  if (scan) {
    scan_columns<N>(W, alpha, beta, mu, sums);
  } else {
    // Q[l][k] = sum_y C[l][y] P[y][k];  S = Q / (alpha + beta (mu_l + mu_k))
    smem_gemm<N, false, false>(Cm, W, acc, ty, tx);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j)
        acc[i][j] *= tc::recip_nr(fmaf(beta, mu[ty + 16 * i] + mu[simt_col<N>(tx, j)], alpha));
    __syncthreads();
    store_tile<N, false>(W, acc, ty, tx);
    __syncthreads();
    // W1[y][k] = sum_l C[l][y] S[l][k]
    smem_gemm<N, true, false>(Cm, W, acc, ty, tx);
    __syncthreads();
    store_tile<N, false>(W, acc, ty, tx);
    __syncthreads();
  }
  // W[y][x] = sum_k W1[y][k] C[k][x]
  smem_gemm<N, false, false>(W, Cm, acc, ty, tx);
  __syncthreads();
  store_tile<N, false>(W, acc, ty, tx);
  __syncthreads();
}

// ------------------------------------------------------------ compensated sums
// A sum of FP32 values or products held as an unevaluated pair s + c: every
// addition's rounding error is recovered exactly (Knuth's two-sum; products by
// FMA) and collected in c, so the sum carries about 46 bits.  The FP64 pipe takes
// 64 cycles per warp instruction and an FP64 dot product needs three of them per
// element (two conversions and an FMA); this needs 11 FP32 instructions.
//
// The exponent range is FP32's: a product above 2^128 overflows, and what is lost of
// products near the smallest value is at most 2^-149 each, 2^-135.8 for 96^2, so 46 bits
// need a sum of kPairMin or more.  A sum out of that range is reported, and the
// proposal solved with Sum64 instead.
constexpr float kPairMin = 0x1p-89f;
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

// The same in FP64, for any range.
struct Sum64 {
  double s = 0.0;
  __device__ __forceinline__ void add(float x) { s += (double)x; }
  __device__ __forceinline__ void add_product(float x, float y) { s += (double)x * (double)y; }
};

// Scratch of cta_reduce.
struct RedScratch {
  float2 part[kSimtThreads / 32];
  double part64[kSimtThreads / 32];
  double out;
};

// f(sum over the CTA), f evaluated in thread 0 (so that its FP64 operations are
// done once); the result in every thread.  ok: cleared in warp 0 by a sum out of the
// pairs' range.
template <class F>
__device__ __forceinline__ double cta_reduce(Pair v, RedScratch* red, bool& ok, F&& f) {
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
    // t.c is a small part of t.s, and finite where t.s is
    ok = ok && fabsf(t.s) >= kPairMin && fabsf(t.s) <= 3.4028234e38f;
    if (lane == 0) red->out = f((double)t.s + (double)t.c);
  }
  __syncthreads();
  return red->out;
}
static_assert(kSimtThreads == 256, "cta_reduce combines 8 warps");

template <class F>
__device__ __forceinline__ double cta_reduce(Sum64 v, RedScratch* red, bool&, F&& f) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v.s += __shfl_xor_sync(0xffffffffu, v.s, o);
  if ((threadIdx.x & 31) == 0) red->part64[threadIdx.x >> 5] = v.s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < kSimtThreads / 32; ++i) t += red->part64[i];
    red->out = f(t);
  }
  __syncthreads();
  return red->out;
}

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
