// rd_scan.cuh -- the tridiagonal half of the 2-D implicit solve.
//
// With one direction in the cosine basis, [alpha I - beta Lap_h] w = r falls
// apart into one system per mode k along the other direction,
//   (lam + 2 beta) x_i - beta (x_{i-1} + x_{i+1}) = r_i,   lam = alpha + beta mu_k,
// with x mirrored at both ends (x_{-1} = x_0, x_N = x_{N-1}).  For lam > 0 and
// beta >= 0 its matrix factors into two first-order recursions,
//   (beta / a) (1 - a S) (1 - a S^-1) x = r,   a + 1/a = 2 + lam / beta,  0 <= a < 1
// (S the shift), so a row is solved by one sweep up and one sweep down:
//   F_i = r_i + a F_{i-1},   X_i = F_i + a X_{i+1},   x = (a / beta) X.
// The mirrored ends are periodic images of the row, so what enters a segment
// from outside is a geometric sum of the row's own values: with
// L = sum a^m r_m and R = sum a^{H-1-m} r_m over a segment of H nodes, the
// values entering at its ends follow from the L and R of the row's segments
// (scan_entries*).  All recursions contract while a, rounded, is below 1.
//
// a is rounded to FP32 first and the output scale a / beta is then taken as
// (1 - a)^2 / lam with that rounded a: the mean of every mode is solved to
// rounding, and the rounding of a acts like a relative change of beta of at
// most 2^-23 / (1 - a), the same at every step.
//
// Range.  1 - a is about sqrt(lam / beta), so with beta / alpha beyond about 2.8e14
// the rounded a is 1 and the row infinite or NaN.  The scan is used up to
// beta / alpha = kScanMaxRatio, where 1 - a = 1e-5 is still 168 units of a's last
// place: rows of N = 16 to 128 are solved to 3e-6 of their norm at most below it and
// 1.5e-6 at it (1e-7 in the median), modelled in float32 against float64 in the
// cosine basis.
#pragma once

#include <cuda_runtime.h>

namespace rd {

constexpr float kScanMaxRatio = 1e10f;  // largest beta / alpha the scan is used for

struct ScanCoef {
  float a;     // ratio of the recursions
  float sc;    // output scale (a / beta) * out_scale
  float g;     // 1 / (1 - a^2)
  float ah;    // a^H, H the segment length
  float an;    // a^N
  float inv;   // 1 / (1 - a^(2N))
};

// Segments of a row: NS of H nodes.
template <int N>
struct ScanSeg {
  static constexpr int NS = N >= 48 ? 2 : 1;
  static constexpr int H = N / NS;
};

// x^K by repeated squaring (K a compile-time constant).
template <int K>
__device__ __forceinline__ float ipow(float x) {
  if constexpr (K == 1) {
    return x;
  } else {
    const float h = ipow<K / 2>(x);
    return (K & 1) ? h * h * x : h * h;
  }
}

// Coefficients of one mode; N a multiple of 16, H the segments' length.
template <int N, int H = ScanSeg<N>::H>
__device__ __forceinline__ ScanCoef scan_coef(float alpha, float beta, float mu, float out_scale) {
  ScanCoef c;
  const float lam = fmaf(beta, mu, alpha);
  float a = 0.f;
  if (beta > 0.f) {
    const float h = 0.5f * __fdiv_rn(lam, beta);
    a = __frcp_rn(1.f + (h + __fsqrt_rn(fmaf(h, h, h + h))));
  }
  const float om = 1.f - a;
  c.a = a;
  c.sc = __fdiv_rn(om * om, lam) * out_scale;
  c.g = __frcp_rn(om * (1.f + a));
  c.ah = ipow<H>(a);
  c.an = ipow<N>(a);
  // 1 - a^(2N) = (1 - a)(1 + a)(1 + a^2)...(1 + a^16)(1 + a^32 + ... ): no
  // cancellation for a near 1
  const float a2 = a * a, a4 = a2 * a2, a8 = a4 * a4, a16 = a8 * a8, a32 = a16 * a16;
  float geo = 1.f;
#pragma unroll
  for (int i = 1; i < N / 16; ++i) geo = fmaf(geo, a32, 1.f);
  const float one_m = om * (1.f + a) * (1.f + a2) * (1.f + a4) * (1.f + a8) * (1.f + a16) * geo;
  c.inv = __frcp_rn(one_m);
  return c;
}

// L = sum_m a^m r_m and R = sum_m a^(H-1-m) r_m.
template <int H>
__device__ __forceinline__ void scan_sums(const float (&r)[H], float a, float& L, float& R) {
  L = r[H - 1];
  R = r[0];
#pragma unroll
  for (int m = 1; m < H; ++m) {
    L = fmaf(a, L, r[H - 1 - m]);
    R = fmaf(a, R, r[m]);
  }
}

// What enters segment s of a row from the left (the value of F before it) and
// from the right (sum a^m r beyond it), from the sums (L, R) of all segments.
template <int NS>
__device__ __forceinline__ void scan_entries(const float2 (&lr)[NS], int s, const ScanCoef& k,
                                             float& left, float& right) {
  float Lt = lr[NS - 1].x, Rt = lr[0].y;  // of the whole row
  if (NS == 2) {
    Lt = fmaf(k.ah, Lt, lr[0].x);
    Rt = fmaf(k.ah, Rt, lr[NS - 1].y);
  }
  left = fmaf(k.an, Rt, Lt) * k.inv;
  right = fmaf(k.an, Lt, Rt) * k.inv;
  if (NS == 2) {
    if (s == 1) left = fmaf(k.ah, left, lr[0].y);
    if (s == 0) right = fmaf(k.ah, right, lr[NS - 1].x);
  }
}

}  // namespace rd
