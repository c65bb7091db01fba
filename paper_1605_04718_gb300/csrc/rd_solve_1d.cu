// rd_solve_1d.cu -- forward solves on the interval, FP64.
//
// The IMEX Euler step of Sec. 3.1.1 or the paper's semi-implicit step, and
// Phi = sum (y - w)^2 / (2 sigma^2) at the observation steps.
//
// What bounds it: the FP64 pipe takes one warp instruction per 64 cycles and
// SM quarter however many lanes are active (a division 345), so a step costs
// its FP64 instructions per warp, and lanes that do the same instruction on
// other data are free.  One thread per proposal is the fewest instructions per
// proposal once every quarter has a full warp (13 n per step for 32 of them),
// but a batch of a few chains leaves all but a few lanes and quarters idle.
// Small batches therefore spread a proposal over a warp:
//  * IMEX: 16 lanes per field, M = n / 16 nodes each; the constant-coefficient
//    tridiagonal solve is the two first-order recursions of rd_scan.cuh with a
//    prefix scan over the lanes, 10 M + 15 instructions a step (55 at n = 64
//    against 832).  4 proposals of 64 nodes: 28.5 -> 2.9 us a step.
//  * semi-implicit: the elimination is serial and its result reproducible to
//    the bit, so only what is independent moves to other lanes: u and v, the
//    divisions for c' and d' of a node, and the coefficients of all nodes.
//    256 proposals of 100 nodes: 227 -> 60 us a step, up to 94 when blocks with work
//    come to share an SM (nothing keeps two of the first n_sm blocks apart).
// The kernel reads the number of queued proposals and takes the path whose
// instructions per SM quarter are fewer (lanes_for).  The IMEX paths agree to rounding
// only, so RD_SOLVER_THOMAS, whose results do not depend on the batch, always gives a
// proposal one thread.
#include <cuda_runtime.h>
#include <math.h>

#include "rd_common.cuh"
#include "rd_internal.h"

namespace rd {

// ---------------------------------------------------------------------------
// One thread per proposal: Thomas algorithm on the tridiagonal Neumann matrix
// (diagonal alpha + 2 beta, alpha + beta in the two boundary rows,
// off-diagonals -beta).
// ---------------------------------------------------------------------------
// Factors of the Thomas elimination for [alpha I - beta Lap_h]: inverse
// pivots inv[i] and modified super-diagonal cp[i] = -beta inv[i].
template <int NMAX>
__device__ __forceinline__ void thomas_factors(int n, double alpha, double beta,
                                               double (&cp)[NMAX], double (&inv)[NMAX]) {
  double prev = 0.0;
  for (int i = 0; i < n; ++i) {
    const double diag = alpha + ((i == 0 || i == n - 1) ? beta : 2.0 * beta);
    const double den = diag + beta * prev;
    inv[i] = 1.0 / den;
    cp[i] = -beta * inv[i];
    prev = cp[i];
  }
}

// Steady-state mode (pb.ss_tol > 0, fixed domain, Sec. 3.1.2): the step loop
// stops at the first step T whose discrete time derivative has
//   (h^dim sum over both fields ((w^{T} - w^{T-1}) / tau)^2)^(1/2) < ss_tol,
// at most n_steps; the single observation is taken at T.  With ss_confirm the
// solve goes on to 2T and requires (h^dim sum (w(2T) - w(T))^2)^(1/2) < ss_tol;
// the reported state stays w(T).  Either failure is RD_P_NOT_CONVERGED.
// steps_out (may be null) receives T (0 when none was reached).
template <int NMAX>
__device__ void solve1d_item(const DevProblem& pb, const DevSize& S,
                             const double th[kNPhys], double* phi_out,
                             uint32_t* st_out, double* fields_out, int* steps_out) {
  double u[NMAX], v[NMAX], ru[NMAX], rv[NMAX];
  double cu[NMAX], cv[NMAX], iu[NMAX], iv[NMAX];
  double up[NMAX], vp[NMAX];  // steady-state mode: previous step, then w(T)
  const int n = S.n;
  for (int i = 0; i < n; ++i) {
    u[i] = S.u0d[i];
    v[i] = S.v0d[i];
  }
  const double a = th[0], b = th[1], d = th[2], g = th[3], r = th[4];
  const double tau = pb.tau, h2inv = (double)n * n, tg = tau * g;
  const int nfo = (S.field_mask & 1) + ((S.field_mask >> 1) & 1);
  const bool grow = (r != 0.0) || pb.growth == RD_GROWTH_POLY4;
  double phi = 0.0;
  bool bad = false;
  int next_obs = 0;
  double alpha = 1.0, bu = tau * h2inv, bv = tau * d * h2inv;
  thomas_factors<NMAX>(n, alpha, bu, cu, iu);
  thomas_factors<NMAX>(n, alpha, bv, cv, iv);
  const bool steady = pb.ss_tol > 0.0;
  int t_ss = 0, phase = 0;  // steady state: 0 seek T, 1 confirm to 2T
  bool conv = !steady;
  for (int step = 0; steady || step < pb.n_steps; ++step) {
    if (steady) {
      if (phase == 0 && step >= pb.n_steps) break;
      if (phase == 0)
        for (int i = 0; i < n; ++i) {
          up[i] = u[i];
          vp[i] = v[i];
        }
    }
    if (pb.scheme == RD_SCHEME_PICARD) {
      // the paper's semi-implicit step: the reaction linearised with u^n, v^n
      // and implicit, so the diagonal varies by node (Thomas, eliminated in
      // place: cu / cv hold c'_i, ru / rv hold d'_i).  Every operation is an
      // explicitly rounded FP64 one (no fused multiply-add) in a fixed order:
      // on a growing domain at large gamma the pattern reached after millions
      // of steps depends on the rounding of each step, so the step is kept
      // reproducible to the bit.
      double rho, q;  // rho_n and rho'/rho at t_n, FP64
      growth_at_rn(pb, th, __dmul_rn((double)step, tau), rho, q);
      if (!(rho > 0.0)) {
        bad = true;
        break;
      }
      const double al = __dadd_rn(1.0, __dmul_rn(__dmul_rn(tau, 1.0), q));  // m = 1 in 1-D
      const double h = __ddiv_rn(1.0, (double)n), hh = __dmul_rn(h, h);
      const double rr = __dmul_rn(rho, rho);
      const double bu1 = __ddiv_rn(__ddiv_rn(__dmul_rn(tau, 1.0), rr), hh);
      const double bv1 = __ddiv_rn(__ddiv_rn(__dmul_rn(tau, d), rr), hh);
      for (int i = 0; i < n; ++i) {
        const double aui = __dadd_rn(al, __dmul_rn(tg, __dsub_rn(1.0, __dmul_rn(u[i], v[i]))));
        const double avi = __dadd_rn(al, __dmul_rn(__dmul_rn(tg, u[i]), u[i]));
        const double rU = __dadd_rn(u[i], __dmul_rn(tg, a));
        const double rV = __dadd_rn(v[i], __dmul_rn(tg, b));
        const double edge = (i == 0 || i == n - 1) ? 1.0 : 2.0;
        const double du = __dadd_rn(__dadd_rn(aui, __dmul_rn(edge, bu1)),
                                    i > 0 ? __dmul_rn(bu1, cu[i - 1]) : 0.0);
        const double dv = __dadd_rn(__dadd_rn(avi, __dmul_rn(edge, bv1)),
                                    i > 0 ? __dmul_rn(bv1, cv[i - 1]) : 0.0);
        cu[i] = (i < n - 1) ? __ddiv_rn(-bu1, du) : 0.0;
        cv[i] = (i < n - 1) ? __ddiv_rn(-bv1, dv) : 0.0;
        ru[i] = __ddiv_rn(__dadd_rn(rU, i > 0 ? __dmul_rn(bu1, ru[i - 1]) : 0.0), du);
        rv[i] = __ddiv_rn(__dadd_rn(rV, i > 0 ? __dmul_rn(bv1, rv[i - 1]) : 0.0), dv);
      }
      u[n - 1] = ru[n - 1];
      v[n - 1] = rv[n - 1];
      for (int i = n - 2; i >= 0; --i) {
        u[i] = __dsub_rn(ru[i], __dmul_rn(cu[i], u[i + 1]));
        v[i] = __dsub_rn(rv[i], __dmul_rn(cv[i], v[i + 1]));
      }
    } else {
    if (grow) {  // rho_n = rho(t_n): the matrix changes every step
      double rho, q;
      growth_at(pb, th, (double)step * tau, rho, q);
      if (!(rho > 0.0)) {
        bad = true;
        break;
      }
      alpha = 1.0 + tau * 1.0 * q;  // m = 1 in 1-D
      bu = tau / (rho * rho) * h2inv;
      bv = tau * d / (rho * rho) * h2inv;
      thomas_factors<NMAX>(n, alpha, bu, cu, iu);
      thomas_factors<NMAX>(n, alpha, bv, cv, iv);
    }
    // explicit reaction fused with the forward elimination
    double pu = 0.0, pv = 0.0;
    for (int i = 0; i < n; ++i) {
      const double uu = u[i], vv = v[i];
      const double u2v = uu * uu * vv;
      const double rU = uu + tg * (a - uu + u2v);
      const double rV = vv + tg * (b - u2v);
      pu = (rU + bu * pu) * iu[i];
      pv = (rV + bv * pv) * iv[i];
      ru[i] = pu;
      rv[i] = pv;
    }
    u[n - 1] = ru[n - 1];
    v[n - 1] = rv[n - 1];
    for (int i = n - 2; i >= 0; --i) {
      u[i] = ru[i] - cu[i] * u[i + 1];
      v[i] = rv[i] - cv[i] * v[i + 1];
    }
    }
    bool observe = !steady && next_obs < S.n_obs && step + 1 == S.obs_steps[next_obs];
    if (steady) {
      double s2 = 0.0;
      for (int i = 0; i < n; ++i)
        s2 += (u[i] - up[i]) * (u[i] - up[i]) + (v[i] - vp[i]) * (v[i] - vp[i]);
      const double h = 1.0 / n;
      if (phase == 0) {
        if (sqrt(h * s2) / tau < pb.ss_tol) {
          t_ss = step + 1;
          observe = true;
          if (!pb.ss_confirm) {
            conv = true;
          } else {
            phase = 1;
            for (int i = 0; i < n; ++i) {
              up[i] = u[i];
              vp[i] = v[i];
            }
          }
        }
      } else if (step + 1 == 2 * t_ss) {
        conv = sqrt(h * s2) < pb.ss_tol;
        for (int i = 0; i < n; ++i) {
          u[i] = up[i];
          v[i] = vp[i];
        }
      }
    }
    if (observe) {
      const double* yo = S.yd + (size_t)next_obs * nfo * n;
      int fo = 0;
      for (int f = 0; f < 2; ++f) {
        if (!(S.field_mask & (1 << f))) continue;
        const double* w = f ? v : u;
        for (int i = 0; i < n; ++i) {
          if (!isfinite(w[i]) || fabs(w[i]) > pb.w_max) bad = true;
          const double e = yo[(size_t)fo * n + i] - w[i];
          phi += e * e;
        }
        ++fo;
      }
      ++next_obs;
    }
    if (steady && ((phase == 0 && t_ss > 0) || (phase == 1 && step + 1 == 2 * t_ss))) break;
  }
  const uint32_t st = (bad ? (uint32_t)RD_P_NONFINITE : 0u) |
                      (conv ? 0u : (uint32_t)RD_P_NOT_CONVERGED);
  *st_out = st;
  *phi_out = st ? (double)INFINITY : phi * S.inv_two_sigma2;
  if (steps_out) *steps_out = t_ss;
  if (fields_out) {
    for (int i = 0; i < n; ++i) {
      fields_out[i] = u[i];
      fields_out[n + i] = v[i];
    }
  }
}

// ---------------------------------------------------------------------------
// One warp per proposal, IMEX step.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double powi(double x, int k) {
  double r = 1.0;
  for (; k > 0; k >>= 1, x *= x)
    if (k & 1) r *= x;
  return r;
}

// This lane's constants of the recursions (see rd_scan.cuh) for its field's
// lam = alpha, beta; lane s of 16 holds nodes [s M, s M + len).
template <int M>
struct Scan1d {
  double a, sc, g;       // ratio, output scale, 1 / (1 - a^2)
  double pm[4];          // a^(M 2^k)
  double alen, as, ae;   // a^len, a^start, a^(n - end)
  double an, inv;        // a^n, 1 / (1 - a^(2n))

  __device__ void set(double alpha, double beta, int n, int start, int len) {
    const double h = 0.5 * alpha / beta;
    a = 1.0 / (1.0 + (h + sqrt(h * (h + 2.0))));
    const double om = 1.0 - a;
    sc = om * om / alpha;
    g = 1.0 / (om * (1.0 + a));
    pm[0] = powi(a, M);
#pragma unroll
    for (int k = 1; k < 4; ++k) pm[k] = pm[k - 1] * pm[k - 1];
    alen = powi(a, len);
    as = powi(a, start);
    ae = len > 0 ? powi(a, n - start - len) : 0.0;
    an = powi(a, n);
    inv = 1.0 / (1.0 - an * an);
  }
};

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Returns false when a step leaves the scan's range (alpha <= 0).
template <int M>
__device__ bool imex1d_warp(const DevProblem& pb, const DevSize& S, const double th[kNPhys],
                            int lane, double* phi_out, uint32_t* st_out, double* fields_out,
                            int* steps_out) {
  constexpr unsigned kAll = 0xffffffffu;
  const int n = S.n, f = lane >> 4, s = lane & 15;
  const int start = s * M;
  const int len = min(max(n - start, 0), M);
  const int s_last = (n - 1) / M;
  double w[M], wp[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    w[j] = j < len ? (f ? S.v0d : S.u0d)[start + j] : 0.0;
    wp[j] = w[j];
  }
  const double tau = pb.tau, h2inv = (double)n * n, tg = tau * th[3];
  const double kin = f ? th[1] : th[0];
  const double D = f ? th[2] : 1.0;
  const int nfo = (S.field_mask & 1) + ((S.field_mask >> 1) & 1);
  const bool observed = (S.field_mask >> f) & 1;
  const int fo = (f == 1 && (S.field_mask & 1)) ? 1 : 0;
  const bool grow = (th[4] != 0.0) || pb.growth == RD_GROWTH_POLY4;
  const bool steady = pb.ss_tol > 0.0;
  Scan1d<M> k;
  if (!grow) k.set(1.0, tau * D * h2inv, n, start, len);
  double phi = 0.0;
  bool bad = false;
  int next_obs = 0, t_ss = 0, phase = 0;  // steady state: 0 seek T, 1 confirm to 2T
  bool conv = !steady;
  for (int step = 0; steady || step < pb.n_steps; ++step) {
    if (steady && phase == 0) {
      if (step >= pb.n_steps) break;
#pragma unroll
      for (int j = 0; j < M; ++j) wp[j] = w[j];
    }
    if (grow) {  // rho_n = rho(t_n): the matrix changes every step
      double rho, q;
      growth_at(pb, th, (double)step * tau, rho, q);
      if (!(rho > 0.0)) {
        bad = true;
        break;
      }
      const double alpha = 1.0 + tau * q;  // m = 1 in 1-D
      if (!(alpha > 0.0)) return false;
      k.set(alpha, tau * D / (rho * rho) * h2inv, n, start, len);
    }
    // explicit reaction, and the sums of this lane's nodes
    double r[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const double o = __shfl_xor_sync(kAll, w[j], 16);
      const double u = f ? o : w[j], v = f ? w[j] : o;
      const double u2v = u * u * v;
      const double c = kin - u;
      const double t = (f ? kin : c) + (f ? -u2v : u2v);
      r[j] = j < len ? fma(tg, t, w[j]) : 0.0;
    }
    double L = r[M - 1], R = r[0];
#pragma unroll
    for (int j = 1; j < M; ++j) {
      L = fma(k.a, L, r[M - 1 - j]);
      const double R1 = fma(k.a, R, r[j]);
      R = j < len ? R1 : R;
    }
    double pre = R, suf = L;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = 1 << i;
      const double x = __shfl_up_sync(kAll, pre, o, 16);
      const double y = __shfl_down_sync(kAll, suf, o, 16);
      const double p1 = fma(k.pm[i], x, pre), s1 = fma(k.pm[i], y, suf);
      pre = s >= o ? p1 : pre;
      suf = s + o < 16 ? s1 : suf;
    }
    const double Lt = __shfl_sync(kAll, suf, 0, 16);
    double left = __shfl_up_sync(kAll, pre, 1, 16);
    double right = __shfl_down_sync(kAll, suf, 1, 16);
    if (s == 0) left = 0.0;
    if (s == 15) right = 0.0;
    const double Rt = __shfl_sync(kAll, fma(k.alen, left, R), s_last, 16);
    left = fma(k.as, fma(k.an, Rt, Lt) * k.inv, left);
    right = fma(k.ae, fma(k.an, Lt, Rt) * k.inv, right);
    double x = left, f_last = 0.0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      x = fma(k.a, x, r[j]);
      r[j] = x;
      f_last = j == len - 1 ? x : f_last;
    }
    x = fma(k.a, f_last, right) * k.g;  // X just past the lane's last node
#pragma unroll
    for (int j = M - 1; j >= 0; --j) {
      const double x1 = fma(k.a, x, r[j]);
      x = j < len ? x1 : x;
      w[j] = j < len ? x1 * k.sc : 0.0;
    }
    bool observe = !steady && next_obs < S.n_obs && step + 1 == S.obs_steps[next_obs];
    if (steady) {
      double s2 = 0.0;
#pragma unroll
      for (int j = 0; j < M; ++j) s2 += (w[j] - wp[j]) * (w[j] - wp[j]);
      s2 = warp_sum(s2);
      const double h = 1.0 / n;
      if (phase == 0) {
        if (sqrt(h * s2) / tau < pb.ss_tol) {
          t_ss = step + 1;
          observe = true;
          if (!pb.ss_confirm) {
            conv = true;
          } else {
            phase = 1;
#pragma unroll
            for (int j = 0; j < M; ++j) wp[j] = w[j];
          }
        }
      } else if (step + 1 == 2 * t_ss) {
        conv = sqrt(h * s2) < pb.ss_tol;
#pragma unroll
        for (int j = 0; j < M; ++j) w[j] = wp[j];
      }
    }
    if (observe) {
      const double* yo = S.yd + (size_t)next_obs * nfo * n + (size_t)fo * n + start;
      double e2 = 0.0;
      bool out = false;
      if (observed) {
#pragma unroll
        for (int j = 0; j < M; ++j)
          if (j < len) {
            if (!isfinite(w[j]) || fabs(w[j]) > pb.w_max) out = true;
            const double e = yo[j] - w[j];
            e2 += e * e;
          }
      }
      phi += warp_sum(e2);
      bad = bad || __any_sync(kAll, out);
      ++next_obs;
    }
    if (steady && ((phase == 0 && t_ss > 0) || (phase == 1 && step + 1 == 2 * t_ss))) break;
  }
  if (lane == 0) {
    const uint32_t st = (bad ? (uint32_t)RD_P_NONFINITE : 0u) |
                        (conv ? 0u : (uint32_t)RD_P_NOT_CONVERGED);
    *st_out = st;
    *phi_out = st ? (double)INFINITY : phi * S.inv_two_sigma2;
    if (steps_out) *steps_out = t_ss;
  }
  if (fields_out)
#pragma unroll
    for (int j = 0; j < M; ++j)
      if (j < len) fields_out[(size_t)f * n + start + j] = w[j];
  return true;
}

template <int MMAX>
__device__ bool imex1d_any(const DevProblem& pb, const DevSize& S, const double th[kNPhys],
                           int lane, double* phi, uint32_t* st, double* fo, int* so) {
  const int m = (S.n + 15) / 16;
  if (MMAX >= 2 && m <= 2) return imex1d_warp<2>(pb, S, th, lane, phi, st, fo, so);
  if (m <= 4) return imex1d_warp<4>(pb, S, th, lane, phi, st, fo, so);
  if constexpr (MMAX > 4) {
    if (m <= 6) return imex1d_warp<6>(pb, S, th, lane, phi, st, fo, so);
    if (m <= 8) return imex1d_warp<8>(pb, S, th, lane, phi, st, fo, so);
    if (m <= 12) return imex1d_warp<12>(pb, S, th, lane, phi, st, fo, so);
    return imex1d_warp<16>(pb, S, th, lane, phi, st, fo, so);
  }
  return false;
}

// ---------------------------------------------------------------------------
// P lanes per proposal, the semi-implicit step: the operations and their order
// are solve1d_item's, so the result is the same to the bit.  Per proposal in
// shared memory: x_u, x_v (the state), then per field the diagonal, replaced
// by c' as it is eliminated, and the right-hand side, replaced by d'.
// ---------------------------------------------------------------------------
template <int P>
__device__ void picard1d_lanes(const DevProblem& pb, const DevSize& S, const double th[kNPhys],
                               int lane, bool active, double* sm, double* phi_out,
                               uint32_t* st_out, double* fields_out) {
  constexpr unsigned kAll = 0xffffffffu;
  const int n = S.n, q = lane % P;
  const int f = q & 1;               // this lane's field in the elimination
  const bool role_d = (q >> 1) & 1;  // and whether it carries d' or c'
  double* xu = sm;
  double* xv = sm + n;
  double* dg_u = sm + 2 * n;
  double* dg_v = sm + 3 * n;
  double* rh_u = sm + 4 * n;
  double* rh_v = sm + 5 * n;
  double* const x_f = f ? xv : xu;
  double* const dg_f = f ? dg_v : dg_u;
  double* const rh_f = f ? rh_v : rh_u;
  for (int i = q; i < n; i += P) {
    xu[i] = S.u0d[i];
    xv[i] = S.v0d[i];
  }
  __syncwarp();
  const double d = th[2], tau = pb.tau, tg = tau * th[3];
  const double ka = __dmul_rn(tg, th[0]), kb = __dmul_rn(tg, th[1]);
  const double h = __ddiv_rn(1.0, (double)n), hh = __dmul_rn(h, h);
  const int nfo = (S.field_mask & 1) + ((S.field_mask >> 1) & 1);
  double phi = 0.0;
  bool bad = false, stop = !active;  // stop: the growth law left rho > 0
  int next_obs = 0;
  for (int step = 0; step < pb.n_steps; ++step) {
    double rho, gq;  // rho_n and rho'/rho at t_n
    growth_at_rn(pb, th, __dmul_rn((double)step, tau), rho, gq);
    if (!(rho > 0.0)) bad = stop = true;
    if (__all_sync(kAll, stop)) break;
    const double al = __dadd_rn(1.0, __dmul_rn(__dmul_rn(tau, 1.0), gq));  // m = 1 in 1-D
    const double rr = __dmul_rn(rho, rho);
    const double b = __ddiv_rn(__ddiv_rn(__dmul_rn(tau, f ? d : 1.0), rr), hh);
    const double bo = __shfl_xor_sync(kAll, b, 1);
    const double bu = f ? bo : b, bv = f ? b : bo;
    for (int i = q; i < n; i += P) {
      const double u = xu[i], v = xv[i];
      const double aui = __dadd_rn(al, __dmul_rn(tg, __dsub_rn(1.0, __dmul_rn(u, v))));
      const double avi = __dadd_rn(al, __dmul_rn(__dmul_rn(tg, u), u));
      const double edge = (i == 0 || i == n - 1) ? 1.0 : 2.0;
      dg_u[i] = __dadd_rn(aui, __dmul_rn(edge, bu));
      dg_v[i] = __dadd_rn(avi, __dmul_rn(edge, bv));
      rh_u[i] = __dadd_rn(u, ka);
      rh_v[i] = __dadd_rn(v, kb);
    }
    __syncwarp();
    double prev = 0.0, dg = dg_f[0], rh = rh_f[0];
    for (int i = 0; i < n; ++i) {
      const double dg1 = i + 1 < n ? dg_f[i + 1] : 0.0, rh1 = i + 1 < n ? rh_f[i + 1] : 0.0;
      const double t = i > 0 ? __dmul_rn(b, prev) : 0.0;
      const double tc = __shfl_sync(kAll, t, lane & ~2);  // beta c'_{i-1}
      const double den = __dadd_rn(dg, tc);
      const double num_d = __dadd_rn(rh, t);
      prev = __ddiv_rn(role_d ? num_d : -b, den);
      if (q < 4) (role_d ? rh_f : dg_f)[i] = prev;
      dg = dg1;
      rh = rh1;
    }
    __syncwarp();
    double x = rh_f[n - 1];
    if (q < 2 && !stop) x_f[n - 1] = x;
    double c1 = n > 1 ? dg_f[n - 2] : 0.0, d1 = n > 1 ? rh_f[n - 2] : 0.0;
    for (int i = n - 2; i >= 0; --i) {
      const double c0 = i > 0 ? dg_f[i - 1] : 0.0, d0 = i > 0 ? rh_f[i - 1] : 0.0;
      x = __dsub_rn(d1, __dmul_rn(c1, x));
      if (q < 2 && !stop) x_f[i] = x;
      c1 = c0;
      d1 = d0;
    }
    __syncwarp();
    if (!stop && next_obs < S.n_obs && step + 1 == S.obs_steps[next_obs]) {
      const double* yo = S.yd + (size_t)next_obs * nfo * n;
      int fo = 0;
      for (int ff = 0; ff < 2; ++ff) {
        if (!(S.field_mask & (1 << ff))) continue;
        const double* w = ff ? xv : xu;
        for (int i = 0; i < n; ++i) {  // in node order, as one thread does
          if (!isfinite(w[i]) || fabs(w[i]) > pb.w_max) bad = true;
          const double e = yo[(size_t)fo * n + i] - w[i];
          phi += e * e;
        }
        ++fo;
      }
      ++next_obs;
    }
  }
  if (!active) return;
  if (q == 0) {
    *st_out = bad ? (uint32_t)RD_P_NONFINITE : 0u;
    *phi_out = bad ? (double)INFINITY : phi * S.inv_two_sigma2;
  }
  if (fields_out)
    for (int i = q; i < n; i += P) {
      fields_out[i] = xu[i];
      fields_out[n + i] = xv[i];
    }
}

// Proposals queued, over all sizes.
__device__ __forceinline__ int queued(const WorkQueue& q) {
  int t = 0;
  for (int k = 0; k < q.n_sizes; ++k) t += *((volatile int*)&q.counts[q.order[k]]);
  return t;
}

// Pops up to m proposals of one size; returns how many, the first in *first.
__device__ __forceinline__ int queue_pop_group(const WorkQueue& q, int m, int* first, int* size) {
  for (int k = 0; k < q.n_sizes; ++k) {
    const int s = q.order[k];
    const int cnt = *((volatile int*)&q.counts[s]);
    if (*((volatile int*)&q.pops[s]) >= cnt) continue;
    const int i = atomicAdd(&q.pops[s], m);
    if (i >= cnt) continue;
    *first = i;
    *size = s;
    return min(m, cnt - i);
  }
  return 0;
}

// One warp takes 32 / P proposals of one size at a time.
template <int P, int NMAX>
__device__ void warp_loop(const DevProblem& pb, const WorkQueue& q, const double* theta,
                          double* phi, uint32_t* status, double* fields, size_t field_stride,
                          int* steps_out, double* sm) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    int first = 0, s = 0, m = 0;
    if (lane == 0) m = queue_pop_group(q, 32 / P, &first, &s);
    m = __shfl_sync(0xffffffffu, m, 0);
    if (m == 0) return;
    first = __shfl_sync(0xffffffffu, first, 0);
    s = __shfl_sync(0xffffffffu, s, 0);
    const DevSize& S = pb.sz[s];
    const int sub = lane / P;
    const bool active = sub < m;
    const int b = q.items[(size_t)s * q.capacity + first + (active ? sub : 0)];
    double th[kNPhys];
    full_theta(pb, theta + (size_t)b * pb.n_params, th);
    double* fo = fields ? fields + (size_t)b * field_stride : nullptr;
    if (pb.scheme == RD_SCHEME_PICARD) {
      picard1d_lanes<P>(pb, S, th, lane, active, sm + (size_t)sub * 6 * S.n, &phi[b], &status[b],
                        fo);
    } else if constexpr (P == 32) {
      bool reg = th[2] >= 0.0 && 1.0 + pb.tau * th[4] > 0.0;
      for (int j = 0; j < kNPhys; ++j) reg = reg && isfinite(th[j]);
      int* so = steps_out ? &steps_out[b] : nullptr;
      if (!reg || !imex1d_any<(NMAX > 64 ? 16 : 4)>(pb, S, th, lane, &phi[b], &status[b], fo, so))
        if (lane == 0) solve1d_item<NMAX>(pb, S, th, &phi[b], &status[b], fo, so);
    }
    __syncwarp();
  }
}

// FP64 instructions per step of one warp, in units of a plain one (a division
// counts 5): the basis of the choice of path.  n nodes; lanes per proposal P
// (1: a thread each).
__host__ __device__ inline long long warp_cost(int n, bool picard, int P) {
  if (picard) return P == 1 ? 42ll * n : 10ll * n + 11ll * n / P + 40;
  if (P == 1) return 13ll * n;
  const int m = (n + 15) / 16;
  return 10ll * (m <= 2 ? 2 : m <= 4 ? 4 : m <= 6 ? 6 : m <= 8 ? 8 : m <= 12 ? 12 : 16) + 15;
}

// Lanes per proposal for `count` queued proposals on `quarters` SM quarters:
// the least instructions on the busiest quarter.
__host__ __device__ inline int lanes_for(int n, bool picard, int count, int quarters) {
  int best = 1;
  long long best_cost = -1;
  const int options[3] = {1, 8, 32};
  for (int i = 0; i < 3; ++i) {
    const int P = options[i];
    if (P == 8 && !picard) continue;
    const long long warps = ((long long)count * P + 31) / 32;
    const long long cost = (warps + quarters - 1) / quarters * warp_cost(n, picard, P);
    if (best_cost < 0 || cost <= best_cost) {
      best_cost = cost;
      best = P;
    }
  }
  return best;
}

// Shared memory for the semi-implicit step's lanes: 4 warps x (32 / P) proposals.
static size_t picard_smem(int n, int P) { return (size_t)4 * (32 / P) * 6 * n * sizeof(double); }

template <int NMAX>
__global__ void __launch_bounds__(128)
    k_solve1d_f64(const __grid_constant__ DevProblem pb, const __grid_constant__ WorkQueue q,
                  const double* theta, double* phi, uint32_t* status, double* fields,
                  size_t field_stride, int* steps_out, int n_sm, int p_min) {
  extern __shared__ __align__(16) double sm1d[];
  const bool picard = pb.scheme == RD_SCHEME_PICARD;
  int P = lanes_for(pb.max_n, picard, queued(q), 4 * n_sm);
  if (picard ? pb.ss_tol > 0.0 : pb.thomas != 0) P = 1;
  if (P > 1 && P < p_min) P = p_min;
  if (P > 1) {
    // at most one warp per SM quarter on average: more would share its FP64 pipe
    if ((int)blockIdx.x >= n_sm) return;
    double* sm = sm1d + (size_t)(threadIdx.x >> 5) * (32 / P) * 6 * pb.max_n;
    if (P == 8)
      warp_loop<8, NMAX>(pb, q, theta, phi, status, fields, field_stride, steps_out, sm);
    else
      warp_loop<32, NMAX>(pb, q, theta, phi, status, fields, field_stride, steps_out, sm);
    return;
  }
  for (;;) {
    int s;
    const int b = queue_pop(q, &s);
    if (b < 0) break;
    double th[kNPhys];
    full_theta(pb, theta + (size_t)b * pb.n_params, th);
    double* fo = fields ? fields + (size_t)b * field_stride : nullptr;
    solve1d_item<NMAX>(pb, pb.sz[s], th, &phi[b], &status[b], fo,
                       steps_out ? &steps_out[b] : nullptr);
  }
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
static const void* kernel_1d(int max_n) {
  return max_n <= 64 ? (const void*)k_solve1d_f64<64> : (const void*)k_solve1d_f64<256>;
}

// 8 lanes per proposal need 4 x 4 proposals' vectors in shared memory.
static int min_lanes_1d(int max_n) { return picard_smem(max_n, 8) <= 96 * 1024 ? 8 : 32; }

cudaError_t setup_solve_1d(int max_n) {
  return cudaFuncSetAttribute(kernel_1d(max_n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)picard_smem(max_n, min_lanes_1d(max_n)));
}

int grid_solve_1d(int max_n, int n_sm) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_1d(max_n), 128, 0) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  return n_sm * per_sm;
}

cudaError_t launch_solve_1d(const DevProblem& pb, const WorkQueue& q, const double* theta,
                            double* phi, uint32_t* status, void* fields, int grid, cudaStream_t st,
                            int* steps_out) {
  size_t stride = (size_t)2 * pb.max_n;
  DevProblem pbv = pb;
  WorkQueue qv = q;
  int n_sm = 0, dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int p_min = min_lanes_1d(pb.max_n);
  const bool lanes = pb.scheme == RD_SCHEME_PICARD && pb.ss_tol <= 0.0;
  const size_t smem = lanes ? picard_smem(pb.max_n, p_min) : 0;
  void* args[] = {&pbv,    &qv,        (void*)&theta, &phi,  &status,
                  &fields, &stride, &steps_out,    &n_sm, &p_min};
  return cudaLaunchKernel(kernel_1d(pb.max_n), dim3(grid), dim3(128), args, smem, st);
}

}  // namespace rd
