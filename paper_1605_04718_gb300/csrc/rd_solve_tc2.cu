// rd_solve_tc2.cu -- 2-D forward solves on the tensor cores, N = 16..128.
//
// The IMEX step of Sec. 3.1.1 (reaction explicit, diffusion and dilution
// implicit) with fields held as deviations from the initial-state mean.  The
// implicit solve [alpha I - beta Lap_h] w = r takes the cosine basis (DCT-II
// matrix C) in one direction only and solves the tridiagonal systems that are
// left along the other (rd_scan.cuh):
//   stage 1  D[k][i] = sum_j C[k][j] R[i][j]     (tensor cores)
//   scan     X[k][.] = [(alpha + beta mu_k) I - beta Lap_1D]^-1 D[k][.]
//   stage 2  W[j][i] = sum_k C[k][j] X[k][i]     (tensor cores)
// against four transforms when both directions are diagonalised: half the
// tensor-core work, two conversions of the data per step instead of four, and
// no 1 / (alpha + beta (mu_k + mu_l)) per point.  The scan is FP32 throughout.
// Measured against the four-transform kernels (GB300): 128^2 9.98 -> 5.5 us a
// step of one proposal per SM; 64^2 18.7 -> 4.5 us for the four proposals an SM
// holds; relative field error after 1000 steps at 128^2 2.2e-7 -> 1.8e-7.
//
// Layout.  A slab is one accumulator of 128 TMEM lanes x 128 columns; a CTA has
// two.  The constant matrices are operand A, read from TMEM, the data operand B
// in shared memory (FP16 hi and lo parts).
//   N > 64:  slab 0 is field u, slab 1 field v of one proposal.
//   N <= 64: a slab holds floor(128 / N)^2 blocks of N x N: proposals along the
//   lanes (A is block-diagonal) and u | v of more proposals along the columns;
//   the two slabs are independent of each other.  64^2: 2 proposals per slab,
//   32^2: 8, 16^2: 32.  Blocks that a small batch leaves empty cost no K blocks
//   and no columns.
// A step maps a state with y on the lanes to one with x on the lanes, so the
// orientation alternates; the operator is symmetric in x and y.
//
// Warps 0-15 convert (TMEM -> registers -> reaction or scan -> split ->
// shared memory), warp 16 issues every MMA from one thread, warp 17 forms the
// growing domain's factors in FP64 one step ahead.
//   N > 64: one proposal's step is a chain -- reaction, stage 1, scan, stage 2 --
//   so it is overlapped within itself.  u and v run one behind the other on the
//   tensor cores; their scans run side by side, eight warps each (scanning u
//   with all 16 warps and then v measured 7.05 us a step against 6.85: v's
//   operand then comes late for stage 2).  Stage 2 of v is issued as two column
//   halves, so the reaction of the first 64 columns runs under the second half
//   (an N = 64 MMA takes 37 cycles against 64 for N = 128), and stage 1 starts
//   with the correction products of those columns while the others are computed.
//   Measured with both together: 6.65 -> 5.79 us, of which the reaction's
//   arithmetic below is 0.3.
//   N <= 64: all 16 warps take slab 0 and then slab 1, so each slab's MMAs run
//   under the other's conversions (5.1 us a step against 5.46 with eight warps
//   per slab).
// The converters bound the kernel: 8 FP32 operations and two splits per point
// for the reaction, 4 FMAs and a split per value for the scan, on an FP32 pipe
// that takes 1.5 cycles per FMA with three register operands and 2 per FP16 pair
// conversion; the tensor pipe is busy 50 to 60 % of a step, the rest of the chain
// is hand-offs (a commit or an arrival reaches its waiter after 350 to 450
// cycles; spinning waiters were no faster).  The issuing loops are unrolled at
// compile time: forming descriptors at run time cost 100 to 150 cycles an MMA
// against 64.  Branches around the stores, one per 8 values, cost 2 %: they end
// the blocks that the compiler schedules the conversions in.
//
// Precision: every FP32 operand x is split into FP16 hi + lo and each product
// formed as hi*hi + hi*lo + lo*hi, about 22 significant bits.  The tensor core
// rounds each MMA's sum toward zero; each stage issues the small correction
// products first and its output is scaled by 1 + N 2^-29, the mean shrink that
// the N / 16 main products leave.  The data's lo part is stored negated (one
// instruction less per pair) and the MMAs that read it set the negate bit.
// Power-of-two scales keep operands inside the FP16 range:
//   R' = 128 r, C' = 8 C -> D' = 1024 D; X' = 16 x; W' = 128 w.
// The state and R' have the same scale, so the reaction's linear term is the
// state as it is; the growing domain's constant (1 - alpha) w_ref only concerns
// mode k = 0 and is added to the scan's result there, in the same operation as
// the output scale.
//
// N <= 64: the block-diagonal A multiplies other proposals' data by zero, so a
// reaction value outside the FP16 range (a diverging solve) must not reach the
// MMA as infinity (nor reach the scan as one: |r| >= 256): it is stored as zero, and
// every later observation or output of its proposal reads NaN, which is what an
// infinite operand leads to.  With that, |D| <= 256 sqrt(N), and the scan's output
// (at most |D| / alpha and the constant's term) stays inside the range too wherever
// `irregular` lets a proposal share a CTA.
//
// Every wait is bounded; a timed-out wait makes the CTA leave, drain its MMAs,
// free its TMEM and raise the error flag.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "rd_common.cuh"
#include "rd_internal.h"
#include "rd_scan.cuh"
#include "rd_tc_ptx.cuh"

namespace rd {

using namespace tc;

namespace tc2 {

constexpr int kMaxItems = 64;  // proposals per CTA (N = 16)
constexpr uint32_t kColA = 0;  // 8C hi | 8C lo | 8C^T hi | 8C^T lo, 64 columns each
constexpr uint32_t kColAcc = 256;  // + 128 g
constexpr uint32_t kTileBytes = 128 * 128 * 2;  // one FP16 operand tile
constexpr uint32_t kOffCtrl = 4 * kTileBytes;   // after slab 0 hi, lo, slab 1 hi, lo
constexpr int kConvWarps = 16;
constexpr int kIssueWarp = 16;  // 17: growth factors
constexpr int kThreads = 32 * 18;

// How proposals of an N x N grid fill a slab (128 lanes x 128 columns).
template <int N>
struct Geo {
  static constexpr bool kPair = N > 64;            // slab 0 = u, slab 1 = v of one proposal
  static constexpr int LB = kPair ? 1 : 128 / N;   // blocks along the lanes
  static constexpr int S = N * LB;                 // slab edge
  static constexpr int QB = kPair ? 1 : LB / 2;    // (u, v) block pairs along the columns
  static constexpr int kCap = kPair ? 1 : 2 * LB * QB;  // proposals per CTA
  static constexpr int NB = N == 16 ? 2 : 1;       // scan blocks per thread and slab
  static constexpr int kOpWarps = kPair ? 8 : 16;  // warps that scan one slab
};

struct alignas(16) React {  // one proposal's step constants
  float fa, fb, ftg, alpha;  // a, b, 128 tau gamma, 1 + tau m r
  float off[2];              // growing domain: the term (1 - alpha) w_ref of k = 0, per field
};

struct Ctrl {
  uint64_t mma_done[2];    // per slab: a stage's MMAs completed (two phases per step)
  uint64_t half_done;      // N > 64: slab 1's stage 2, first 64 columns
  uint64_t op_ready[2];    // per slab: scanned operand written
  uint64_t rx[2];          // N > 64: first / second half of both slabs' reaction written;
                           // N <= 64: slab 0 / 1's reaction written (16 warps)
  uint64_t seg[2][4][2];   // N >= 48: the sums of (slab, quadrant, block) written (2 warps)
  uint64_t grow;           // growing domain: this step's beta written
  uint64_t fin;
  uint64_t never;          // completed by nothing (failure-path test aid)
  uint32_t tmem_base;
  int abort;
  int n_items;
  int size;
  int slow;               // an irregular proposal, alone in the CTA
  int n_chunk, next;      // popped items, of which already run
  int chunk[kMaxItems];
  int items[kMaxItems];
  int bad[kMaxItems];
  int blown[kMaxItems];   // N <= 64: a reaction value left the FP16 range
  double phi[kMaxItems];
  double th[kMaxItems][kNPhys];
  float beta[2][kMaxItems][2];  // growing domain: per step parity, item, field
  React rk[kMaxItems];
  alignas(16) float mu[128];
  float2 sums[2][4][128];       // (L, R) per slab, block and segment, lane
};
constexpr uint32_t kSmemBytes = 1024 + kOffCtrl + (uint32_t)((sizeof(Ctrl) + 127) / 128 * 128);

// Parities of the barriers' phases at the start of an item: those of the step's
// first slab (each completes once a step), and slab 1's (not in use in every item).
struct Parity {
  uint32_t p0 = 0, p1 = 0, seg = 0;
};

// The 1024-byte aligned start of shared memory, derived from the shared symbol
// so that the compiler keeps the address space (plain shared accesses).
__device__ __forceinline__ uint8_t* shared_base() {
  extern __shared__ uint8_t smem_raw[];
  return smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
}
__device__ __forceinline__ Ctrl* shared_ctl() {
  return reinterpret_cast<Ctrl*>(shared_base() + kOffCtrl);
}

// Shared address of slab g's hi tile (its lo tile follows).
__device__ __forceinline__ uint32_t tile(int g) {
  return smem_u32(shared_base()) + (uint32_t)(2 * g) * kTileBytes;
}

__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                       uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// Byte offset (in 16-byte units) of K block kk of an operand tile with `rows`
// rows: K-major (stage 1) or MN-major (stage 2).
__device__ __forceinline__ constexpr uint32_t kblock_off(int stage, int rows, int kk) {
  return (stage == 1 ? (uint32_t)(kk >> 2) * (uint32_t)rows * 128u + (uint32_t)(kk & 3) * 32u
                     : (uint32_t)kk * 2048u) >> 4;
}

// K blocks [K0, K1) of one stage of slab g: the correction products (lo
// operand parts), the main products, or both.  kb < K1 skips the blocks from kb.
// COL0 (0 or 64, stage 2): the first of the ncols columns.
template <int STAGE, int ROWS, bool CORR, bool MAIN, int K0, int K1, bool FIRST, int COL0 = 0>
__device__ __forceinline__ void issue_blocks(uint32_t sbase, uint32_t tmem, int g, int ncols,
                                             int kb) {
  constexpr int b_mn = STAGE == 2;
  const uint32_t idesc = idesc_f16_f32(128, ncols, 0, b_mn);
  const uint32_t idesc_nb = idesc_f16_f32(128, ncols, 0, b_mn, 1);  // B = the negated lo
  const uint32_t a_hi = tmem + kColA + (STAGE == 1 ? 0u : 128u), a_lo = a_hi + 64u;
  constexpr uint32_t lbo = STAGE == 1 ? 16u : (uint32_t)ROWS * 128u;
  static_assert(COL0 == 0 || (COL0 == 64 && STAGE == 2), "columns start at a 64-column block");
  const uint32_t tb = sbase + (uint32_t)(2 * g) * kTileBytes + (uint32_t)COL0 / 64u * ROWS * 128u;
  const uint64_t bh = sdesc_sw128(tb, lbo, 1024u);
  const uint64_t bl = sdesc_sw128(tb + kTileBytes, lbo, 1024u);
  const uint32_t d = tmem + kColAcc + (uint32_t)(128 * g + COL0);
  if (CORR) {
#pragma unroll
    for (int kk = K0; kk < K1; ++kk) {
      if (kk >= kb) break;
      const uint32_t off = kblock_off(STAGE, ROWS, kk);
      mma_ts(d, a_hi + (uint32_t)(kk * 8), bl + off, idesc_nb, (kk > K0 || !FIRST) ? 1u : 0u);
      mma_ts(d, a_lo + (uint32_t)(kk * 8), bh + off, idesc, 1u);
    }
  }
  if (MAIN) {
#pragma unroll
    for (int kk = K0; kk < K1; ++kk) {
      if (kk >= kb) break;
      mma_ts(d, a_hi + (uint32_t)(kk * 8), bh + kblock_off(STAGE, ROWS, kk), idesc, 1u);
    }
  }
}

// Predicated 16-byte shared store: a branch instead would end the basic block
// that the compiler schedules the conversions in.
__device__ __forceinline__ void st_shared16(uint32_t addr, const uint32_t (&v)[4], bool on) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
      "@p st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(addr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"((uint32_t)on)
      : "memory");
}

// Splits 8 values (x scale + off) of row r, columns c..c+7 into the hi tile and,
// kTileBytes behind it, the negated lo tile: one 16-byte store each.
__device__ __forceinline__ void store8(uint32_t hi, int rows, int r, int c, const float* x,
                                       float scale, float off, bool on) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float y0 = x[2 * j], y1 = x[2 * j + 1];
    fma_pair(y0, y1, scale, off);
    split_f16x2_neglo(y0, y1, h[j], l[j]);
  }
  const uint32_t a = hi + sw128_offset(rows, r, c);
  st_shared16(a, h, on);
  st_shared16(a + kTileBytes, l, on);
}

// As store8 without a scale; returns a word with bit 15 or 31 set where a value
// is 2^15 or larger (or NaN): |r| >= 256.
__device__ __forceinline__ uint32_t store8n(uint32_t hi, int rows, int r, int c, const float* x,
                                            bool on) {
  uint32_t h[4], l[4], e = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    split_f16x2_neglo(x[2 * j], x[2 * j + 1], h[j], l[j]);
    e |= (h[j] & 0x7C007C00u) + 0x08000800u;
  }
  const uint32_t a = hi + sw128_offset(rows, r, c);
  st_shared16(a, h, on);
  st_shared16(a + kTileBytes, l, on);
  return e;
}

// Explicit reaction in place on 8 points, all times 128 (the operand scale is the
// state's, so the linear term is the state itself):
// r_u = du + tau gamma (a - u + u^2 v), r_v = dv + tau gamma (b - u^2 v), as
// deviations from the reference state.
__device__ __forceinline__ void react8(float* u, float* v, float ref_u, float ref_v,
                                       const React& k) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float uu = fmaf(u[j], 0x1p-7f, ref_u), vv = fmaf(v[j], 0x1p-7f, ref_v);
    const float uv = uu * vv;
    u[j] = fmaf(k.ftg, fmaf(uu, uv, k.fa - uu), u[j]);
    v[j] = fmaf(k.ftg, fmaf(-uu, uv, k.fb), v[j]);
  }
}

// Observation misfit and final-field output of this thread's points of one
// slab pair: column indices c0 + 8 step_c j, j < n8, of lane index idx, u at
// TMEM columns t_u + c, v at t_v + c.  sl: the proposal's slot, -1 for idle rows.
__device__ __noinline__ void observe(const DevProblem& pb, int size, int sl, int idx, int c0,
                                     int step_c, int n8, uint32_t t_u, uint32_t t_v,
                                     int step, int obs, float* fields, size_t field_stride) {
  Ctrl* ctl = shared_ctl();
  const DevSize& S = pb.sz[size];
  const int n = S.n;
  const bool odd = step & 1;
  const bool out = step == pb.n_steps && fields && sl >= 0;
  const int nfo = (S.field_mask & 1) + ((S.field_mask >> 1) & 1);
  const float* yo = obs >= 0 ? S.yf + (size_t)obs * nfo * S.npts : nullptr;
  float* fo = out ? fields + (size_t)ctl->items[sl] * field_stride : nullptr;
  const bool blown = sl >= 0 && ctl->blown[sl];
  // NaN where the solve would have reached it
  const float sw = blown ? __int_as_float(0x7fffffff) : 0x1p-7f;
  double phi = 0.0;
  int bad = 0;
  for (int k = 0; k < n8; ++k) {
    const int c = c0 + 8 * step_c * k;
    float u[8], v[8];
    __syncwarp();
    tmem_ld8(t_u + (uint32_t)c, u);
    tmem_ld8(t_v + (uint32_t)c, v);
    tmem_wait_ld();
    if (sl < 0) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const size_t pt = odd ? (size_t)(c + j) * n + idx : (size_t)idx * n + c + j;  // y n + x
      const float du = u[j] * sw, dv = v[j] * sw;
      if (yo) {
        int kf = 0;
        if (S.field_mask & 1) {
          const double w = (double)S.ref_u + (double)du;
          if (!(fabs(w) <= pb.w_max)) bad = 1;
          const double e = (double)yo[pt] - w;
          phi += e * e;
          ++kf;
        }
        if (S.field_mask & 2) {
          const double w = (double)S.ref_v + (double)dv;
          if (!(fabs(w) <= pb.w_max)) bad = 1;
          const double e = (double)yo[(size_t)kf * S.npts + pt] - w;
          phi += e * e;
        }
      }
      if (out) {
        fo[pt] = S.ref_u + du;
        fo[(size_t)S.npts + pt] = S.ref_v + dv;
      }
    }
  }
  if (!yo) return;
  // 16 neighbouring lanes always hold the same proposal
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) phi += __shfl_xor_sync(0xffffffffu, phi, o);
  if (sl >= 0) {
    if ((threadIdx.x & 15) == 0) atomicAdd(&ctl->phi[sl], phi);
    if (bad) atomicOr(&ctl->bad[sl], 1);
  }
}

// A whole row of N nodes by Gaussian elimination (any lam and beta), from the
// accumulator columns at t to the operand row l, columns col0...  For alpha, beta > 0
// the pivots are beta + e_i with e_0 = lam, e_i = lam + e_{i-1} / (1 + e_{i-1} / beta),
// the last one e_{N-1}: sums of positive terms, so that lam is not lost beside a
// large beta (lam + 2 beta + beta c'_{i-1} loses 1.5e-5 of the row at beta / alpha = 1e4
// and the whole row from 1e8 on; this form at most 3e-6 up to 1e25, in float32).
template <int N>
__device__ __noinline__ void slow_row(uint32_t t, int g, int rows, int l, int col0, bool store,
                                      float alpha, float beta, float mu, float out_scale,
                                      float off) {
  float c[N], d[N];  // x_i = d_i + c_i x_{i+1}
  const float lam = fmaf(beta, mu, alpha);
  const bool positive = alpha > 0.f && beta > 0.f;
  float cp = 0.f, dp = 0.f, e = 0.f, s = 0.f;
#pragma unroll 1
  for (int x = 0; x < N; x += 8) {
    float v[8];
    __syncwarp();
    tmem_ld8(t + (uint32_t)x, v);
    tmem_wait_ld();
    for (int j = 0; j < 8; ++j) {
      const int i = x + j;
      if (positive) {
        e = fmaf(e, cp, lam);
        s = fmaf(s, cp, v[j]);
        cp = 1.f / (1.f + e / beta);
        dp = s / (i == N - 1 ? e : e + beta);
      } else {
        const float den = lam + ((i == 0 || i == N - 1) ? beta : 2.f * beta) - beta * cp;
        cp = beta / den;
        dp = (v[j] + beta * dp) / den;
      }
      c[i] = cp;
      d[i] = dp;
    }
  }
  float x1 = 0.f;
#pragma unroll 1
  for (int i = N - 1; i >= 0; --i) {
    x1 = d[i] + (i < N - 1 ? c[i] * x1 : 0.f);
    d[i] = x1;
  }
#pragma unroll 1
  for (int x = 0; x < N; x += 8) store8(tile(g), rows, l, col0 + x, d + x, out_scale, off, store);
}

// Starts the load of H columns: tmem_wait_ld() before they are read.
template <int H>
__device__ __forceinline__ void load_cols(uint32_t t, float (&r)[H]) {
  __syncwarp();
  if constexpr (H % 16 == 0) {
#pragma unroll
    for (int x = 0; x < H; x += 16)
      tmem_ld16(t + (uint32_t)x, *reinterpret_cast<float(*)[16]>(r + x));
  } else {
#pragma unroll
    for (int x = 0; x < H; x += 8)
      tmem_ld8(t + (uint32_t)x, *reinterpret_cast<float(*)[8]>(r + x));
  }
}

// One scan segment r (segment seg of a row) of slab g -> operand row l, columns
// col0...  slot: where the row's sums are exchanged.
template <int N>
__device__ __forceinline__ bool scan_segment(uint64_t wait_ns, float (&r)[ScanSeg<N>::H], int g, int seg,
                                             int slot, int quad, uint32_t parity, int lane,
                                             int col0, bool row_used, const ScanCoef& k,
                                             float off) {
  using SG = ScanSeg<N>;
  constexpr int E = Geo<N>::S, H = SG::H;
  Ctrl* const ctl = shared_ctl();
  const int l = 32 * quad + lane;
  float left, right;
  {
    float2 lr[SG::NS];
    float L, R;
    scan_sums<H>(r, k.a, L, R);
    if constexpr (SG::NS > 1) {
      ctl->sums[g][2 * slot + seg][l] = make_float2(L, R);
      __syncwarp();
      uint64_t* bar = &ctl->seg[g][quad][slot];
      if (lane == 0) mbar_arrive(bar);
      if (!mbar_wait_bounded(bar, parity, &ctl->abort, wait_ns)) return false;
      const float2 other = ctl->sums[g][2 * slot + (seg ^ 1)][l];
      lr[0] = seg ? other : make_float2(L, R);
      lr[1] = seg ? make_float2(L, R) : other;
    } else {
      lr[0] = make_float2(L, R);
    }
    scan_entries<SG::NS>(lr, seg, k, left, right);
  }
  float x = left;
#pragma unroll
  for (int m = 0; m < H; ++m) {
    x = fmaf(k.a, x, r[m]);
    r[m] = x;
  }
  // down: X_{H-1} = (F_{H-1} + a right) / (1 - a^2), X_m = F_m + a X_{m+1}
  x = fmaf(k.a, right, x) * k.g;
  r[H - 1] = x;
#pragma unroll
  for (int m = H - 2; m >= 0; --m) {
    x = fmaf(k.a, x, r[m]);
    r[m] = x;
    if (m % 8 == 0) store8(tile(g), E, l, col0 + m, r + m, k.sc, off, row_used);
  }
  return true;
}

// The 16 converter warps, warp % 4 the TMEM lane quadrant, w4 = warp / 4 along
// the columns.  N > 64: all of them do the reaction, then w4 = 0, 1 scan slab 0
// and 2, 3 slab 1.  N <= 64: all of them do slab 0, then slab 1.
template <int N>
__device__ __forceinline__ void converter(const DevProblem& pb, uint32_t tmem, int warp, int lane,
                                          const Parity& par, float* fields, size_t field_stride) {
  using G = Geo<N>;
  using SG = ScanSeg<N>;
  constexpr int E = G::S;  // slab edge
  Ctrl* const ctl = shared_ctl();
  const int size = ctl->size;
  const DevSize& S = pb.sz[size];
  volatile int* abort = &ctl->abort;
  const uint64_t wait_ns = pb.wait_ns;
  const int n_steps = pb.n_steps;
  const bool growth = pb.growth != 0;
  const int w4 = warp >> 2, quad = warp & 3;
  const int l = 32 * quad + lane;
  const int n_items = ctl->n_items;
  const int slabs = (G::kPair || n_items > G::QB) ? 2 : 1;
  const int p = G::kPair ? 0 : l / N;
  const int idx = l - p * N;  // index along the lanes within the block
  const int pmax = G::kPair ? 1 : (n_items + 2 * G::QB - 1) / (2 * G::QB);
  const bool row_used = N == 128 || (l < E && p < pmax);
  const uint32_t t_acc = tmem + ((uint32_t)(32 * quad) << 16) + kColAcc;
  const float ref_u = S.ref_u, ref_v = S.ref_v;
  const float mu_l = l < E ? ctl->mu[idx] : 0.f;
  // X' = 16 x from D' = 1024 D, with both stages' compensation
  const float kap = (float)N * 0x1p-29f;
  const float out_scale = 0x1p-6f * (1.f + 2.f * kap);
  const bool slow = ctl->slow != 0;
  // the slot of pair q in slab g: -1 for idle rows and blocks
  auto slot = [&](int g, int q) {
    const int s = G::kPair ? 0 : q + G::QB * (g + 2 * p);
    return (row_used && s < n_items) ? s : -1;
  };
  // scan block i of this thread in a slab: its column block 2 q + f
  auto block_of = [&](int i) {
    return G::kPair ? 0 : (N >= 48 ? (w4 >> 1) : (N == 32 ? w4 : 2 * w4 + i));
  };
  constexpr int NG = G::kPair ? 1 : 2;  // slabs scanned by one thread
  const int g0 = G::kPair ? (w4 >> 1) : 0;
  const int seg = N >= 48 ? (w4 & 1) : 0;
  auto alpha_beta = [&](int g, int i, int step, float& alpha, float& beta, float& off) {
    const int s = slot(g, G::kPair ? 0 : block_of(i) >> 1);
    const int f = G::kPair ? g : (block_of(i) & 1);
    alpha = 1.f;
    beta = off = 0.f;
    if (s >= 0) {
      alpha = ctl->rk[s].alpha;
      beta = ctl->beta[growth ? step & 1 : 0][s][f];
      if (idx == 0) off = ctl->rk[s].off[f];
    }
  };
  ScanCoef sc[NG][G::NB];  // recomputed each step on a growing domain
  float off[NG][G::NB];
  auto set_coef = [&](int step) {
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < G::NB; ++i) {
        float alpha, beta;
        alpha_beta(g0 + g, i, step, alpha, beta, off[g][i]);
        sc[g][i] = scan_coef<N>(alpha, beta, mu_l, out_scale);
      }
  };
  if (!growth) set_coef(0);
  int next_obs = 0;
  for (int step = 0;; ++step) {
    const bool last = step == n_steps;
    const uint32_t ph = (uint32_t)step & 1u;
    const int obs = (next_obs < S.n_obs && step == S.obs_steps[next_obs]) ? next_obs++ : -1;
    if (growth && !last) {  // this step's beta is ready (see grower)
      if (!mbar_wait_bounded(&ctl->grow, ph ^ par.p0, abort, wait_ns)) return;
    }
    // ---- observation / output, then the reaction -> stage-1 operands
    if constexpr (G::kPair) {
      // stage 2 of slab 0 (the second commit of a step ends an odd phase) and of
      // slab 1's first 64 columns; the rest of slab 1 runs under the first half's
      // reaction
      if (step > 0) {
        if (!mbar_wait_bounded(&ctl->mma_done[0], 1u, abort, wait_ns)) return;
        if (!mbar_wait_bounded(&ctl->half_done, ph ^ 1u ^ par.p0, abort, wait_ns)) return;
        tc_fence_after();
      }
      if (obs >= 0 || last) {
        if (step > 0) {
          if (!mbar_wait_bounded(&ctl->mma_done[1], 1u, abort, wait_ns)) return;
          tc_fence_after();
        }
        observe(pb, size, slot(0, 0), idx, 8 * w4, 4, (N - 8 * w4 + 31) / 32, t_acc, t_acc + 128u,
                step, obs, fields, field_stride);
      }
      if (last) return;
      const int s = slot(0, 0);
      React k = {0.f, 0.f, 0.f, 1.f, {0.f, 0.f}};
      if (s >= 0) k = ctl->rk[s];
      // 8-column chunks 32 j + 8 w4, j = 0..3, of both fields, in two halves.  The
      // first half's MMAs overwrite the state, so the second is loaded before the
      // first is handed over
      auto chunk_on = [&](int j) {  // compile-time for all but one j
        return 32 * j + 32 <= N || (32 * j < N && 32 * j + 8 * w4 < N);
      };
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        if (hf == 1 && step > 0) {  // the rest of slab 1
          if (!mbar_wait_bounded(&ctl->mma_done[1], 1u, abort, wait_ns)) return;
          tc_fence_after();
        }
        float u[16], v[16];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t c = (uint32_t)(64 * hf + 32 * j + 8 * w4);
          if (chunk_on(2 * hf + j)) {
            tmem_ld8(t_acc + c, *reinterpret_cast<float(*)[8]>(u + 8 * j));
            tmem_ld8(t_acc + 128u + c, *reinterpret_cast<float(*)[8]>(v + 8 * j));
          }
        }
        tmem_wait_ld();
        if (hf == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&ctl->rx[0]);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = 64 * hf + 32 * j + 8 * w4;
          if (chunk_on(2 * hf + j)) {
            react8(u + 8 * j, v + 8 * j, ref_u, ref_v, k);
            store8n(tile(0), E, idx, c, u + 8 * j, row_used);
            store8n(tile(1), E, idx, c, v + 8 * j, row_used);
          }
        }
        fence_proxy_async_smem();
        if (hf == 1) {
          __syncwarp();
          if (lane == 0) mbar_arrive(&ctl->rx[1]);
        }
      }
    } else {
      // 8-column chunks of this warp: N = 64: 2, 48: 2 or 1, 32 and 16: 2 of one pair
      const int q = N >= 48 ? 0 : (N == 32 ? (w4 >> 1) : w4);
      const int c0 = N >= 48 ? 8 * w4 : (N == 32 ? 16 * (w4 & 1) : 0);
      constexpr int CS = N >= 48 ? 32 : 8;  // stride between the chunks
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g >= slabs) break;
        if (step > 0) {
          if (!mbar_wait_bounded(&ctl->mma_done[g], 1u, abort, wait_ns)) return;
          tc_fence_after();
        }
        const uint32_t t_u = t_acc + (uint32_t)(128 * g + 2 * q * N), t_v = t_u + (uint32_t)N;
        const int s = slot(g, q);
        if (obs >= 0 || last)
          observe(pb, size, s, idx, c0, CS / 8, c0 + CS < N ? 2 : 1, t_u, t_v, step, obs,
                  fields, field_stride);
        if (last) continue;
        React k = {0.f, 0.f, 0.f, 1.f, {0.f, 0.f}};
        if (s >= 0) k = ctl->rk[s];
        auto chunk_on = [&](int j) { return N != 48 || j == 0 || c0 + CS < N; };
        float u[16], v[16];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = c0 + CS * j;
          if (chunk_on(j)) {
            tmem_ld8(t_u + (uint32_t)c, *reinterpret_cast<float(*)[8]>(u + 8 * j));
            tmem_ld8(t_v + (uint32_t)c, *reinterpret_cast<float(*)[8]>(v + 8 * j));
          }
        }
        tmem_wait_ld();
        const int row = 2 * q * N + idx;
        uint32_t e = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = c0 + CS * j;
          if (chunk_on(j)) {
            react8(u + 8 * j, v + 8 * j, ref_u, ref_v, k);
            e |= store8n(tile(g), E, row, p * N + c, u + 8 * j, row_used);
            e |= store8n(tile(g), E, row + N, p * N + c, v + 8 * j, row_used);
          }
        }
        if ((e & 0x80008000u) && row_used) {  // rare: see the top of the file
          if (s >= 0) ctl->blown[s] = 1;
          const uint32_t zero[4] = {0u, 0u, 0u, 0u};
          for (int j = 0; j < 2; ++j)
            if (chunk_on(j))
              for (int f = 0; f < 2; ++f) {
                const uint32_t a =
                    tile(g) + sw128_offset(E, row + f * N, p * N + c0 + CS * j);
                st_shared16(a, zero, true);
                st_shared16(a + kTileBytes, zero, true);
              }
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->rx[g]);
      }
      if (last) return;
    }
    // ---- stage 1 done: solve along the columns -> operand of stage 2
    if (growth) set_coef(step);
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
      if (gi >= slabs) break;
      const int g = g0 + gi;
      if (!mbar_wait_bounded(&ctl->mma_done[g], 0u, abort, wait_ns)) return;
      tc_fence_after();
#pragma unroll
      for (int i = 0; i < G::NB; ++i) {
        const int col0 = block_of(i) * N + seg * SG::H;
        const uint32_t t = t_acc + (uint32_t)(128 * g + col0);
        if (slow) {
          if (seg == 0) {
            float alpha, beta, o;
            alpha_beta(g, i, step, alpha, beta, o);
            slow_row<N>(t, g, E, l, col0, row_used, alpha, beta, mu_l, out_scale, o);
          }
        } else {
          float r[SG::H];
          load_cols<SG::H>(t, r);
          tmem_wait_ld();
          if (!scan_segment<N>(wait_ns, r, g, seg, G::kPair ? 0 : block_of(i) & 1, quad,
                               ph ^ (NG == 2 && gi == 1 ? par.seg >> 1 : par.seg & 1u), lane, col0,
                               row_used, sc[gi][i], off[gi][i]))
            return;
        }
      }
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->op_ready[g]);
    }
  }
}

// The MMA-issuing warp.
template <int N>
__device__ __forceinline__ bool issuer(const DevProblem& pb, uint32_t tmem, int lane,
                                       const Parity& par) {
  using G = Geo<N>;
  constexpr int E = G::S, KB = E / 16;
  Ctrl* const ctl = shared_ctl();
  // warp-uniform values, so that the descriptors stay in uniform registers
  const uint32_t sbase = __shfl_sync(0xffffffffu, smem_u32(shared_base()), 0);
  tmem = __shfl_sync(0xffffffffu, tmem, 0);
  volatile int* abort = &ctl->abort;
  const int items = ctl->n_items;
  const int pmax = G::kPair ? 1 : (items + 2 * G::QB - 1) / (2 * G::QB);
  const int kb = G::kPair ? KB : pmax * N / 16;                                // K blocks in use
  const int ncols = G::kPair ? N : 2 * N * (items < G::QB ? items : G::QB);    // columns in use
  const int slabs = (G::kPair || items > G::QB) ? 2 : 1;
  const int n_steps = pb.n_steps;
  const uint64_t wait_ns = pb.wait_ns;
  for (int step = 0; step < n_steps; ++step) {
    const uint32_t ph = (uint32_t)step & 1u;
    if constexpr (G::kPair) {
      // the correction products of the reaction's first half (64 columns)
      // while its second half is computed
      if (!mbar_wait_bounded(&ctl->rx[0], ph ^ par.p0, abort, wait_ns)) return false;
      tc_fence_after();
      if (elect_one()) {
        issue_blocks<1, E, true, false, 0, 4, true>(sbase, tmem, 0, N, KB);
        issue_blocks<1, E, true, false, 0, 2, true>(sbase, tmem, 1, N, KB);
      }
      __syncwarp();
      if (!mbar_wait_bounded(&ctl->rx[1], ph ^ par.p1, abort, wait_ns)) return false;
      tc_fence_after();
      if (elect_one()) {
        issue_blocks<1, E, true, false, 4, KB, false>(sbase, tmem, 0, N, KB);
        issue_blocks<1, E, false, true, 0, KB, false>(sbase, tmem, 0, N, KB);
        mma_commit(&ctl->mma_done[0]);
        issue_blocks<1, E, true, false, 2, KB, false>(sbase, tmem, 1, N, KB);
        issue_blocks<1, E, false, true, 0, KB, false>(sbase, tmem, 1, N, KB);
        mma_commit(&ctl->mma_done[1]);
      }
      __syncwarp();
    } else {
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g >= slabs) break;
        if (!mbar_wait_bounded(&ctl->rx[g], ph ^ (g ? par.p1 : par.p0), abort, wait_ns))
          return false;
        tc_fence_after();
        if (elect_one()) {
          issue_blocks<1, E, true, true, 0, KB, true>(sbase, tmem, g, ncols, kb);
          mma_commit(&ctl->mma_done[g]);
        }
        __syncwarp();
      }
    }
    if (step == pb.stall_step) {  // test aid: wait on a barrier nothing completes
      mbar_wait_bounded(&ctl->never, 0u, abort, wait_ns);
      return false;
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (g >= slabs) break;
      if (!mbar_wait_bounded(&ctl->op_ready[g], ph ^ (g ? par.p1 : par.p0), abort, wait_ns))
        return false;
      tc_fence_after();
      if (elect_one()) {
        if (G::kPair && g == 1) {  // in two column halves, see the converters
          issue_blocks<2, E, true, true, 0, KB, true>(sbase, tmem, g, 64, kb);
          mma_commit(&ctl->half_done);
          issue_blocks<2, E, true, true, 0, KB, true, 64>(sbase, tmem, g, N - 64, kb);
        } else {
          issue_blocks<2, E, true, true, 0, KB, true>(sbase, tmem, g, ncols, kb);
        }
        mma_commit(&ctl->mma_done[g]);
      }
      __syncwarp();
    }
  }
  return true;
}

// Growing domain: one warp forms the steps' beta = tau D / (rho_n^2 h^2) in
// FP64 (rho_n = exp(r n tau)), one step ahead of the converters.
template <int N>
__device__ __noinline__ bool grower(const DevProblem& pb, int lane, Parity par) {
  using G = Geo<N>;
  Ctrl* const ctl = shared_ctl();
  volatile int* abort = &ctl->abort;
  const int items = ctl->n_items;
  const int slabs = (G::kPair || items > G::QB) ? 2 : 1;
  const double tau = pb.tau;
  for (int step = 0; step < pb.n_steps; ++step) {
    // once the reaction of step - 1 is written, every converter has taken the
    // beta of step - 2 (this buffer) and passed its wait for that of step - 1
    for (int g = 0; step >= 1 && g < slabs; ++g)
      if (!mbar_wait_bounded(&ctl->rx[g], ((uint32_t)(step - 1) & 1u) ^ (g ? par.p1 : par.p0),
                             abort, pb.wait_ns))
        return false;
    for (int i = lane; i < items; i += 32) {
      const double rho2inv = exp(-2.0 * ctl->th[i][4] * (double)step * tau);
      ctl->beta[step & 1][i][0] = (float)(tau * rho2inv * (double)N * N);
      ctl->beta[step & 1][i][1] = (float)(tau * ctl->th[i][2] * rho2inv * (double)N * N);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&ctl->grow);
  }
  return true;
}

// Proposals the scan does not cover (negative diffusion, alpha <= 0, a beta / alpha
// above kScanMaxRatio at any step, non-finite parameters): solved alone, by
// elimination.  So are, at N <= 64, those whose scanned values could leave the FP16
// range (|x| <= 256 sqrt(N) / alpha, see the top of the file): as infinities they
// would reach the other proposals of the block-diagonal products.
template <int N>
__device__ __forceinline__ bool irregular(const DevProblem& pb, const DevSize& S,
                                          const double th[kNPhys]) {
  bool fin = true;
  for (int j = 0; j < kNPhys; ++j) fin = fin && isfinite(th[j]);
  if (!fin || !(th[2] >= 0.0)) return true;
  // FP32: the line is far from where either side fails, and an overflow is beyond it
  float alpha = 1.f, top = (float)pb.tau * (float)(N * N) * fmaxf(1.f, (float)th[2]);
  if (pb.growth) {
    const double r2 = 2.0 * pb.tau * th[4], al = 1.0 + r2;
    if (!(al > 0.0)) return true;
    alpha = (float)al;
    if (th[4] < 0.0) top *= expf(-(float)r2 * (float)pb.n_steps);
    const float ref = fmaxf(fabsf(S.ref_u), fabsf(S.ref_v));
    if (N <= 64 &&
        !(16.f * sqrtf((float)N) * (256.f + fabsf((float)r2) * ref) <= 65000.f * alpha))
      return true;
  }
  return !(top <= kScanMaxRatio * alpha);
}

// Pops proposals of one size of the queue: as many as a CTA holds, fewer when
// the batch is too small to fill every CTA that way.  Irregular ones go last.
template <int N>
__device__ __forceinline__ void pop_chunk(const DevProblem& pb, const WorkQueue& q,
                                          const double* theta, Ctrl* ctl) {
  constexpr int cap = Geo<N>::kCap;
  ctl->n_chunk = ctl->next = 0;
  int full = 0;  // CTAs that the whole batch would fill
  for (int k = 0; k < q.n_sizes; ++k)
    full += (*((volatile int*)&q.counts[q.order[k]]) + cap - 1) / cap;
  const int take = full < (int)gridDim.x ? (cap * full + (int)gridDim.x - 1) / (int)gridDim.x : cap;
  for (int k = 0; k < q.n_sizes; ++k) {
    const int s = q.order[k];
    const int cnt = *((volatile int*)&q.counts[s]);
    if (*((volatile int*)&q.pops[s]) >= cnt) continue;
    const int i = atomicAdd(&q.pops[s], take);
    if (i >= cnt) continue;
    const int m = min(take, cnt - i);
    int a = 0, z = m;
    for (int j = 0; j < m; ++j) {
      const int item = q.items[(size_t)s * q.capacity + i + j];
      double th[kNPhys];
      full_theta(pb, theta + (size_t)item * pb.n_params, th);
      if (irregular<N>(pb, pb.sz[s], th))
        ctl->chunk[--z] = item;
      else
        ctl->chunk[a++] = item;
    }
    ctl->n_chunk = m;
    ctl->slow = a;  // regular items at the front
    ctl->size = s;
    return;
  }
}

// The next proposals to solve, into ctl: a chunk's regular ones together, its
// irregular ones one by one (ctl->slow counts the regular ones until then).
template <int N>
__device__ __noinline__ void next_items(const DevProblem& pb, const WorkQueue& q,
                                        const double* theta) {
  Ctrl* const ctl = shared_ctl();
  ctl->n_items = 0;
  if (ctl->abort) return;
  if (ctl->next >= ctl->n_chunk) pop_chunk<N>(pb, q, theta, ctl);
  if (ctl->next >= ctl->n_chunk) return;
  const int reg = ctl->next == 0 ? ctl->slow : 0;
  const int m = reg > 0 ? reg : 1;
  for (int j = 0; j < m; ++j) {
    ctl->items[j] = ctl->chunk[ctl->next + j];
    full_theta(pb, theta + (size_t)ctl->items[j] * pb.n_params, ctl->th[j]);
  }
  ctl->next += m;
  ctl->slow = reg > 0 ? 0 : 1;
  ctl->n_items = m;
}

// Step constants of item j (the growing domain's beta: see grower).
__device__ __forceinline__ void item_constants(const DevProblem& pb, const DevSize& S, Ctrl* ctl,
                                               int j) {
  const double* th = ctl->th[j];
  const double tau = pb.tau;
  React k;
  k.fa = (float)th[0];
  k.fb = (float)th[1];
  k.ftg = (float)(128.0 * tau * th[3]);
  k.off[0] = k.off[1] = 0.f;
  k.alpha = 1.f;
  if (pb.growth) {
    // the constant (1 - alpha) w_ref has the k = 0 coefficient sqrt(N) of it,
    // which the implicit solve divides by alpha; times 16 and stage 2's
    // compensation
    const double al = 1.0 + tau * 2.0 * th[4];
    const double c = 16.0 * sqrt((double)S.n) * (1.0 - al) / al * (1.0 + S.n * 0x1p-29);
    k.alpha = (float)al;
    k.off[0] = (float)(c * (double)S.ref_u);
    k.off[1] = (float)(c * (double)S.ref_v);
  } else {
    ctl->beta[0][j][0] = (float)(tau * (double)S.n * S.n);
    ctl->beta[0][j][1] = (float)(tau * th[2] * (double)S.n * S.n);
  }
  ctl->rk[j] = k;
  ctl->phi[j] = 0.0;
  ctl->bad[j] = ctl->blown[j] = 0;
}

// A size's 8C and 8C^T, block-diagonal over the slab's lane blocks, as split
// FP16 into TMEM (lane = output index): converter warps 0-7 C, 8-15 C^T.
template <int N>
__device__ __noinline__ void fill_constants(const DevSize& S, uint32_t tmem, int warp, int lane) {
  constexpr int n = N, edge = Geo<N>::S;
  Ctrl* const ctl = shared_ctl();
  const bool tr = warp >= 8;
  const int m = 32 * (warp & 3) + lane;
  const int mb = m / n, mi = m - mb * n;
  const uint32_t t = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + kColA + (tr ? 128u : 0u);
  const int cbase = 32 * ((warp >> 2) & 1);
  for (int c0 = cbase; c0 < cbase + 32; c0 += 8) {
    float vh[8], vl[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float e[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int kc = 2 * (c0 + j) + k, kb = kc / n, ki = kc - kb * n;
        e[k] = (m < edge && kc < edge && kb == mb)
                   ? 8.f * (tr ? S.cmat[(size_t)ki * n + mi] : S.cmat[(size_t)mi * n + ki])
                   : 0.f;
      }
      __half h0, l0, h1, l1;
      split_f16(e[0], h0, l0);
      split_f16(e[1], h1, l1);
      vh[j] = __uint_as_float((uint32_t)__half_as_ushort(h0) |
                              ((uint32_t)__half_as_ushort(h1) << 16));
      vl[j] = __uint_as_float((uint32_t)__half_as_ushort(l0) |
                              ((uint32_t)__half_as_ushort(l1) << 16));
    }
    __syncwarp();
    tmem_st8(t + (uint32_t)c0, vh);
    tmem_st8(t + 64u + (uint32_t)c0, vl);
  }
  tmem_wait_st();
  for (int i = 32 * warp + lane; i < n; i += 32 * kConvWarps) ctl->mu[i] = S.mu[i];
}

// Initial deviations (x 128), y on the lanes: four warps per quadrant share the
// 256 accumulator columns.
template <int N>
__device__ __forceinline__ void initial_state(const DevSize& S, uint32_t tmem, int warp,
                                              int lane) {
  using G = Geo<N>;
  const int l = 32 * (warp & 3) + lane;
  const uint32_t t = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + kColAcc;
  const int y = l < G::S ? l % N : 0;
  for (int c8 = 8 * (warp >> 2); c8 < 256; c8 += 32) {
    const int g = c8 >> 7, c = c8 & 127;
    if (c >= G::S) continue;  // warp-uniform
    const int f = G::kPair ? g : ((c / N) & 1);
    const int x = G::kPair ? c : c % N;
    const float ref = f ? S.ref_v : S.ref_u;
    const float* w0 = f ? S.v0f : S.u0f;
    float v8[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v8[j] = (w0[(size_t)y * N + x + j] - ref) * 128.f;
    __syncwarp();
    tmem_st8(t + (uint32_t)c8, v8);
  }
  tmem_wait_st();
}

// The persistent CTA: takes proposals from the queue until it is empty.
template <int N>
__device__ __forceinline__ void solve_loop(const DevProblem& pb, const WorkQueue& q,
                                           const double* theta, double* phi, uint32_t* status,
                                           float* fields, size_t field_stride, int* err) {
  Ctrl* const ctl = shared_ctl();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == kIssueWarp) {
    tmem_alloc(&ctl->tmem_base, 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int g = 0; g < 2; ++g) {
      mbar_init(&ctl->mma_done[g], 1);
      mbar_init(&ctl->op_ready[g], Geo<N>::kOpWarps);
      mbar_init(&ctl->rx[g], kConvWarps);
      for (int i = 0; i < 8; ++i) mbar_init(&ctl->seg[g][i >> 1][i & 1], 2);
    }
    mbar_init(&ctl->half_done, 1);
    mbar_init(&ctl->grow, 1);
    mbar_init(&ctl->fin, 1);
    mbar_init(&ctl->never, 1);
    ctl->abort = 0;
    ctl->n_chunk = ctl->next = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // a batch of several grid sizes is one launch per size: the next one's CTAs may
  // take the SMs that this one does not fill or has left
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem = ctl->tmem_base;
  // every size of this launch is N x N: one DCT matrix serves all
  if (warp < kConvWarps) fill_constants<N>(pb.sz[q.order[0]], tmem, warp, lane);
  Parity par;
  for (;;) {
    if (tid == 0) next_items<N>(pb, q, theta);
    __syncthreads();
    const int n_items = ctl->n_items;
    if (n_items == 0) break;
    const DevSize& S = pb.sz[ctl->size];
    if (tid < n_items) item_constants(pb, S, ctl, tid);
    if (warp < kConvWarps) initial_state<N>(S, tmem, warp, lane);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp < kConvWarps)
      converter<N>(pb, tmem, warp, lane, par, fields, field_stride);
    else if (warp == kIssueWarp)
      issuer<N>(pb, tmem, lane, par);
    else if (pb.growth)
      grower<N>(pb, lane, par);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (pb.n_steps & 1) {
      const bool both = Geo<N>::kPair || n_items > Geo<N>::QB;
      par.p0 ^= 1u;
      if (both) par.p1 ^= 1u;
      if (!ctl->slow) par.seg ^= both ? 3u : 1u;
    }
    if (!ctl->abort && tid < n_items) {
      const int b = ctl->items[tid];
      status[b] = ctl->bad[tid] ? (uint32_t)RD_P_NONFINITE : 0u;
      phi[b] = ctl->bad[tid] ? (double)INFINITY : ctl->phi[tid] * S.inv_two_sigma2;
    }
    __syncthreads();
  }
  if (warp == kIssueWarp) {
    // by the lane that issued the MMAs: a commit covers its own thread's alone
    if (elect_one()) mma_commit(&ctl->fin);
    __syncwarp();
    volatile int never = 0;
    mbar_wait_bounded(&ctl->fin, 0, &never);
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && ctl->abort) atomicOr(err, 1);
  // ... and this launch ends no sooner than the one before it
  if (blockIdx.x == 0 && tid == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace tc2

template <int N>
__global__ void __launch_bounds__(tc2::kThreads, 1)
    k_solve2d_tc(const __grid_constant__ DevProblem pb, const __grid_constant__ WorkQueue q,
                 const double* theta, double* phi, uint32_t* status, float* fields,
                 size_t field_stride, int* err) {
  tc2::solve_loop<N>(pb, q, theta, phi, status, fields, field_stride, err);
}

// 128 x 128: SLABS accumulator slabs, one per field.
template <int SLABS>
__global__ void __launch_bounds__(tc2::kThreads, 1)
    k_solve2d_tc128(const __grid_constant__ DevProblem pb, const __grid_constant__ WorkQueue q,
                    const double* theta, double* phi, uint32_t* status, float* fields,
                    size_t field_stride, int* err) {
  static_assert(SLABS == 2, "the barriers and TMEM columns are laid out for two slabs");
  tc2::solve_loop<128>(pb, q, theta, phi, status, fields, field_stride, err);
}

static const void* tc_kernel(int n) {
  switch (n) {
    case 16: return (const void*)k_solve2d_tc<16>;
    case 32: return (const void*)k_solve2d_tc<32>;
    case 48: return (const void*)k_solve2d_tc<48>;
    case 80: return (const void*)k_solve2d_tc<80>;
    case 96: return (const void*)k_solve2d_tc<96>;
    case 112: return (const void*)k_solve2d_tc<112>;
    case 64: return (const void*)k_solve2d_tc<64>;
    default: return (const void*)k_solve2d_tc128<2>;
  }
}

cudaError_t setup_solve_tc(int n) {
  return cudaFuncSetAttribute(tc_kernel(n), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)tc2::kSmemBytes);
}

int grid_solve_tc(int n_sm) { return n_sm; }

cudaError_t launch_solve_tc(const DevProblem& pb, const WorkQueue& q, const double* theta,
                            double* phi, uint32_t* status, void* fields, int grid, int* err,
                            cudaStream_t st, bool after_tc) {
  size_t stride = (size_t)2 * pb.max_n * pb.max_n;
  DevProblem pbv = pb;
  WorkQueue qv = q;
  float* fo = (float*)fields;
  void* args[] = {&pbv, &qv, (void*)&theta, &phi, &status, &fo, &stride, &err};
  // A launch that follows another size's only needs what both read (the queue and
  // the parameters, written before the first of them) and may start early: 512
  // proposals of each of 64^2, 96^2 and 128^2, 400 steps, 18.26 -> 16.04 ms; 12
  // of each, 300 steps, take 1.82 ms, no longer than the 12 of 128^2 alone.
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(tc2::kThreads);
  cfg.dynamicSmemBytes = tc2::kSmemBytes;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = after_tc ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, tc_kernel(pb.sz[q.order[0]].n), args);
}

}  // namespace rd
