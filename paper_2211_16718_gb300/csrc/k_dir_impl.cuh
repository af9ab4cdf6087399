// Fused per-direction pass of the right-hand side (arXiv 2211.16718, Sec. 2.2):
// for every grid line along direction D, component-wise WENO5 reconstruction of
// u and f_D (left- and right-biased, Jiang-Shu weights), Roe flux with Harten's
// entropy fix at every interface, conservative difference of the interface
// fluxes, 4th-order central divergence of the viscous flux along D, and the
// accumulation / Runge-Kutta stage epilogue.
//
// One CTA owns a tile of TP points along D times W lines (periodic halo of 3
// points each side, fetched with wrapped indices).  Everything is staged in
// shared memory and computed in five phases separated by barriers:
//   A  load state, primitives, viscous flux; point fluxes f_D        [NP x W]
//   B  smoothness indicators of every 3-point window for the 9
//      reconstructed scalars (u_0..u_4, f_1..f_4)                      [9 x NW x W]
//   C  left/right WENO5 reconstructions of the 9 scalars at every
//      interface (MODE 1: as their double-float sum and jump)          [9 x NI x W]
//   D  Roe flux at every interface                                     [NI x W]
//   E  flux difference + viscous divergence + epilogue, global writes  [TP x W]
// The mass flux f_0 = (rho u_D) is the momentum component u_{1+D} itself, so its
// reconstructions are those of u_{1+D}.
//
// With b_k = 4(eps + beta_k) and B_k = b_k^2, the weights are
// omega_k = (c_k/B_k) / sum_j (c_j/B_j) = c_k prod_{m!=k} B_m / sum_j c_j prod_{m!=j} B_m.
// The three squared indicators of a window serve the left-biased reconstruction
// at one interface and the right-biased one at another, so each is computed once.
//
// Since sum omega = 1, fhat = F_2 + omega_1 (F_1 - F_2) + omega_3 (F_3 - F_2): the reconstructions
// are candidate 2 and an offset, F_1 - F_2 and F_3 - F_2 being third differences of the data.
// MODE 0 (all FP64): bound by the FP64 pipe (2 lanes per SM and clock), so written for its operation
// count: with D = B_2/6 the offset is D [B_3 (F_1 - F_2) + 3 B_1 (F_3 - F_2)] / [D B_3 + B_1 (B_3 + 3 D)],
// six operations and a reciprocal; jump and sum of the two reconstructions share their linear parts.
// 496 FP64 operations per point and pass with the halo's share (459 without) where candidates, IEEE
// divisions and separate left and right values took 726: 96^3 pass 1.26 / 1.31 / 1.35 -> 0.91 / 0.92 / 0.95 ms (x / y / z, FP64 pipe 87 %
// busy), the error of a right-hand side against 64 bits 13-19 % smaller.
// MODE 1 (FP64 values, double-float weights): the weights, which only multiply these small
// differences, are evaluated in double-float arithmetic (~48 bits) on the FP32
// pipe.  The reconstructed values themselves are never formed: the Roe flux needs
// fhat_L + fhat_R and the jump fhat_R - fhat_L, whose linear parts combine (phase C),
// both kept in double-float, so the FP64 pipe sees only the first differences, the
// point sums and one combination per flux component.  The result agrees with the all-FP64 evaluation to rounding.
// Phases A2, B and C of MODE 1 take two lines of the tile per item and run their
// double-float arithmetic on both at once with the packed FP32 instructions
// (df2.cuh): each lane computes what a one-line evaluation would, with half the
// issued instructions.
#include <math.h>

#include <type_traits>

#pragma once

#include "df.cuh"
#include "df2.cuh"
#include "k_dir_common.cuh"
#include "k_point_impl.cuh"
#include "ns3d_internal.cuh"

namespace ns3d {

constexpr int NQ = 9;             // reconstructed scalars

// Tile plan of a direction pass: TP points along the pencil times W lines.
// Shared memory in 8-byte words (doubles, or double-float pairs in MODE 1):
//   MODE 0: Q [NQ][NP*W] point values, ROE [5][NP*W] sqrt(rho), u, v, w, H,
//           FV [4][NP*W] viscous flux, B [NQ][4][NW*W] per window B_1, B_2/6, B_3 and a third
//           of its third difference (later the epilogue operands), R [10][NI*W]: jumps of u_0..u_4
//           (slots 0-4) and sums of the flux components (slots 5-9), later [5][NI*W] interface fluxes.
//           73.9 KB for 32 x 4: three CTAs of 256 threads share an SM.
//   MODE 1: Q [NQ][NP*W], dead after phase A2: ROE [5][NR*W] then arrives there by cp.async (as
//           FP64) while phases B and C run, and phase C puts T [5][NI*W] behind it, the double-float
//           part of fhat_L + fhat_R of the five flux scalars;
//           B [NQ][3][NW*W/2] squared indicators, dead after phase C: the epilogue operands and
//           FV [4][NV*W] then arrive there; S [NQ][NW*W/2] third differences;
//           G [NQ][NG*W/2] first differences (B, S, G: double-float values of the two
//           lines of a line pair side by side, 16 bytes (hi0, hi1, lo0, lo1), indexed
//           like the lines with W/2 line pairs); R [10][NI*W]: jumps du of u_0..u_4
//           (double-float, slots 0-4) and the left point values of the five flux scalars
//           (FP64, slots 5-9), later [5][NI*W] interface fluxes.
//   The MODE 1 plan of a 24 x 4 tile is 57.2 KB, so that four CTAs of 256 threads
//   (64 registers) share an SM.  MODE 1 tiles have an even number of lines.
template <int MODE, int TP_, int W_>
struct Plan {
  static constexpr int TP = TP_;                    // points per tile along the pencil
  static constexpr int W = W_;                      // lines per tile
  static constexpr int THREADS = 256;  // 8 warps share the tile (latency hiding)
  static constexpr int MIN_CTAS = (MODE == 0) ? 3 : 4;     // resident CTAs per SM the registers allow
  static constexpr int NP = TP + 6;                 // points incl. 3-point halo each side
  static constexpr int NW = TP + 4;                 // 3-point windows centred at -2 .. TP+1
  static constexpr int NI = TP + 1;                 // interfaces -1/2 .. TP-1/2
  static constexpr int NG = NP - 1;                 // first differences
  static constexpr int NR = (MODE == 1) ? TP + 2 : NP;  // Roe-average inputs: the interfaces' own points
  static constexpr int NV = (MODE == 1) ? TP + 4 : NP;  // viscous flux: 2-point halo
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_ROE = (MODE == 1) ? OFF_Q : OFF_Q + NQ * NP * W;
  static constexpr int OFF_T = OFF_ROE + 5 * NR * W;    // MODE 1
  static constexpr int END_T = OFF_T + 5 * NI * W;
  static constexpr int OFF_B = (MODE == 0)          ? OFF_ROE + (5 + 4) * NP * W
                               : (END_T > NQ * NP * W) ? (END_T + 1) / 2 * 2
                                                       : OFF_Q + NQ * NP * W;
  static constexpr int OFF_FV = (MODE == 1) ? OFF_B + 20 * TP * W : OFF_ROE + 5 * NP * W;
  static constexpr int OFF_S = OFF_B + NQ * (MODE == 0 ? 4 : 3) * NW * W;  // MODE 1: third differences
  static constexpr int OFF_G = OFF_S + (MODE == 1 ? NQ * NW * W : 0);
  static constexpr int OFF_R = OFF_G + (MODE == 1 ? NQ * NG * W : 0);
  static constexpr int R_SLOTS = 10;
  static constexpr int WORDS = OFF_R + R_SLOTS * NI * W;
  static constexpr int BYTES = WORDS * 8;
  static_assert(MODE == 0 || OFF_FV + 4 * NV * W <= OFF_S, "epilogue operands and FV fit the dead indicators");
  // the threads that fetch the epilogue operands (MODE 1: and FV) while the others run phase D
  static constexpr int FETCH0 = THREADS / 2;
  static_assert(MODE == 0 || (NI * W <= FETCH0 && NV * W <= THREADS - FETCH0), "phase D and the fetches side by side");
};

// Index of conserved component c among the reconstructed scalars.  MODE 0 keeps
// the order u_0..u_4, f_1..f_4.  MODE 1 stores the normal momentum u_{1+D} fifth,
// (u_0, u_{1+T1}, u_{1+T2}, u_4, u_{1+D}, f_1..f_4), so that scalars 0-4 are the
// conserved variables and scalars 4-8 the five flux components (f_0 = u_{1+D}).
template <int MODE, int D>
__host__ __device__ constexpr int scalar_of(int c) {
  if (MODE == 0 || c == 0) return c;
  constexpr int T1 = (D == 0) ? 1 : 0, T2 = (D == 2) ? 1 : 2;
  return (c == 1 + D) ? 4 : (c == 1 + T1) ? 1 : (c == 1 + T2) ? 2 : 3;
}

// FP64 reciprocal and reciprocal square root: the special-function unit's approximation (PTX
// rcp / rsqrt.approx.ftz.f64) and one third-order Householder correction, that is the series of 1/x in
// e = 1 - x r (r + r e + r e^2) or of x^(-1/2) in e = 1 - x r^2 (r + r e/2 + 3 r e^2/8) cut before e^3.
// Three and five FP64 operations.  The first rounds once at full size (error below 0.6 ulp), the second
// also in x r (below 1.1 ulp).  What the approximations flush or overflow on (rcp: magnitudes outside
// [2^-1021, 2^1020); rsqrt: subnormals), zeros and non-finite values take the IEEE operations.
__device__ __forceinline__ double rcp_cubic(double x) {
  const uint32_t e11 = ((uint32_t)__double2hiint(x) >> 20) & 0x7ffu;
  if (e11 - 2u >= 2041u) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double rsqrt_cubic(double x) {
  const uint32_t e11 = ((uint32_t)__double2hiint(x) >> 20) & 0x7ffu;
  if (e11 - 1u >= 2046u) return 1.0 / sqrt(x);
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

// Range of the scaled indicators b_k inside which df2_offset3 needs no rescaling of the B_k = b_k^2:
// products of two B_k stay below 2^80, so that they times a third difference (below 2^12 for such
// tiles, since |third difference| <= 4 |first differences| <= 4 b^(1/2)) stay inside the float
// range; and above 2^-100, so that their TwoProd error terms stay normal floats and the products
// keep full precision.  b_k >= 4 eps, so the lower end is a condition on eps alone (with a margin
// for the rounding of b_k).
constexpr float DFB_LO = 0x1.01p-25f, DFB_HI = 0x1p20f;

// 1/6 as a double-float.
__device__ __forceinline__ df2 df2_sixth() {
  constexpr float hi = (float)(1.0 / 6.0), lo = (float)(1.0 / 6.0 - (double)hi);
  return df2_splat(df{hi, lo});
}

// The cut of df2_offset3 for rescaled B_k: 2 at most (lo drops out with hi).
__device__ __forceinline__ df2 df2_cut2(df2 x) {
  const bool c0 = !(x.hi.x < 2.0f), c1 = !(x.hi.y < 2.0f);
  return df2{make_float2(c0 ? 2.0f : x.hi.x, c1 ? 2.0f : x.hi.y), make_float2(c0 ? 0.0f : x.lo.x, c1 ? 0.0f : x.lo.y)};
}

// Offset omega_1 (F_1 - F_2) + omega_3 (F_3 - F_2) of one reconstruction from its candidate 2, in
// double-float, from the three squared scaled indicators B_k (candidate order 1, 2, 3) and the third
// differences ta = 3 (F_1 - F_2), tb = 6 (F_3 - F_2), both given divided by 6; with
// omega_k = c_k prod_{m!=k} B_m / den and den = B2 B3 + 6 B1 B3 + 3 B1 B2,
//   d = B2 [2 B3 ta/6 + 3 B1 tb/6] / [B2 B3 + 3 B1 (2 B3 + B2)]        (one division).
// SCALE: rescale the B_k by a common power of two first (the weights are scale-free), the largest
// to [1, 2); without it every B_k must lie in [DFB_LO^2, DFB_HI^2).  den is at least the product of
// the two largest B_k.  Next to constant data two of them are (4 eps)^2 and the third goes with the
// fourth power of the jump, so a B_k more than 2^96 above the smallest is cut to that ratio: den then
// stays above 2^-96, with its error terms normal floats.  The weight of such a window is below 2^-95
// either way, far under the rounding of the largest difference.
// The numerator and denominator are renormalised and the division's seed refined (8 of the 71 packed
// operations): at a jump the offsets are a third of it, and their rounding is what is left of the
// reconstruction's error there.  In units of 2^-48 of the largest difference, against long double:
// a jump of 0.9 in noise of 0.01 1.7 (1.5 for the form over the common denominator that includes the
// linear part, 3.8 without these), random differences 1.0 (4.5), smooth data below 0.1 (5.6).
// Evaluated for two lines at once (two-lane double-float; each lane exactly as the
// one-lane evaluation, its scale chosen from its own B_k).
template <bool SCALE = true>
__device__ __forceinline__ df2 df2_offset3(df2 B1, df2 B2, df2 B3, df2 ta6, df2 tb6) {
  if (SCALE) {
    const int x1 = exponent_of(B1.hi.x), x2 = exponent_of(B2.hi.x), x3 = exponent_of(B3.hi.x);
    const int y1 = exponent_of(B1.hi.y), y2 = exponent_of(B2.hi.y), y3 = exponent_of(B3.hi.y);
    int E0 = max(x1, max(x2, x3)), E1 = max(y1, max(y2, y3));
    const int cut0 = min(x1, min(x2, x3)) + 96, cut1 = min(y1, min(y2, y3)) + 96;
    const bool wide = E0 > cut0 || E1 > cut1;
    E0 = min(E0, cut0);
    E1 = min(E1, cut1);
    const float2 sc = make_float2(pow2f(-E0), pow2f(-E1));
    B1 = df2_scale(B1, sc);
    B2 = df2_scale(B2, sc);
    B3 = df2_scale(B3, sc);
    if (wide) {
      B1 = df2_cut2(B1);
      B2 = df2_cut2(B2);
      B3 = df2_cut2(B3);
    }
  }
  const df2 b1 = df2_mul_f_u(B1, 3.0f), b3 = df2_twice(B3);
  const df2 den = df2_add_pos_u(df2_mul_u(B2, B3), df2_mul_u(b1, df2_add_pos_u(b3, B2)));
  const df2 num = df2_mul(B2, df2_add_fast(df2_mul_u(b3, ta6), df2_mul_u(b1, tb6)));
  return df2_div_ru(num, fast_two_sum2(den.hi, den.lo));
}

// One tile of the direction-D pass, executed by the whole CTA on the shared memory sm (PL::BYTES):
// the points [s0, s0 + len) along D (len <= TP), line group ty, tile row bz.  Used by the standalone
// kernels (one tile per CTA), the batched kernels and the persistent ensemble kernel (many tiles per
// CTA, with a barrier between tiles).  NC selects read-only-cache loads, valid only when the inputs
// are not written during the kernel (false in the persistent kernel).
// The phases loop over the extents of this tile, not the plan's: a 32-point line as 24 + 8 with all
// 24 computed in the second tile did the work of 48 points, balanced and trimmed 16 + 16 that of 32.
template <int D, int MODE, int TP_, int W_, bool NC = true>
__device__ __forceinline__ void dir_tile(const DirArgs& a, double* sm, int s0, int len, int ty, int bz) {
  using PL = Plan<MODE, TP_, W_>;
  constexpr int TP = PL::TP, NP = PL::NP, NW = PL::NW, NI = PL::NI, W = PL::W;
  constexpr int W2 = (W + 1) / 2;  // line pairs (MODE 1)
  static_assert(MODE == 0 || W % 2 == 0, "MODE 1 tiles pair their lines");
  static_assert(NP < 64, "extents fit c_rcp20");
  const int np = len + 6, nw = len + 4, ni = len + 1;  // this tile's points with halo, windows, interfaces
  const int nD = a.g.n[D];
  constexpr int AX = (D == 0) ? 1 : 0;   // axis of the W lines
  constexpr int BX = (D == 2) ? 1 : 2;   // axis of blockIdx.z
  const int na = a.g.n[AX];
  const int nx = a.g.n[0], ny = a.g.n[1];
  const long long N = a.g.N;
  const int a0 = ty * W;
  const int tid = threadIdx.x;
  auto wrap = [&](int c) { return (c < 0 || c >= nD) ? wrap_idx(c, nD) : c; };

  auto flat = [&](int c, int la) -> long long {
    int idx[3];
    idx[D] = c;
    idx[AX] = la;
    idx[BX] = bz;
    return ((long long)idx[2] * ny + idx[1]) * nx + idx[0];
  };

  // ---- A: load --------------------------------------------------------------
  for (int item = tid; item < np * W; item += PL::THREADS) {
    int pos, line;
    item_split<D, W>(item, np, c_rcp20.v[np], pos, line);
    const int c = wrap(s0 - 3 + pos);
    const int la = min(a0 + line, na - 1);
    const long long p = flat(c, la);
    double U[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) U[v] = ldx<NC>(a.u + v * N + p);
    const double vx = ldx<NC>(a.pm + PM_U * N + p), vy = ldx<NC>(a.pm + PM_V * N + p), vz = ldx<NC>(a.pm + PM_W * N + p);
    const double pr = ldx<NC>(a.pm + PM_P * N + p);
    const double un = (D == 0) ? vx : (D == 1) ? vy : vz;
    const int s = tile_idx<D, W>(pos, line, NP);
    double* q = sm + PL::OFF_Q;
#pragma unroll
    for (int v = 0; v < 5; ++v) q[scalar_of<MODE, D>(v) * NP * W + s] = U[v];
    q[5 * NP * W + s] = (D == 0) ? fma(U[1], un, pr) : U[1] * un;
    q[6 * NP * W + s] = (D == 1) ? fma(U[2], un, pr) : U[2] * un;
    q[7 * NP * W + s] = (D == 2) ? fma(U[3], un, pr) : U[3] * un;
    q[8 * NP * W + s] = (U[4] + pr) * un;
    if (MODE == 0) {  // MODE 1 fetches these after phase A2 (cp.async into the dead point values)
      double* r = sm + PL::OFF_ROE;
      r[0 * NP * W + s] = ldx<NC>(a.pm + PM_SR * N + p);
      r[1 * NP * W + s] = vx;
      r[2 * NP * W + s] = vy;
      r[3 * NP * W + s] = vz;
      r[4 * NP * W + s] = ldx<NC>(a.pm + PM_H * N + p);
      if (a.fv != nullptr) {
        double* f = sm + PL::OFF_FV;
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) f[cc * NP * W + s] = ldx<NC>(a.fv + (long long)(a.fv_dstride * D + cc) * N + p);
      }
    }
  }
  __syncthreads();

  // ---- A2 (MODE 1): first differences g_j = q_{j+1} - q_j in FP64, kept as double-float,
  //      and the point values q_j of the five flux scalars copied to interface j - 2
  constexpr int NR = PL::NR, NV = PL::NV;
  const int nr = len + 2;                       // points 2 .. np - 3: both sides of every interface
  const int pf = tid - (PL::THREADS - nr * W);  // prefetched point of this thread (MODE 1; none if negative)
  static_assert(MODE == 0 || NP * W <= PL::THREADS, "one prefetched point per thread");
  if constexpr (MODE == 1) {
    constexpr int NG = PL::NG;
    const double* q = sm + PL::OFF_Q;
    float4* G = reinterpret_cast<float4*>(sm + PL::OFF_G);
    double* R = sm + PL::OFF_R;
    // one item per line pair (lines 2 lp, 2 lp + 1), stored as (hi0, hi1, lo0, lo1)
    const int ng = len + 5;
    const unsigned rcp_ng = c_rcp20.v[ng];
    for (int item = tid; item < NQ * ng * W2; item += PL::THREADS) {
      int m, j, lp;
      item_split<D, W2>(item, ng, rcp_ng, m, j, lp);
      const double* qm = q + m * NP * W;
      const int l0 = 2 * lp, l1 = l0 + 1;
      const double qa0 = qm[tile_idx<D, W>(j, l0, NP)], qb0 = qm[tile_idx<D, W>(j + 1, l0, NP)];
      const double qa1 = qm[tile_idx<D, W>(j, l1, NP)], qb1 = qm[tile_idx<D, W>(j + 1, l1, NP)];
      const df g0 = d2df_bits(qb0 - qa0), g1 = d2df_bits(qb1 - qa1);
      G[m * NG * W2 + tile_idx<D, W2>(j, lp, NG)] = make_float4(g0.hi, g1.hi, g0.lo, g1.lo);
      if (m >= 4 && j >= 2 && j < ni + 2) {
        R[(1 + m) * NI * W + tile_idx<D, W>(j - 2, l0, NI)] = qa0;
        R[(1 + m) * NI * W + tile_idx<D, W>(j - 2, l1, NI)] = qa1;
      }
    }
    __syncthreads();
    // the point values are dead: fetch the Roe-average inputs into their space while phases B
    // and C run.  One point per thread, on the last nr*W threads (those with the fewest phase-C
    // items), which also convert their Roe inputs to double-float in place before the barrier
    // that ends phase C.
    if (pf >= 0) {
      int pos, line;
      item_split<D, W>(pf, nr, c_rcp20.v[nr], pos, line);
      const long long p = flat(wrap(s0 - 1 + pos), min(a0 + line, na - 1));
      double* r = sm + PL::OFF_ROE + tile_idx<D, W>(pos, line, NR);
      cp_async8(r + 0 * NR * W, a.pm + PM_SR * N + p);
      cp_async8(r + 1 * NR * W, a.pm + PM_U * N + p);
      cp_async8(r + 2 * NR * W, a.pm + PM_V * N + p);
      cp_async8(r + 3 * NR * W, a.pm + PM_W * N + p);
      cp_async8(r + 4 * NR * W, a.pm + PM_H * N + p);
    }
    cp_async_commit();
  }

  // ---- B: squared scaled smoothness indicators of every window ----------------
  int need_scale = 0;
  if constexpr (MODE == 0) {
    // one item per line and four adjacent windows, which share differences
    const double* q = sm + PL::OFF_Q;
    const int nw4 = (nw + 3) / 4;
    const unsigned rcp_nw4 = c_rcp20.v[nw4];
    for (int item = tid; item < NQ * nw4 * W; item += PL::THREADS) {
      int m, w4, line;
      item_split<D, W>(item, nw4, rcp_nw4, m, w4, line);
      const double* qm = q + m * NP * W;
      double* bw = sm + PL::OFF_B + m * 4 * NW * W;
      auto ldq = [&](int j) { return qm[tile_idx<D, W>(min(j, np - 1), line, NP)]; };
      double q1 = ldq(4 * w4 + 1), q2 = ldq(4 * w4 + 2);
      double gm = q1 - ldq(4 * w4), gp = q2 - q1, s0 = gp - gm;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int w = 4 * w4 + k;
        if (w >= nw) break;
        const int o = tile_idx<D, W>(w, line, NW);
        // the third difference of the last window needs a point beyond the tile and is never read
        const double q3 = ldq(w + 3), gn = q3 - q2, s1 = gn - gp;
        bw[3 * NW * W + o] = (1.0 / 3.0) * (s0 - s1);
        const double aa = fma((13.0 / 3.0) * s0, s0, a.eps4);
        const double u1 = fma(3.0, gp, -gm);   // x - 4y + 3z
        const double u2 = gm + gp;             // z - x
        const double u3 = fma(-3.0, gm, gp);   // 3x - 4y + z
        const double b1 = fma(u1, u1, aa), b2 = fma(u2, u2, aa), b3 = fma(u3, u3, aa);
        bw[0 * NW * W + o] = b1 * b1;
        bw[1 * NW * W + o] = b2 * ((1.0 / 6.0) * b2);
        bw[2 * NW * W + o] = b3 * b3;
        q2 = q3;
        gm = gp;
        gp = gn;
        s0 = s1;
      }
    }
  } else {
    // one item per line pair and two adjacent windows: two-lane double-float arithmetic (packed FP32
    // instructions); the windows share a second difference, and a 24-point tile has 252 items for
    // its 256 threads
    int range_bad = 0;
    need_scale = !(a.eps4_hi >= DFB_LO);
    float4* bw = reinterpret_cast<float4*>(sm + PL::OFF_B);
    float4* S = reinterpret_cast<float4*>(sm + PL::OFF_S);
    const df2 c133 = df2_splat(df{a.c133_hi, a.c133_lo});
    const df2 eps4 = df2_splat(df{a.eps4_hi, a.eps4_lo});
    const int nw2 = (nw + 1) / 2;
    const unsigned rcp_nw2 = c_rcp20.v[nw2];
    for (int item = tid; item < NQ * nw2 * W2; item += PL::THREADS) {
      int m, w2, lp;
      item_split<D, W2>(item, nw2, rcp_nw2, m, w2, lp);
      const float4* G = reinterpret_cast<const float4*>(sm + PL::OFF_G) + m * PL::NG * W2;
      auto ldG = [&](int j) { return df2_from4(G[tile_idx<D, W2>(j, lp, PL::NG)]); };
      df2 g0 = ldG(2 * w2), g1 = ldG(2 * w2 + 1);
      df2 s0 = df2_add_fast(g1, df2_neg(g0));  // second difference of the window
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int w = 2 * w2 + k;
        if (w >= nw) break;
        const int o = tile_idx<D, W2>(w, lp, NW);
        // third difference T_w = s_w - s_{w+1}, divided by 6 (phase C needs T_f, T_{f+1}, T_{f+2}; the
        // last window has no s_{w+1} in the tile and its T is never read)
        const df2 g2 = ldG(min(w + 2, len + 4));
        const df2 s1 = df2_add_fast(g2, df2_neg(g1));
        S[m * NW * W2 + o] = df2_to4(df2_mul_u(df2_add_fast(s0, df2_neg(s1)), df2_sixth()));
        // scaled indicators b_k = u_k^2 + aa, aa = (13/3) s^2 + 4 eps, with u_2 = z - x and
        // u_1 = x - 4y + 3z = u_2 + 2s, u_3 = 3x - 4y + z = 2s - u_2:
        //   b_2 = u_2^2 + aa,  b_{1,3} = (b_2 + 4 s^2) +- 4 u_2 s   (b_k >= aa >= (13/3) s^2, so
        // b_2 + 4 s^2 <= ~3 b_{1,3}: no harmful cancellation)
        const df2 s2 = df2_sqr_u(s0);
        const df2 aa = df2_add_pos_u(df2_mul_u(s2, c133), eps4);
        const df2 u2 = df2_add_fast(g0, g1);
        const df2 b2 = df2_add_pos_u(df2_sqr_u(u2), aa);
        // Fast2Sum order with margins: b_2 >= aa >= (13/12) 4 s^2, and
        // pq = u_2^2 + (4 + 13/3) s^2 + 4 eps >= 1.44 |4 u_2 s| (minimum over u_2)
        const float2 four = f2splat(4.0f);
        const df2 pq = df2_add_ordered_u(b2, df2_scale(s2, four));
        const df2 r4 = df2_scale(df2_mul_u(u2, s0), four);
        const df2 B1 = df2_sqr_u(df2_add_ordered(pq, r4));
        const df2 B2 = df2_sqr_u(b2);
        const df2 B3 = df2_sqr_u(df2_add_ordered(pq, df2_neg(r4)));
        bw[(m * 3 + 0) * NW * W2 + o] = df2_to4(B1);
        bw[(m * 3 + 1) * NW * W2 + o] = df2_to4(B2);
        bw[(m * 3 + 2) * NW * W2 + o] = df2_to4(B3);
        // every b_k of both lanes is at most the sum of the lanes' pq + |r4|.  The float exponent
        // range bounds the indicators (differences of the data up to ~1e9); beyond it the host
        // reports NS3D_ERANGE instead of a NaN
        if (!((pq.hi.x + fabsf(r4.hi.x)) + (pq.hi.y + fabsf(r4.hi.y)) < DFB_HI)) {
          need_scale = 1;
          range_bad |= !(fmaxf(B1.hi.x, fmaxf(B2.hi.x, B3.hi.x)) < 1e36f) ||
                       !(fmaxf(B1.hi.y, fmaxf(B2.hi.y, B3.hi.y)) < 1e36f);
        }
        g0 = g1;
        g1 = g2;
        s0 = s1;
      }
    }
    if (__any_sync(0xffffffffu, range_bad) && (tid & 31) == 0) atomicOr(a.status, ST_DF_RANGE);
  }
  // one CTA-wide decision: rescaled weights only for tiles with extreme indicators
  const bool tile_scale = __syncthreads_or(need_scale) != 0;

  // ---- C: left/right WENO5 reconstructions at every interface -------------------
  if constexpr (MODE == 0) {
    // F_1 - F_2 = T_f/3, 3 (F_3 - F_2) = T_{f+1}/2 (left), the mirror image with -T (right); as in
    // MODE 1 the jump is T_{f+1}/6 + oR - oL, the sum [7 (P2 + P3) - (P1 + P4)]/6 + oL + oR
    const double* q = sm + PL::OFF_Q;
    double* rec = sm + PL::OFF_R;
    const unsigned rcp_ni = c_rcp20.v[ni];
    for (int item = tid; item < NQ * ni * W; item += PL::THREADS) {
      int m, f, line;
      item_split<D, W>(item, ni, rcp_ni, m, f, line);
      const double* b = sm + PL::OFF_B + m * 4 * NW * W;
      auto ld = [&](int k, int w) { return b[k * NW * W + tile_idx<D, W>(w, line, NW)]; };
      const double Tc = ld(3, f + 1), T2 = 1.5 * Tc;
      auto offset = [&](double B1, double D2, double B3, double T3, double& num, double& r) {
        num = D2 * fma(B3, T3, B1 * T2);
        r = rcp_cubic(fma(B1, fma(3.0, D2, B3), D2 * B3));
      };
      double nL, rL, nR, rR;  // oL = nL rL, oR = -nR rR
      offset(ld(0, f), ld(1, f + 1), ld(2, f + 2), ld(3, f), nL, rL);
      offset(ld(2, f + 3), ld(1, f + 2), ld(0, f + 1), ld(3, f + 2), nR, rR);
      const int o = tile_idx<D, W>(f, line, NI);
      if (m < 5) rec[m * NI * W + o] = fma(-nR, rR, fma(-nL, rL, 0.5 * Tc));
      if (m >= 5 || m == 1 + D) {  // f_0 = u_{1+D}
        const double* qm = q + m * NP * W;
        const double P1 = qm[tile_idx<D, W>(f + 1, line, NP)], P2 = qm[tile_idx<D, W>(f + 2, line, NP)];
        const double P3 = qm[tile_idx<D, W>(f + 3, line, NP)], P4 = qm[tile_idx<D, W>(f + 4, line, NP)];
        const double lin = fma(7.0 / 6.0, P2 + P3, (-1.0 / 6.0) * (P1 + P4));
        rec[(m < 5 ? 5 : m + 1) * NI * W + o] = fma(-nR, rR, fma(nL, rL, lin));
      }
    }
  } else {
    // fhat_L = P2 + (2 g2 + g1)/6 + oL, fhat_R = P3 - (2 g2 + g3)/6 - oR: candidate 2 and the
    // nonlinear offsets of df2_offset3 (oR with its sign reversed, so that both use +T), from the
    // third differences T_f, T_{f+1}, T_{f+2} of phase B.  Evaluated in double-float on the FP32
    // pipe.  The interface values are never formed in FP64, and the linear parts combine:
    //   fhat_R - fhat_L = T_{f+1}/6 - (oL + oR)                          (u-scalars; double-float)
    //   fhat_L + fhat_R = 2 P2 + [g2 + (g1 - g3)/6 + (oL - oR)]          (flux scalars; the bracket
    //                                                                    in double-float)
    // One item per line pair, in two-lane double-float arithmetic.
    float2* rf = reinterpret_cast<float2*>(sm + PL::OFF_R);
    auto phase_c = [&](auto scaled) {
      constexpr bool SCALE = decltype(scaled)::value;
      const unsigned rcp_ni = c_rcp20.v[ni];
      for (int item = tid; item < NQ * ni * W2; item += PL::THREADS) {
        int m, f, lp;
        item_split<D, W2>(item, ni, rcp_ni, m, f, lp);
        const float4* S = reinterpret_cast<const float4*>(sm + PL::OFF_S) + m * NW * W2;
        const float4* G = reinterpret_cast<const float4*>(sm + PL::OFF_G) + m * PL::NG * W2;
        const float4* b = reinterpret_cast<const float4*>(sm + PL::OFF_B) + m * 3 * NW * W2;
        auto ldS = [&](int w) { return df2_from4(S[tile_idx<D, W2>(w, lp, NW)]); };
        auto ldG = [&](int j) { return df2_from4(G[tile_idx<D, W2>(j, lp, PL::NG)]); };
        auto ld = [&](int k, int w) { return df2_from4(b[k * NW * W2 + tile_idx<D, W2>(w, lp, NW)]); };
        const df2 T1 = ldS(f + 1);
        const df2 oL = df2_offset3<SCALE>(ld(0, f), ld(1, f + 1), ld(2, f + 2), ldS(f), T1);
        const df2 oR = df2_offset3<SCALE>(ld(2, f + 3), ld(1, f + 2), ld(0, f + 1), ldS(f + 2), T1);
        const int o0 = tile_idx<D, W>(f, 2 * lp, NI), o1 = tile_idx<D, W>(f, 2 * lp + 1, NI);
        if (m < 5) {
          const df2 du = df2_add_fast(T1, df2_neg(df2_add_fast(oL, oR)));
          rf[m * NI * W + o0] = make_float2(du.hi.x, du.lo.x);
          rf[m * NI * W + o1] = make_float2(du.hi.y, du.lo.y);
        }
        if (m >= 4) {  // flux scalar; P2 copied in phase A2
          const df2 lin = df2_add_fast(ldG(f + 2), df2_mul_u(df2_add_fast(ldG(f + 1), df2_neg(ldG(f + 3))), df2_sixth()));
          const df2 t = df2_add_fast(lin, df2_add_fast(oL, df2_neg(oR)));
          float2* F = reinterpret_cast<float2*>(sm + PL::OFF_T) + (m - 4) * NI * W;
          F[o0] = make_float2(t.hi.x, t.lo.x);
          F[o1] = make_float2(t.hi.y, t.lo.y);
        }
      }
    };
    if (tile_scale)
      phase_c(std::true_type{});
    else
      phase_c(std::false_type{});
    cp_async_wait_all();  // this thread's ROE copies; the barrier publishes them
    if (pf >= 0) {  // velocities to double-float, in place (sqrt(rho) and H arrive as
                       // double-float: planes of the NS3D_FP64 primitive layout)
      int pos, line;
      item_split<D, W>(pf, nr, c_rcp20.v[nr], pos, line);
      double* r = sm + PL::OFF_ROE + tile_idx<D, W>(pos, line, NR);
#pragma unroll
      for (int k = 1; k < 4; ++k) {
        const df x = d2df_bits(r[k * NR * W]);
        reinterpret_cast<float2*>(r)[k * NR * W] = make_float2(x.hi, x.lo);
      }
    }
  }
  __syncthreads();

  // ---- epilogue operands, and in MODE 1 the viscous flux: fetched asynchronously into the (now
  //      unused) indicator space while phase D runs, by the threads that have no interface.
  //      cp.async.ca reads through L1 like a plain load, so in the persistent kernel (NC
  //      false), where the operands were written by other CTAs before the last grid-wide
  //      barrier, it sees them exactly as the plain loads it replaces would.
  static_assert(PL::TP * PL::W <= PL::THREADS, "one epilogue point per thread");
  static_assert(20 * PL::TP * PL::W <= NQ * 3 * PL::NW * PL::W, "prefetch slots fit the indicator space");
  //      The z pass with nx even takes two x-adjacent points (lines 2j, 2j + 1 of the tile: their flat
  //      index is even) per 16-byte copy, past L1: half the copies.  U_n and the stage input may be
  //      the caller's and only 8-byte aligned; the rest is the library's.  z pass with the RK4
  //      epilogue at 128^3: 502 -> 471 us (16-byte copies through L1: 505).  Not so the y pass, which
  //      has 9 operands instead of up to 19 (415 -> 425 us), nor the Roe inputs above (phase A has
  //      just read three of their five planes through L1).
  const bool pair16 = D == 2 && W % 2 == 0 && (na & 1) == 0 && (((uintptr_t)a.un | (uintptr_t)a.u) & 15) == 0;
  constexpr int TS = TP * W;
  double* pre = sm + PL::OFF_B;  // [20][TP*W]
  const int ft = tid - PL::FETCH0;
  auto fetch_epilogue = [&](auto pair) {
    constexpr bool PAIR = decltype(pair)::value;
    constexpr int S = PAIR ? 2 : 1;
    if (ft < len * (W / S)) {
      int pp, l;
      item_split<D, W / S>(ft, len, c_rcp20.v[len], pp, l);
      if (a0 + S * l < na) epilogue_prefetch<PAIR, TS>(a, flat(s0 + pp, a0 + S * l), pre + S * ft);
    }
    if (MODE == 1 && a.fv != nullptr && ft < nw * (W / S)) {  // points 1 .. np - 2
      int pos, l;
      item_split<D, W / S>(ft, nw, c_rcp20.v[nw], pos, l);
      const long long p = flat(wrap(s0 - 2 + pos), min(a0 + S * l, na - S));
      double* f = sm + PL::OFF_FV + tile_idx<D, W>(pos, S * l, NV);
#pragma unroll
      for (int cc = 0; cc < 4; ++cc)
        cp_async_d<PAIR>(f + cc * NV * W, a.fv + (long long)(a.fv_dstride * D + cc) * N + p);
    }
  };
  if (ft >= 0) {
    if (D == 2 && pair16) fetch_epilogue(std::bool_constant<D == 2>{});
    else fetch_epilogue(std::false_type{});
  }
  cp_async_commit();

  // ---- D: Roe flux at every interface -------------------------------------------
  {
    const double gm1 = a.gamma - 1.0;
    const double* r = sm + PL::OFF_ROE;
    double* rec = sm + PL::OFF_R;
    int bad = 0, range_bad = 0;
    for (int item = tid; item < ni * W; item += PL::THREADS) {
      int f, line;
      item_split<D, W>(item, ni, c_rcp20.v[ni], f, line);
      const int o = tile_idx<D, W>(f, line, NI);
      const int ia = (MODE == 1) ? f : f + 2;  // the interface's left point among the Roe inputs
      const int sa = tile_idx<D, W>(ia, line, NR), sb = tile_idx<D, W>(ia + 1, line, NR);
      if (MODE == 1) {
        // Roe dissipation X|Lambda|X^{-1} du in double-float from the double-float jumps
        // du of phase C and the double-float Roe-average inputs; twice the flux is 2 P2 + (t - diss),
        // t the double-float part of fhat_L + fhat_R = 2 P2 + t: two FP64 operations per component.
        // Phase E divides the difference by 2 dx in FP64.  Formed in double-float here, (t - diss)/(2 dx)
        // rounded at 2^-48 of a jump: mean error of 48 shock-tube right-hand sides 1.311e-14, now
        // 1.288e-14 (1.296e-14 with the sums in FP64), for one FP64 operation more per point (128^3
        // step 5.73 -> 5.77 ms)
        const float2* rf = reinterpret_cast<const float2*>(r);
        auto ldr = [&](int k, int sp) { const float2 v = rf[k * NR * W + sp]; return df{v.x, v.y}; };
        const float2* rj = reinterpret_cast<const float2*>(rec);
        df du[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const float2 j = rj[scalar_of<MODE, D>(v) * NI * W + o];
          du[v] = df{j.x, j.y};
        }
        // what comes in twos runs on the two lanes of the packed operations: the states (a, b), the
        // tangential directions, the acoustic fields, (V_D, H), flux components 0 and 1 + D.  The phase
        // has one item per interface on half of the warps, so its length counts: 128^3 passes
        // 397 / 415 / 471 -> 393 / 412 / 459 us (x / y / z)
        constexpr int T1 = (D == 0) ? 1 : 0;
        constexpr int T2 = (D == 2) ? 1 : 2;
        const df2 gm1d = df2_splat(df{a.gm1_hi, a.gm1_lo});
        auto l0 = [](df2 x) { return df2_lane0(x); };
        auto l1 = [](df2 x) { return df2_lane1(x); };
        auto ab = [&](int k) { return df2_pack(ldr(k, sa), ldr(k, sb)); };
        const df2 r2 = ab(0);
        const df rsum = df_add_pos(l0(r2), l1(r2));
        const df rs = df_div_r(df{1.0f, 0.0f}, rsum);  // refined, as 1/c and c below: at jumps their errors lead
        const df2 w = df2_mul_u(r2, df2_splat(rs));
        const df2 xt1 = df2_mul_u(w, ab(1 + T1)), xt2 = df2_mul_u(w, ab(1 + T2));
        const df2 vt = df2_add_fast(df2_pack(l0(xt1), l0(xt2)), df2_pack(l1(xt1), l1(xt2)));  // (V_T1, V_T2)
        const df2 xn = df2_mul_u(w, ab(1 + D)), xh = df2_mul_u(w, ab(4));
        const df2 uH = df2_add_fast(df2_pack(l0(xn), l0(xh)), df2_pack(l1(xn), l1(xh)));  // (V_D, H)
        const df un = l0(uH);
        const df2 vq = df2_sqr_u(vt);
        const df q2 = df_add_pos_u(df_sqr_u(un), df_add_pos_u(l0(vq), l1(vq)));
        const df q2h = df{0.5f * q2.hi, 0.5f * q2.lo};
        const df c2 = df_mul(df_add_fast(l1(uH), df_neg(q2h)), l0(gm1d));
        bad |= !(c2.hi > 0.0f);
        range_bad |= !(c2.hi > 1e-30f && c2.hi < 1e30f && rsum.hi > 1e-30f && rsum.hi < 1e30f);
        const df c = df_sqrt_r(c2);
        const df rc = df_div_r(df{1.0f, 0.0f}, c);
        const df2 dut = df2_pack(du[1 + T1], du[1 + T2]);
        const df2 vd = df2_mul_u(vt, dut);
        const df2 ud = df2_mul_u(df2_pack(un, q2h), df2_pack(du[1 + D], du[0]));
        const df vdm = df_add_fast(l0(ud), df_add_fast(l0(vd), l1(vd)));
        const df phi = df_mul_u(df_mul_u(l0(gm1d), df_sqr_u(rc)), df_add_fast(df_add_fast(l1(ud), du[4]), df_neg(vdm)));
        const df a2 = df_add_fast(du[0], df_neg(phi));
        const df2 a34 = df2_add_fast(dut, df2_neg(df2_mul_u(vt, df2_splat(du[0]))));
        const df ach = df_mul_u(df_add_fast(df_mul_u(un, du[0]), df_neg(du[1 + D])), rc);
        // (a1, a5) = (phi +- ach)/2
        const df2 a15 = df2_scale(df2_add_fast(df2_splat(phi), df2_pack(ach, df_neg(ach))), f2splat(0.5f));
        const df2 lam = df2_add_fast(df2_splat(un), df2_pack(df_neg(c), c));
        df h1 = df_abs(l0(lam)), h5 = df_abs(l1(lam));
        const df h2 = df_abs(un);
        const df delta = df_mul(c, df{a.hd_hi, a.hd_lo});
        if (df_lt(h1, delta)) h1 = df_div(df_add_pos_u(df_sqr_u(h1), df_sqr_u(delta)), df_twice(delta));
        if (df_lt(h5, delta)) h5 = df_div(df_add_pos_u(df_sqr_u(h5), df_sqr_u(delta)), df_twice(delta));
        const df2 A15 = df2_mul_u(df2_pack(h1, h5), a15), A34 = df2_mul_u(df2_splat(h2), a34);
        const df A2 = df_mul_u(h2, a2);
        const df S = df_add_fast(l0(A15), l1(A15));
        const df d0 = df_add_fast(S, A2);
        const df cD = df_mul_u(c, df_add_fast(l1(A15), df_neg(l0(A15))));
        const df2 dT = df2_add_fast(df2_mul_u(df2_splat(d0), vt), A34);
        const df dn = df_add_fast(df_mul_u(d0, un), cD);
        const df2 e1 = df2_mul_u(df2_pack(S, cD), df2_pack(l1(uH), un));
        const df2 e2 = df2_mul_u(A34, vt);
        const df de = df_add_fast(df_add_fast(l0(e1), l1(e1)),
                                  df_add_fast(df_mul_u(A2, q2h), df_add_fast(l0(e2), l1(e2))));
        const float2* ts = reinterpret_cast<const float2*>(sm + PL::OFF_T);
        auto ldt = [&](int v) { const float2 tv = ts[v * NI * W + o]; return df{tv.x, tv.y}; };
        auto put = [&](int v, df t) {  // flux component 0 is u_{1+D}
          rec[v * NI * W + o] = fma(2.0, rec[(5 + v) * NI * W + o], f2d_bits(t.hi)) + f2d_bits(t.lo);
        };
        const df2 f0n = df2_add_fast(df2_pack(ldt(0), ldt(1 + D)), df2_neg(df2_pack(d0, dn)));
        put(0, l0(f0n));
        put(1 + D, l1(f0n));
        const df2 fT = df2_add_fast(df2_pack(ldt(1 + T1), ldt(1 + T2)), df2_neg(dT));
        put(1 + T1, l0(fT));
        put(1 + T2, l1(fT));
        put(4, df_add_fast(ldt(4), df_neg(de)));
        continue;
      }
      double du[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) du[v] = rec[v * NI * W + o];
      const double ra = r[sa], rb = r[sb];
      const double rs = rcp_cubic(ra + rb);
      const double wa = ra * rs, wb = rb * rs;
      double V[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) V[m] = fma(wa, r[(1 + m) * NP * W + sa], wb * r[(1 + m) * NP * W + sb]);
      const double H = fma(wa, r[4 * NP * W + sa], wb * r[4 * NP * W + sb]);
      const double q2h = 0.5 * fma(V[0], V[0], fma(V[1], V[1], V[2] * V[2]));
      const double c2 = gm1 * (H - q2h);
      bad |= !(c2 > 0.0);
      const double rc = rsqrt_cubic(c2), c = c2 * rc;
      constexpr int T1 = (D == 0) ? 1 : 0;
      constexpr int T2 = (D == 2) ? 1 : 2;
      const double un = V[D], vt1 = V[T1], vt2 = V[T2];
      const double b1 = gm1 * (rc * rc);
      const double vdm = fma(V[0], du[1], fma(V[1], du[2], V[2] * du[3]));
      const double phi = b1 * (fma(q2h, du[0], du[4]) - vdm);
      const double a2 = du[0] - phi;
      const double a3 = fma(-vt1, du[0], du[1 + T1]);
      const double a4 = fma(-vt2, du[0], du[1 + T2]);
      const double ach = 0.5 * (fma(un, du[0], -du[1 + D]) * rc);
      const double ph = 0.5 * phi;
      const double a1 = ph + ach, a5 = ph - ach;
      double l1 = fabs(un - c), l5 = fabs(un + c);
      const double l2 = fabs(un);
      const double delta = a.hdelta * c;
      if (l1 < delta) l1 = (l1 * l1 + delta * delta) / (2.0 * delta);
      if (l5 < delta) l5 = (l5 * l5 + delta * delta) / (2.0 * delta);
      const double A1 = l1 * a1, A2 = l2 * a2, A3 = l2 * a3, A4 = l2 * a4, A5 = l5 * a5;
      const double S = A1 + A5;
      const double d0 = S + A2;
      const double cD = c * (A5 - A1);
      double diss[5];
      diss[0] = d0;
      diss[1 + D] = fma(d0, un, cD);
      diss[1 + T1] = fma(d0, vt1, A3);
      diss[1 + T2] = fma(d0, vt2, A4);
      diss[4] = fma(S, H, fma(cD, un, fma(A2, q2h, fma(A3, vt1, A4 * vt2))));
#pragma unroll
      for (int v = 0; v < 5; ++v) rec[v * NI * W + o] = a.g.hrh[D] * (rec[(5 + v) * NI * W + o] - diss[v]);  // / dx
    }
    if (__any_sync(0xffffffffu, bad) && (tid & 31) == 0) atomicOr(a.status, ST_NONPHYS);
    if (MODE == 1 && __any_sync(0xffffffffu, range_bad) && (tid & 31) == 0) atomicOr(a.status, ST_DF_RANGE);
  }
  cp_async_wait_all();
  __syncthreads();

  // ---- E: conservative difference + viscous divergence + epilogue ----------------
  {
    const double r12 = a.g.r12h[D];
    const double* F = sm + PL::OFF_R;
    const double* fvs = sm + PL::OFF_FV;
    for (int item = tid; item < len * W; item += PL::THREADS) {
      int pp, line;
      item_split<D, W>(item, len, c_rcp20.v[len], pp, line);
      if (a0 + line >= na) continue;
      double cv[5];
      const int op = tile_idx<D, W>(pp + 1, line, NI), om = tile_idx<D, W>(pp, line, NI);
      if (MODE == 1) {  // twice the interface fluxes; viscous fluxes double-float
        const double hr = a.g.hrh[D];
#pragma unroll
        for (int v = 0; v < 5; ++v) cv[v] = F[v * NI * W + om] - F[v * NI * W + op];
        cv[0] *= hr;
        if (a.fv == nullptr) {
#pragma unroll
          for (int v = 1; v < 5; ++v) cv[v] *= hr;
        } else {
          const df r12d = d2df_bits(r12);
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const float2* fc = reinterpret_cast<const float2*>(fvs + cc * NV * W);
            auto ld = [&](int j) { const float2 v = fc[tile_idx<D, W>(j, line, NV)]; return df{v.x, v.y}; };
            const df t = d4_dfv(ld(pp), ld(pp + 1), ld(pp + 3), ld(pp + 4), r12d);
            cv[1 + cc] = fma(cv[1 + cc], hr, f2d_bits(t.hi)) + f2d_bits(t.lo);
          }
        }
        dir_epilogue_pre<TS>(a, flat(s0 + pp, a0 + line), cv, pre + item);
        continue;
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) cv[v] = F[v * NI * W + om] - F[v * NI * W + op];
      if (a.fv != nullptr) {
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          const double* fc = fvs + cc * NP * W;
          const double d1 = fc[tile_idx<D, W>(pp + 4, line, NP)] - fc[tile_idx<D, W>(pp + 2, line, NP)];
          const double d2 = fc[tile_idx<D, W>(pp + 5, line, NP)] - fc[tile_idx<D, W>(pp + 1, line, NP)];
          cv[1 + cc] = fma(fma(8.0, d1, -d2), r12, cv[1 + cc]);
        }
      }
      const long long p = flat(s0 + pp, a0 + line);
      dir_epilogue_pre<TS>(a, p, cv, pre + item);
    }
  }
}

}  // namespace ns3d
