// FP32-bulk direction pass (precision NS3D_FP32_BULK): the fused WENO5 + Roe +
// conservative difference + viscous divergence of k_dir.cu with the primitive
// variables, point fluxes, smoothness indicators, weights, interface values, the
// Roe flux and the viscous interface flux in FP32 (arXiv 2211.16718, Sec. 2.2
// arithmetic unchanged, precision reduced).  The total interface flux is widened
// to FP64 before the conservative difference, so the sums over the grid still
// telescope exactly; the accumulation / RK stage update and the state stay FP64.
//
// Layout of one tile (TP points along the pencil x W lines, 256 threads):
//  A   load the state (FP64, converted to FP32 by bit manipulation) at the tile's
//      points and a 3-point halo, form the primitive variables and point fluxes in
//      registers (no primitive planes are read), and the viscous flux of this
//      direction (FP32 planes of the viscous kernel);
//  BC  one item = one scalar on one line over SEG consecutive interfaces: the
//      SEG + 5 point values are read once (vector loads) and slid through in
//      registers: the window indicators, the left- and right-biased WENO5 values,
//      and their jump (conserved variables) or sum (flux components);
//  D   per interface: Roe average, wave strengths with Harten's fix, the central
//      part, the viscous interface flux (-f_{i-1} + 7 f_i + 7 f_{i+1} - f_{i+2})/12,
//      divided by dx and widened to FP64;
//  E   per point: FP64 difference of its two interface fluxes, then the
//      accumulation / RK epilogue (its operands prefetched by cp.async during D, in the y
//      and z passes two x-adjacent points per 16-byte copy).
#include <math.h>

#include "df.cuh"
#include "k_dir_common.cuh"
#include "ns3d_internal.cuh"

namespace ns3d {

namespace {

constexpr int THREADS = 256;
// At most 27 points along x, 26 along y and z (balanced tiles, k_dir_common.cuh) x 8 lines.  26 are 256
// points with the halo, one per thread in phase A; 27 take a second round of 8, and pay where they save a
// short line a tile.  Passes over 2^24 points with 27 / 26, where the number of tiles differs (elsewhere
// the two are equal):
//   x at nx = 54 156 / 184 us, 160 451 / 462, 320 675 / 725, 500 646 / 696, 512 663 / 661
//   y at ny = 54 182 / 216 us, 160 509 / 521, 320 795 / 799, 400 789 / 787, 512 768 / 756
//   z at nz = 54 241 / 283 us, 160 702 / 732, 320 1058 / 1057, 400 1048 / 1039, 512 1023 / 1012
// so that 27 is the better limit along x at every length, while along y and z 26 is the better one only
// from 400 points up, the sizes that this mode is for.  The 512^3 step with 24 everywhere is 2 % slower,
// with 23 5 %.  Before, full tiles of 27 with a remainder computed in full and two points per thread in E:
// 5.59 / 6.85 / 10.21 ms at 512^3 where these take 5.55 / 6.26 / 10.28 (and 69 % of the work wasted on a
// 32-point line).
__host__ __device__ constexpr int tile_max(int d) { return d == 0 ? 27 : 26; }
constexpr int TP = tile_max(0), W = 8;
constexpr int NP = TP + 6;      // positions per line: 3-point halo on each side
constexpr int NI = TP + 1;      // interfaces per line
constexpr int SEG = 4;          // interfaces per reconstruction item
constexpr int NSEG = (NI + SEG - 1) / SEG;  // 7
constexpr int NQ = 9;           // reconstructed scalars: 5 conserved, 4 flux components (f_0 = u_{1+D})
constexpr int RS = 28;          // line stride (floats) of the reconstruction results: whole segments
constexpr int NREC = 10;        // per interface: 5 jumps, the sum of u_{1+D}, 4 flux sums
constexpr int LS = 36;          // line stride (floats) of the scalar planes: >= SEG*NSEG + 5 and a multiple of 4
constexpr int L4 = NP;          // line stride (float4) of the Roe-input and viscous planes (odd: no bank conflicts)
static_assert(SEG * (NSEG - 1) + 12 <= LS && LS % 4 == 0 && RS == SEG * NSEG, "segment reads (three float4) stay in the line");
// shared-memory plan (bytes)
constexpr int OFF_R4 = 0;                             // float4 [W][L4]: sqrt(rho), u, v, w
constexpr int OFF_H = OFF_R4 + W * L4 * 16;           // float  [W][L4]: H
constexpr int OFF_V4 = OFF_H + ((W * L4 * 4 + 15) & ~15);  // float4 [W][L4]: viscous flux of this direction
constexpr int OFF_REC = OFF_V4 + W * L4 * 16;         // float  [NREC][W][RS]
constexpr int FS = 30;          // line stride (doubles) of the interface fluxes (no bank conflicts in y, z)
constexpr int OFF_F = OFF_REC + NREC * W * RS * 4;    // double [5][W][FS]: interface flux / dx
constexpr int OFF_Q = OFF_F + 5 * W * FS * 8;          // float  [NQ][W][LS]; dead after BC: the epilogue operands,
constexpr int TS = TP * W;                            //   double [15][TP*W], from here on
constexpr int BYTES = OFF_Q + 15 * TS * 8;
static_assert(FS >= NI, "interface-flux line");
static_assert(NQ * W * LS * 4 <= 15 * TS * 8, "the scalar planes fit the operands' space");
static_assert(BYTES + 1024 <= 233472 / 4, "four CTAs per SM");
static_assert(OFF_Q % 16 == 0 && OFF_V4 % 16 == 0 && OFF_F % 8 == 0 && OFF_REC % 16 == 0, "alignment");
static_assert(TP * W <= THREADS && NI * W <= THREADS, "one point / interface per thread in D and E");

// FP64 -> FP32 by truncating the bit pattern (integer instructions only): sign and exponent
// exact for |x| in [2^-126, 2^128); smaller magnitudes give signed zero, larger ones, infinities
// and NaNs give +-inf (a non-finite state is then reported by the checks of phase A).
__device__ __forceinline__ float d2f_tz(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t e11 = (h >> 20) & 0x7ffu;
  uint32_t b = __funnelshift_l(l, h, 3) + 0x40000000u;  // rebased exponent, top 23 mantissa bits
  b = (e11 <= 896u) ? 0u : b;
  b = (e11 >= 1151u) ? 0x7f800000u : b;
  return __uint_as_float(b | (h & 0x80000000u));
}

__device__ __forceinline__ float rcp_a(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_a(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Weighted WENO5 value written as an offset from the candidate c with the linear weight 6/10
// (Sec. 2.2: sum_k omega_k F_k = F_2 + omega_1 (F_1 - F_2) + omega_3 (F_3 - F_2)), the candidate
// differences being third differences of the data: with omega_k ~ c_k / B_k, c = (1, 6, 3)/10
// and B_k = (4 (eps + beta_k))^2, over the common denominator,
//   value = c + (B2 B3 d1 + 3 B1 B2 d3) / (B2 B3 + 6 B1 B3 + 3 B1 B2),
// d1 = F_1 - F_2, d3 = F_3 - F_2.  Unscaled products and an approximate reciprocal: valid while
// every B and product stays in the normal FP32 range (checked by the caller).
__device__ __forceinline__ float weno_fast(float B1, float B2, float B3, float c, float d1, float d3x3) {
  const float p23 = B2 * B3, p12 = B1 * B2;
  const float den = fmaf(6.0f * B1, B3, fmaf(3.0f, p12, p23));
  const float num = fmaf(p23, d1, p12 * d3x3);
  return fmaf(num, rcp_a(den), c);
}

// The same for any data whose squared indicators are finite (differences up to ~1e9; else bit 1 of
// bad is set): the B_k rescaled by a common power of two, the largest to [1, 2), and an IEEE
// division.  A B_k more than 2^96 above the smallest is cut to that ratio (constant data next to a
// large jump), so that den, at least the product of the two largest, stays a normal float.
__device__ __forceinline__ float weno_safe(float B1, float B2, float B3, float c, float d1, float d3x3, int& bad) {
  const int e1 = exponent_of(B1), e2 = exponent_of(B2), e3 = exponent_of(B3);
  const int top = max(e1, max(e2, e3));
  bad |= (top >= 128) ? 2 : 0;
  const float sc = pow2f(-min(min(top, min(e1, min(e2, e3)) + 96), 126));
  B1 = fminf(B1 * sc, 2.0f);
  B2 = fminf(B2 * sc, 2.0f);
  B3 = fminf(B3 * sc, 2.0f);
  const float p23 = B2 * B3, p12 = B1 * B2;
  const float den = fmaf(6.0f * B1, B3, fmaf(3.0f, p12, p23));
  const float num = fmaf(p23, d1, p12 * d3x3);
  return c + __fdiv_rn(num, den);
}

template <int D>
__global__ void __launch_bounds__(THREADS, 4) k_dir32(const DirArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  float* Q = reinterpret_cast<float*>(smem + OFF_Q);
  float4* R4 = reinterpret_cast<float4*>(smem + OFF_R4);
  float* HS = reinterpret_cast<float*>(smem + OFF_H);
  float4* V4 = reinterpret_cast<float4*>(smem + OFF_V4);
  float* REC = reinterpret_cast<float*>(smem + OFF_REC);
  double* FD = reinterpret_cast<double*>(smem + OFF_F);
  double* PRE = reinterpret_cast<double*>(smem + OFF_Q);

  constexpr int AX = (D == 0) ? 1 : 0;
  const int nD = a.g.n[D], na = a.g.n[AX];
  const long long N = a.g.N;
  const bool swap = (D == 2 && a.zorder);  // z pass with the line groups first (dir_zorder)
  int s0, len;
  tile_span(1, nD, a.tile_u, a.tile_r, swap ? blockIdx.y : blockIdx.x, s0, len);
  const int np = len + 6, ni = len + 1, nseg = (ni + SEG - 1) / SEG;  // this tile's positions, interfaces, segments
  const int a0 = (swap ? blockIdx.x : blockIdx.y) * W;
  const int bz = blockIdx.z;
  const int tid = threadIdx.x;
  const float* fvf = reinterpret_cast<const float*>(a.fv);
  const long long fv_plane = (long long)(a.fv_dstride * D);
  // FP32 parameters rounded on the host (an FP64 -> FP32 conversion per thread would occupy the FP64 pipe)
  const float gm1 = a.gm1_hi;

  // ---- A: load, convert, primitive variables and point fluxes -------------------------
  int bad = 0;  // bit 0: non-physical, bit 1: differences beyond the indicators' range
  for (int it = tid; it < np * W; it += THREADS) {
    int pos, line;
    if (D == 0) {
      line = (int)(((unsigned)it * c_rcp20.v[np]) >> 20);
      pos = it - line * np;
    } else {
      pos = it / W;
      line = it - pos * W;
    }
    int c = s0 - 3 + pos;
    if (c < 0 || c >= nD) c = wrap_idx(c, nD);
    const int la = min(a0 + line, na - 1);
    const long long p = tile_flat<D>(a.g, c, la, bz);
    const float rho = d2f_tz(__ldg(a.u + p)), mx = d2f_tz(__ldg(a.u + N + p));
    const float my = d2f_tz(__ldg(a.u + 2 * N + p)), mz = d2f_tz(__ldg(a.u + 3 * N + p));
    const float e = d2f_tz(__ldg(a.u + 4 * N + p));
    float4 fv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (fvf != nullptr) {
      const float* fp = fvf + fv_plane * N + p;
      fv = make_float4(__ldg(fp), __ldg(fp + N), __ldg(fp + 2 * N), __ldg(fp + 3 * N));
    }
    const float ri = rcp_a(rho);
    const float vx = mx * ri, vy = my * ri, vz = mz * ri;
    const float ke2 = fmaf(mx, vx, fmaf(my, vy, mz * vz));
    const float pr = gm1 * fmaf(-0.5f, ke2, e);
    const float ep = e + pr;
    bad |= !(rho > 0.0f && rho < INFINITY && pr > 0.0f && pr < INFINITY);
    const float un = (D == 0) ? vx : (D == 1) ? vy : vz;
    float* q = Q + line * LS + pos;
    const float sc[NQ] = {rho, mx, my, mz, e, (D == 0) ? fmaf(mx, un, pr) : mx * un, (D == 1) ? fmaf(my, un, pr) : my * un,
                          (D == 2) ? fmaf(mz, un, pr) : mz * un, ep * un};
#pragma unroll
    for (int m = 0; m < NQ; ++m) q[m * W * LS] = sc[m];
    // the last segment's points beyond the tile repeat the last one (no difference, no effect on the
    // segment's choice of arithmetic); their interfaces are never read
    if (pos == np - 1) {
      for (int k = 1; k <= nseg * SEG - ni; ++k)
#pragma unroll
        for (int m = 0; m < NQ; ++m) q[m * W * LS + k] = sc[m];
    }
    float sr;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(sr) : "f"(rho));
    R4[line * L4 + pos] = make_float4(sr, vx, vy, vz);
    HS[line * L4 + pos] = ep * ri;
    V4[line * L4 + pos] = fv;
  }
  __syncthreads();

  // ---- BC: WENO5 left/right values, SEG interfaces of one scalar on one line per item -------
  // Items run over lines fastest, then segments, then scalars, so that the 8 threads of a
  // shared-memory phase read and write 8 different banks.
  {
    const float eps4 = a.eps4_hi;
    const bool eps_ok = eps4 >= 1e-9f && eps4 <= 1.0f;  // unscaled products stay in range (see below)
    const unsigned rcp_nseg = c_rcp20.v[nseg];
    for (int it = tid; it < NQ * W * nseg; it += THREADS) {
      const int ms = it / W, line = it - ms * W;
      const int m = (int)(((unsigned)ms * rcp_nseg) >> 20), seg = ms - m * nseg;
      const float* q = Q + (m * W + line) * LS + SEG * seg;
      const float4 qa = *reinterpret_cast<const float4*>(q);
      const float4 qb = *reinterpret_cast<const float4*>(q + 4);
      const float4 qc = *reinterpret_cast<const float4*>(q + 8);
      const float P[SEG + 5] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w, qc.x};
      // first, second and third differences; window w = points w, w+1, w+2
      float g[SEG + 4], sd[SEG + 3], T3[SEG + 2], T2[SEG + 2];
      float gmax = 0.0f;
#pragma unroll
      for (int k = 0; k < SEG + 4; ++k) {
        g[k] = P[k + 1] - P[k];
        gmax = fmaxf(gmax, fabsf(g[k]));
      }
#pragma unroll
      for (int w = 0; w < SEG + 3; ++w) sd[w] = g[w + 1] - g[w];
#pragma unroll
      for (int k = 0; k < SEG + 2; ++k) {
        const float T = sd[k + 1] - sd[k];
        T3[k] = (1.0f / 3.0f) * T;
        T2[k] = 0.5f * T;
      }
      // window indicators, roles 1..3 (first-derivative term at the window's right end, centre,
      // left end)
      float B[SEG + 3][3];
#pragma unroll
      for (int w = 0; w < SEG + 3; ++w) {
        const float gm = g[w], gp = g[w + 1];
        const float aa = fmaf((13.0f / 3.0f) * sd[w], sd[w], eps4);
        const float u1 = fmaf(3.0f, gp, -gm), u2 = gm + gp, u3 = fmaf(-3.0f, gm, gp);
        const float b1 = fmaf(u1, u1, aa), b2 = fmaf(u2, u2, aa), b3 = fmaf(u3, u3, aa);
        B[w][0] = b1 * b1;
        B[w][1] = b2 * b2;
        B[w][2] = b3 * b3;
      }
      // With every first difference <= 64 in magnitude and 1e-9 <= 4 eps <= 1, each B lies in
      // [(4 eps)^2, (34 * 64^2 + 1)^2] and the products and the numerator stay within the normal
      // FP32 range: the unscaled form is exact to FP32 rounding.
      const bool fast = eps_ok && gmax <= 64.0f;
      float vL[SEG], vR[SEG];
#pragma unroll
      for (int j = 0; j < SEG; ++j) {
        // interface j: left-biased from points j..j+4, right-biased from j+1..j+5; candidate-2
        // values eR (left) and eL (right); F_1 - F_2 = -T_j/3, F_3 - F_2 = -T_{j+1}/6 (left),
        // F_1 - F_2 = T_{j+2}/3, F_3 - F_2 = T_{j+1}/6 (right)
        const float eR = fmaf(1.0f / 3.0f, g[j + 2], fmaf(1.0f / 6.0f, g[j + 1], P[j + 2]));
        const float eL = fmaf(-1.0f / 6.0f, g[j + 3], fmaf(-1.0f / 3.0f, g[j + 2], P[j + 3]));
        if (fast) {
          vL[j] = weno_fast(B[j][0], B[j + 1][1], B[j + 2][2], eR, -T3[j], -T2[j + 1]);
          vR[j] = weno_fast(B[j + 3][2], B[j + 2][1], B[j + 1][0], eL, T3[j + 2], T2[j + 1]);
        } else {
          vL[j] = weno_safe(B[j][0], B[j + 1][1], B[j + 2][2], eR, -T3[j], -T2[j + 1], bad);
          vR[j] = weno_safe(B[j + 3][2], B[j + 2][1], B[j + 1][0], eL, T3[j + 2], T2[j + 1], bad);
        }
      }
      float* r = REC + line * RS + SEG * seg;
      if (m < 5) {
        *reinterpret_cast<float4*>(r + m * W * RS) =
            make_float4(vR[0] - vL[0], vR[1] - vL[1], vR[2] - vL[2], vR[3] - vL[3]);
        if (m == 1 + D)
          *reinterpret_cast<float4*>(r + 5 * W * RS) =
              make_float4(vL[0] + vR[0], vL[1] + vR[1], vL[2] + vR[2], vL[3] + vR[3]);
      } else {
        *reinterpret_cast<float4*>(r + (m + 1) * W * RS) =
            make_float4(vL[0] + vR[0], vL[1] + vR[1], vL[2] + vR[2], vL[3] + vR[3]);
      }
    }
  }
  __syncthreads();

  // ---- epilogue operands: fetched asynchronously into the dead scalar planes and behind them while D
  //      runs.  y and z passes on grids with nx even take two x-adjacent points (lines 2j, 2j+1 of the
  //      tile; their flat index is even) per 16-byte copy.  U_n and the stage input may be the
  //      caller's and only 8-byte aligned; the rest is the library's.
  const bool pairs = D != 0 && (a.g.n[0] & 1) == 0 && (((uintptr_t)a.un | (uintptr_t)a.u) & 15) == 0;
  auto point_of = [&](int it, int& pp, int& line) {
    if (D == 0) {
      line = (int)(((unsigned)it * c_rcp20.v[len]) >> 20);
      pp = it - line * len;
    } else {
      pp = it / W;
      line = it - pp * W;
    }
  };
  if (pairs) {
    if (tid < len * W / 2) {
      const int pp = tid / (W / 2), l0 = 2 * (tid - pp * (W / 2));
      if (a0 + l0 < na)  // na = nx is even: the second point exists too
        epilogue_prefetch<true, TS>(a, tile_flat<D>(a.g, s0 + pp, a0 + l0, bz), PRE + 2 * tid);
    }
  } else if (tid < len * W) {
    int pp, line;
    point_of(tid, pp, line);
    if (a0 + line < na) epilogue_prefetch<false, TS>(a, tile_flat<D>(a.g, s0 + pp, a0 + line, bz), PRE + tid);
  }
  cp_async_commit();

  // ---- D: Roe flux + viscous interface flux, / dx, widened to FP64 ----------------------
  if (tid < ni * W) {
    int r, line;
    if (D == 0) {
      line = (int)(((unsigned)tid * c_rcp20.v[ni]) >> 20);
      r = tid - line * ni;
    } else {
      r = tid / W;
      line = tid - r * W;
    }
    // interface r lies between the tile's points r - 1 and r, i.e. positions r + 2 and r + 3
    const float* rc_ = REC + line * RS + r;
    float du[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) du[v] = rc_[v * W * RS];
    const float S0 = rc_[5 * W * RS];
    const float S1 = rc_[6 * W * RS], S2 = rc_[7 * W * RS], S3 = rc_[8 * W * RS], S4 = rc_[9 * W * RS];
    const float4 qa = R4[line * L4 + r + 2], qb = R4[line * L4 + r + 3];
    const float Ha = HS[line * L4 + r + 2], Hb = HS[line * L4 + r + 3];
    const float rs = rcp_a(qa.x + qb.x);
    const float wa = qa.x * rs, wb = qb.x * rs;
    const float V0 = fmaf(wa, qa.y, wb * qb.y), V1 = fmaf(wa, qa.z, wb * qb.z), V2 = fmaf(wa, qa.w, wb * qb.w);
    const float H = fmaf(wa, Ha, wb * Hb);
    const float q2h = 0.5f * fmaf(V0, V0, fmaf(V1, V1, V2 * V2));
    const float c2 = gm1 * (H - q2h);
    bad |= !(c2 > 0.0f);
    const float rc = rsqrt_a(c2);
    const float c = c2 * rc;
    constexpr int T1 = (D == 0) ? 1 : 0;
    constexpr int T2 = (D == 2) ? 1 : 2;
    const float V[3] = {V0, V1, V2};
    const float un = V[D], vt1 = V[T1], vt2 = V[T2];
    const float b1 = gm1 * (rc * rc);
    const float vdm = fmaf(V0, du[1], fmaf(V1, du[2], V2 * du[3]));
    const float phi = b1 * (fmaf(q2h, du[0], du[4]) - vdm);
    const float a2 = du[0] - phi;
    const float a3 = fmaf(-vt1, du[0], du[1 + T1]);
    const float a4 = fmaf(-vt2, du[0], du[1 + T2]);
    const float ach = 0.5f * (fmaf(un, du[0], -du[1 + D]) * rc);
    const float ph = 0.5f * phi;
    const float a1 = ph + ach, a5 = ph - ach;
    float l1 = fabsf(un - c), l5 = fabsf(un + c);
    const float l2 = fabsf(un);
    const float hd = a.hd_hi;
    const float delta = hd * c;
    if (l1 < delta) l1 = fmaf(l1, l1, delta * delta) * __fdividef(0.5f, delta);
    if (l5 < delta) l5 = fmaf(l5, l5, delta * delta) * __fdividef(0.5f, delta);
    const float A1 = l1 * a1, A2 = l2 * a2, A3 = l2 * a3, A4 = l2 * a4, A5 = l5 * a5;
    const float S = A1 + A5;
    const float d0 = S + A2;
    const float cD = c * (A5 - A1);
    float diss[5];
    diss[0] = d0;
    diss[1 + D] = fmaf(d0, un, cD);
    diss[1 + T1] = fmaf(d0, vt1, A3);
    diss[1 + T2] = fmaf(d0, vt2, A4);
    diss[4] = fmaf(S, H, fmaf(cD, un, fmaf(A2, q2h, fmaf(A3, vt1, A4 * vt2))));
    // viscous interface flux: its difference over the two faces of a point is the 4th-order
    // central derivative (f_{i-2} - 8 f_{i-1} + 8 f_{i+1} - f_{i+2}) / 12 of the point values
    const float4 fm1 = V4[line * L4 + r + 1], f0 = V4[line * L4 + r + 2];
    const float4 f1 = V4[line * L4 + r + 3], f2 = V4[line * L4 + r + 4];
    const float G0 = fmaf(7.0f / 12.0f, f0.x + f1.x, (-1.0f / 12.0f) * (fm1.x + f2.x));
    const float G1 = fmaf(7.0f / 12.0f, f0.y + f1.y, (-1.0f / 12.0f) * (fm1.y + f2.y));
    const float G2 = fmaf(7.0f / 12.0f, f0.z + f1.z, (-1.0f / 12.0f) * (fm1.z + f2.z));
    const float G3 = fmaf(7.0f / 12.0f, f0.w + f1.w, (-1.0f / 12.0f) * (fm1.w + f2.w));
    const float rdx = a.g.rh_f[D];
    const float F0 = 0.5f * (S0 - diss[0]);
    const float F1 = fmaf(0.5f, S1 - diss[1], -G0);
    const float F2 = fmaf(0.5f, S2 - diss[2], -G1);
    const float F3 = fmaf(0.5f, S3 - diss[3], -G2);
    const float F4 = fmaf(0.5f, S4 - diss[4], -G3);
    double* fd = FD + line * FS + r;
    fd[0 * W * FS] = f2d_bits(F0 * rdx);
    fd[1 * W * FS] = f2d_bits(F1 * rdx);
    fd[2 * W * FS] = f2d_bits(F2 * rdx);
    fd[3 * W * FS] = f2d_bits(F3 * rdx);
    fd[4 * W * FS] = f2d_bits(F4 * rdx);
  }
  if (__any_sync(0xffffffffu, bad)) {
    const int any = __reduce_or_sync(0xffffffffu, bad);
    if ((tid & 31) == 0) atomicOr(a.status, ((any & 1) ? ST_NONPHYS : 0) | ((any & 2) ? ST_DF_RANGE : 0));
  }
  cp_async_wait_all();
  __syncthreads();

  // ---- E: FP64 difference + epilogue, one point per thread (the FP64 work then spreads over
  //      seven warps; two points per thread left it on four.  512^3 y pass 6.85 -> 6.23 ms)
  if (tid < len * W) {
    int pp, line;
    point_of(tid, pp, line);
    if (a0 + line < na) {
      const double* fd = FD + line * FS + pp;
      double cv[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) cv[v] = fd[v * W * FS] - fd[v * W * FS + 1];
      dir_epilogue_pre<TS>(a, tile_flat<D>(a.g, s0 + pp, a0 + line, bz), cv, PRE + tid);
    }
  }
}

template <int D>
cudaError_t launch32(const DirArgs& a, cudaStream_t s) {
  constexpr int AX = (D == 0) ? 1 : 0;
  constexpr int BX = (D == 2) ? 1 : 2;
  constexpr int TM = tile_max(D);
  dim3 grid((a.g.n[D] + TM - 1) / TM, (a.g.n[AX] + W - 1) / W, a.g.n[BX]);
  if (D == 2 && a.zorder) {
    const unsigned t = grid.x;
    grid.x = grid.y;
    grid.y = t;
  }
  DirArgs r = a;
  tile_split_units(1, a.g.n[D], (a.g.n[D] + TM - 1) / TM, r.tile_u, r.tile_r);  // units of one point
  k_dir32<D><<<grid, THREADS, BYTES, s>>>(r);
  return cudaGetLastError();
}

template <int D>
cudaError_t attr32() {
  cudaError_t e = cudaFuncSetAttribute(k_dir32<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_dir32<D>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

}  // namespace

cudaError_t prepare_dir32_kernels() {
  cudaError_t e = attr32<0>();
  if (e == cudaSuccess) e = attr32<1>();
  if (e == cudaSuccess) e = attr32<2>();
  return e;
}

// One tile shape for every pass; the tile variants of the FP64 modes do not apply.
cudaError_t launch_dir32(int d, const DirArgs& a, cudaStream_t s) {
  if (d == 0) return launch32<0>(a, s);
  if (d == 1) return launch32<1>(a, s);
  return launch32<2>(a, s);
}

}  // namespace ns3d
