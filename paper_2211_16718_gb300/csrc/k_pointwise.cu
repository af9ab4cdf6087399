// Pointwise and stencil-reduction kernels of libns3d.so:
//  - primitive variables (Sec. 2.1 equation of state),
//  - velocity/temperature gradients -> viscous flux vectors f^v, g^v, h^v
//    (Sec. 2.1 stresses and heat flux, 4th-order central differences),
//  - statistics (conservation sums, kinetic energy, enstrophy, extrema, CFL)
//    with a deterministic two-level FP64 reduction (fixed-order folds per block, then
//    over the blocks' partials).
#include <math.h>

#include <algorithm>

#include "df.cuh"
#include "df2.cuh"
#include "k_point_impl.cuh"
#include "ns3d_internal.cuh"

namespace ns3d {

namespace {

constexpr int PW_THREADS = 256;

int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  long long cap = 152LL * 16;
  return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}

// Primitive variables of every point (body: prim_point; DF: the NS3D_FP64 layout).
template <bool DF>
__global__ void __launch_bounds__(PW_THREADS) k_prim(const double* __restrict__ u, double* __restrict__ pm,
                                                     long long N, long long p0, long long p1, double gamma,
                                                     int* __restrict__ status) {
  int bad = 0;
  for (long long p = p0 + blockIdx.x * (long long)blockDim.x + threadIdx.x; p < p1; p += (long long)gridDim.x * blockDim.x)
    bad |= prim_point<DF>(u, pm, N, p, gamma);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(status, ST_NONPHYS);
}

// Gradients of (u, v, w, T) at every point, then the three viscous flux vectors, all FP64
// (NS3D_FP64_STRICT; body: visc_point_ijk).  The NS3D_FP64 form is k_visc_tiled below.
__global__ void __launch_bounds__(PW_THREADS) k_visc(const double* __restrict__ pm, double* __restrict__ fv,
                                                     int nx, int ny, int nz, double r12hx, double r12hy,
                                                     double r12hz, double mu, double kappa, int only_d, int z0) {
  // one thread per point of a 32 x 8 block of an x-y plane; blockIdx.z = the plane (from z0)
  const int i = blockIdx.x * 32 + threadIdx.x % 32, j = blockIdx.y * 8 + threadIdx.x / 32, k = z0 + blockIdx.z;
  if (i >= nx || j >= ny) return;
  const double r12[3] = {r12hx, r12hy, r12hz};
  visc_point_ijk(pm, fv, nx, ny, nz, i, j, k, r12, mu, kappa, only_d);
}

// Tiled NS3D_FP64 viscous-flux kernel (primitives in the layout of prim_point<true>).  A CTA
// owns a 32 x 8 block of x-y columns and marches along z through cz planes (visc_chunk).  Each plane of
// (u, v, w, T), with a 2-point x-y halo, is converted to double-float once into a ring of 5
// planes (z-2 .. z+2) in shared memory, so every stencil value is converted once rather than
// once per stencil that uses it (12 times).  The ring holds the fields in pairs, (u, v) and
// (w, T), each position a 16-byte record (hi, hi, lo, lo): the 12 gradient stencils run as 6
// two-lane double-float stencils on the packed FP32 instructions (df2.cuh; each lane the
// operations of d4_dfv), the flux assembly reads the lanes as scalars.  The per-point
// arithmetic is that of visc_point_df_ijk: the same conversions, the same gradient and flux
// operations, so the same bits.
constexpr int VT_X = 32, VT_Y = 8, VT_HX = VT_X + 4, VT_HY = VT_Y + 4, VT_PLANE = VT_HX * VT_HY;
constexpr int VT_RING = 5;
constexpr int VT_SMEM = VT_RING * 2 * VT_PLANE * (int)sizeof(float4);  // 69,120 bytes

// d4_dfv on two lanes.
__device__ __forceinline__ df2 d4_dfv2(df2 qm2, df2 qm1, df2 qp1, df2 qp2, df2 r12h) {
  const df2 d1 = df2_add_fast(qp1, df2_neg(qm1));
  const df2 d2 = df2_add_fast(qp2, df2_neg(qm2));
  return df2_mul_u(df2_add_fast(df2_mul_f_u(d1, 8.0f), df2_neg(d2)), r12h);
}

__global__ void __launch_bounds__(VT_X * VT_Y, 3) k_visc_tiled(const double* __restrict__ pm, double* __restrict__ fv,
                                                                const Grid g, double mu, double kappa, int only_d,
                                                                int zb, int ze, int cz) {
  extern __shared__ float4 ring4[];  // [VT_RING][2][VT_HY][VT_HX]: (u, v) and (w, T)
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const long long N = g.N;
  const int x0 = blockIdx.x * VT_X, y0 = blockIdx.y * VT_Y, z0 = zb + blockIdx.z * cz;
  const int z1 = min(z0 + cz, ze);
  const int tid = threadIdx.x, tx = tid % VT_X, ty = tid / VT_X;
  const df2 r12[3] = {df2_splat(d2df_bits(g.r12h[0])), df2_splat(d2df_bits(g.r12h[1])),
                      df2_splat(d2df_bits(g.r12h[2]))};
  auto slot = [&](int zz) { return ring4 + ((zz - z0 + 2) % VT_RING) * 2 * VT_PLANE; };
  // in-plane offsets of this thread's halo-tile positions (the same for every plane)
  constexpr int NPOS = (VT_PLANE + VT_X * VT_Y - 1) / (VT_X * VT_Y);
  int xy[NPOS];
#pragma unroll
  for (int k = 0; k < NPOS; ++k) {
    const int pos = tid + k * VT_X * VT_Y;
    const int hy = pos / VT_HX, hx = pos - hy * VT_HX;
    xy[k] = wrap_idx(y0 - 2 + hy, ny) * nx + wrap_idx(x0 - 2 + hx, nx);
  }
  const long long plane_n = (long long)nx * ny;
  auto load_plane = [&](int zz) {  // plane zz (periodic) of the four fields, with halo
    const long long zoff = (long long)wrap_idx(zz, nz) * plane_n;
    float4* R = slot(zz);
#pragma unroll
    for (int k = 0; k < NPOS; ++k) {
      const int pos = tid + k * VT_X * VT_Y;
      if (pos >= VT_PLANE) break;
      const long long p = zoff + xy[k];
      const df vu = d2df_bits(__ldg(pm + (long long)PM_U * N + p));
      const df vv = d2df_bits(__ldg(pm + (long long)PM_V * N + p));
      const df vw = d2df_bits(__ldg(pm + (long long)PM_W * N + p));
      const float2 vT = __ldg(reinterpret_cast<const float2*>(pm + (long long)PM_T * N + p));  // double-float plane
      R[pos] = make_float4(vu.hi, vv.hi, vu.lo, vv.lo);
      R[VT_PLANE + pos] = make_float4(vw.hi, vT.x, vw.lo, vT.y);
    }
  };
  auto ld = [](const float4* P, int i) { return df2_from4(P[i]); };
  for (int zz = z0 - 2; zz < z0 + 2; ++zz) load_plane(zz);
  for (int z = z0; z < z1; ++z) {
    load_plane(z + 2);
    __syncthreads();
    if (x0 + tx < nx && y0 + ty < ny) {
      const int c = (ty + 2) * VT_HX + (tx + 2);
      const float4 *Zm2 = slot(z - 2), *Zm1 = slot(z - 1), *Z0 = slot(z), *Zp1 = slot(z + 1), *Zp2 = slot(z + 2);
      // the flux along only_d (lean storage) needs 8 of the 12 gradients: d(u, v, w, T)/dx_d, the
      // derivatives of the velocity component along only_d, and the diagonal (divergence)
      auto need = [&](int q, int e) { return only_d < 0 || e == only_d || (q < 3 && (q == only_d || q == e)); };
      df G[4][3];
#pragma unroll
      for (int k = 0; k < 2; ++k) {  // field pair k: (u, v) or (w, T)
        const float4* P = Z0 + k * VT_PLANE;
        const int o = k * VT_PLANE + c;
        df2 Gk[3];
        const df2 zero{f2splat(0.0f), f2splat(0.0f)};
        Gk[0] = (need(2 * k, 0) || need(2 * k + 1, 0))
                    ? d4_dfv2(ld(P, c - 2), ld(P, c - 1), ld(P, c + 1), ld(P, c + 2), r12[0]) : zero;
        Gk[1] = (need(2 * k, 1) || need(2 * k + 1, 1))
                    ? d4_dfv2(ld(P, c - 2 * VT_HX), ld(P, c - VT_HX), ld(P, c + VT_HX), ld(P, c + 2 * VT_HX), r12[1])
                    : zero;
        Gk[2] = (need(2 * k, 2) || need(2 * k + 1, 2)) ? d4_dfv2(ld(Zm2, o), ld(Zm1, o), ld(Zp1, o), ld(Zp2, o), r12[2])
                                                      : zero;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const df dz{0.0f, 0.0f};
          G[2 * k][e] = need(2 * k, e) ? df2_lane0(Gk[e]) : dz;
          G[2 * k + 1][e] = need(2 * k + 1, e) ? df2_lane1(Gk[e]) : dz;
        }
      }
      const df2 uv = ld(Z0, c), wT = ld(Z0 + VT_PLANE, c);
      const df vel[3] = {df2_lane0(uv), df2_lane1(uv), df2_lane0(wT)};
      visc_fluxes_df(G, vel, mu, kappa, fv, N, flat3(x0 + tx, y0 + ty, z, nx, ny), only_d);
    }
    __syncthreads();  // the slot of plane z - 2 takes plane z + 3 next
  }
}

// Launch geometry of the stencil point kernels: 32 x 8 x 1 blocks over (x, y, z).
inline dim3 plane_grid(const Grid& g) { return dim3((g.n[0] + 31) / 32, (g.n[1] + 7) / 8, g.n[2]); }

// ---- FP32-bulk viscous fluxes (NS3D_FP32_BULK) ---------------------------------------
// The tiled form of k_visc_tiled in FP32, straight from the conserved state: a CTA owns a
// 32 x 8 block of x-y columns and marches along z through cz planes (visc_chunk); every plane of
// (u, v, w, T), with a 2-point x-y halo, is formed once from the state (converted to FP32 by
// bit manipulation) into a ring of 5 planes (z-2 .. z+2) of float4 in shared memory.  Each
// point then takes the 12 gradients with the 4th-order central difference and writes the
// viscous flux vectors as FP32 planes fv[4 d + c][N] (only_d = d: fv[c][N]), which the FP32-bulk
// direction passes read.
__device__ __forceinline__ float d2f_trunc_fast(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t e11 = (h >> 20) & 0x7ffu;
  uint32_t b = __funnelshift_l(l, h, 3) + 0x40000000u;
  b = (e11 <= 896u) ? 0u : b;
  b = (e11 >= 1151u) ? 0x7f800000u : b;
  return __uint_as_float(b | (h & 0x80000000u));
}

// Five CTAs per SM (48 registers) instead of four: 512^3 2.69 -> 2.51 ms; six spill (step 2.3 % slower).
constexpr int V32_SMEM = VT_RING * VT_PLANE * (int)sizeof(float4);  // 34,560 bytes

__global__ void __launch_bounds__(VT_X * VT_Y, 5) k_visc32t(const double* __restrict__ u, float* __restrict__ fv,
                                                             const Grid g, float gamma, float mu, float kappa,
                                                             int only_d, int cz) {
  extern __shared__ float4 ring4[];  // [VT_RING][VT_HY][VT_HX]: u, v, w, T
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const long long N = g.N;
  const int x0 = blockIdx.x * VT_X, y0 = blockIdx.y * VT_Y, z0 = blockIdx.z * cz;
  const int z1 = min(z0 + cz, nz);
  const int tid = threadIdx.x, tx = tid % VT_X, ty = tid / VT_X;
  const float r12[3] = {(float)g.r12h[0], (float)g.r12h[1], (float)g.r12h[2]};
  const float gm1 = gamma - 1.0f;
  auto slot = [&](int zz) { return ring4 + ((zz - z0 + 2) % VT_RING) * VT_PLANE; };
  constexpr int NPOS = (VT_PLANE + VT_X * VT_Y - 1) / (VT_X * VT_Y);
  int xy[NPOS];
#pragma unroll
  for (int k = 0; k < NPOS; ++k) {
    const int pos = tid + k * VT_X * VT_Y;
    const int hy = pos / VT_HX, hx = pos - hy * VT_HX;
    xy[k] = wrap_idx(y0 - 2 + hy, ny) * nx + wrap_idx(x0 - 2 + hx, nx);
  }
  const long long plane_n = (long long)nx * ny;
  auto load_plane = [&](int zz) {
    const long long zoff = (long long)wrap_idx(zz, nz) * plane_n;
    float4* R = slot(zz);
#pragma unroll
    for (int k = 0; k < NPOS; ++k) {
      const int pos = tid + k * VT_X * VT_Y;
      if (pos >= VT_PLANE) break;
      const long long p = zoff + xy[k];
      const float rho = d2f_trunc_fast(__ldg(u + p)), mx = d2f_trunc_fast(__ldg(u + N + p));
      const float my = d2f_trunc_fast(__ldg(u + 2 * N + p)), mz = d2f_trunc_fast(__ldg(u + 3 * N + p));
      const float e = d2f_trunc_fast(__ldg(u + 4 * N + p));
      const float ri = __fdividef(1.0f, rho);
      const float vx = mx * ri, vy = my * ri, vz = mz * ri;
      const float pr = gm1 * fmaf(-0.5f, fmaf(mx, vx, fmaf(my, vy, mz * vz)), e);
      R[pos] = make_float4(vx, vy, vz, gamma * pr * ri);
    }
  };
  for (int zz = z0 - 2; zz < z0 + 2; ++zz) load_plane(zz);
  for (int z = z0; z < z1; ++z) {
    load_plane(z + 2);
    __syncthreads();
    if (x0 + tx < nx && y0 + ty < ny) {
      const int c = (ty + 2) * VT_HX + (tx + 2);
      const float4 *Zm2 = slot(z - 2), *Zm1 = slot(z - 1), *Z0 = slot(z), *Zp1 = slot(z + 1), *Zp2 = slot(z + 2);
      auto d4v = [](float4 m2, float4 m1, float4 p1, float4 p2, float r) {
        return make_float4(fmaf(8.0f, p1.x - m1.x, -(p2.x - m2.x)) * r, fmaf(8.0f, p1.y - m1.y, -(p2.y - m2.y)) * r,
                           fmaf(8.0f, p1.z - m1.z, -(p2.z - m2.z)) * r, fmaf(8.0f, p1.w - m1.w, -(p2.w - m2.w)) * r);
      };
      // G[d] = d(u, v, w, T)/dx_d
      const float4 Gd[3] = {d4v(Z0[c - 2], Z0[c - 1], Z0[c + 1], Z0[c + 2], r12[0]),
                            d4v(Z0[c - 2 * VT_HX], Z0[c - VT_HX], Z0[c + VT_HX], Z0[c + 2 * VT_HX], r12[1]),
                            d4v(Zm2[c], Zm1[c], Zp1[c], Zp2[c], r12[2])};
      float G[4][3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        G[0][d] = Gd[d].x;
        G[1][d] = Gd[d].y;
        G[2][d] = Gd[d].z;
        G[3][d] = Gd[d].w;
      }
      const float4 v0 = Z0[c];
      const float vel[3] = {v0.x, v0.y, v0.z};
      const float tdiv = (2.0f / 3.0f) * (G[0][0] + G[1][1] + G[2][2]);
      const long long p = flat3(x0 + tx, y0 + ty, z, nx, ny);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (only_d >= 0 && d != only_d) continue;
        const int b = (only_d >= 0) ? 0 : 4 * d;
        float tau[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) tau[m] = (m == d) ? mu * fmaf(2.0f, G[d][d], -tdiv) : mu * (G[m][d] + G[d][m]);
        const float en = fmaf(vel[0], tau[0], fmaf(vel[1], tau[1], fmaf(vel[2], tau[2], kappa * G[3][d])));
        fv[(long long)(b + 0) * N + p] = tau[0];
        fv[(long long)(b + 1) * N + p] = tau[1];
        fv[(long long)(b + 2) * N + p] = tau[2];
        fv[(long long)(b + 3) * N + p] = en;
      }
    }
    __syncthreads();  // the slot of plane z - 2 takes plane z + 3 next
  }
}

// ---- statistics ------------------------------------------------------------
constexpr int ST_THREADS = 256;
constexpr int ST_SLOTS = 152 * 4;  // CTAs of k_stats_tiled the GPU holds at once (4 per SM)
constexpr int NSUM = 7;   // mass, 3 momenta, energy, ke, enstrophy
constexpr int NRED = 10;  // + rho_min, p_min, max wavespeed/dx
constexpr int ST_FINAL_THREADS = 32 * NRED;

// Order of the doubles as signed 64-bit integers (for minima without the FP64 pipe): a < b if and
// only if dkey(a) < dkey(b); NaNs lie outside [dkey(-inf), dkey(+inf)].  Its own inverse.
__device__ __forceinline__ long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
constexpr long long DKEY_NINF = (long long)0x800fffffffffffffULL, DKEY_PINF = 0x7ff0000000000000LL;
// kmin = min(kmin, dkey(x)), a NaN x ignored (as fmin)
__device__ __forceinline__ void key_min(long long& kmin, double x) {
  const long long k = dkey(x);
  if (k < kmin && k >= DKEY_NINF) kmin = k;
}

// Sum (M = 0), minimum (1) or maximum (2) of the lanes' values in a fixed order; the result in lane 0.
template <int M>
__device__ __forceinline__ double warp_fold(double x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double y = __shfl_down_sync(0xffffffffu, x, off);
    x = (M == 0) ? x + y : (M == 1) ? fmin(x, y) : fmax(x, y);
  }
  return x;
}

// Fold of one quantity (0..NSUM-1: sum, NSUM and NSUM+1: minimum, last: maximum) by one warp over
// the n values v[0 .. n): every lane folds its values in order, then the lanes.
__device__ __forceinline__ double fold_column(int q, const double* v, int n, int lane) {
  double x = (q < NSUM) ? 0.0 : (q < NRED - 1) ? INFINITY : 0.0;
  if (q < NSUM) {
    for (int i = lane; i < n; i += 32) x += v[i];
    return warp_fold<0>(x);
  }
  if (q < NRED - 1) {
    for (int i = lane; i < n; i += 32) x = fmin(x, v[i]);
    return warp_fold<1>(x);
  }
  for (int i = lane; i < n; i += 32) x = fmax(x, v[i]);
  return warp_fold<2>(x);
}

// Statistics: a block walks its tiles of 32 x 8 x-y columns times cz planes in a fixed order; the
// velocity planes, with a 2-point x-y halo, are converted to double-float once into a 5-plane ring
// (z-2 .. z+2) for the vorticity stencils.  The accumulation order is fixed by the grid shape, so
// the result is deterministic.  Sums in FP64; kinetic energy, vorticity, enstrophy and wave speed in
// double-float on the FP32 pipe, their low words summed apart (compensated, FP32) so that a point
// costs 7 FP64 additions; minima as integers.  DFT: the temperature plane holds double-float pairs
// (prim_point<true>).
// What bounds it: FP64 additions and plane-load latency.  The block ends with one fold per quantity
// by one warp each through shared memory: 84 FP64 warp instructions where ten shuffle reductions by
// every warp took 400, and stats_plan launches no block without a tile.  128^3: 185 -> 86 us,
// 256^3: 618 -> 568 us, 32^3: 59 -> 11 us (ncu, cold cache).
constexpr int SR_SMEM = VT_RING * 3 * VT_PLANE * (int)sizeof(float2);  // 51,840 bytes
static_assert(NRED * ST_THREADS * (int)sizeof(double) <= SR_SMEM, "the block's fold fits the ring");

template <bool DFT>
__global__ void __launch_bounds__(ST_THREADS, 4) k_stats_tiled(const double* __restrict__ u, const double* __restrict__ pm,
                                                                const Grid g, double* __restrict__ partials, int ntx,
                                                                int nty, long long ntiles, int cz) {
  extern __shared__ float2 ring[];  // [VT_RING][3][VT_HY][VT_HX]
  static_assert(VT_X * VT_Y == ST_THREADS, "one point per thread and plane");
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const long long N = g.N;
  const long long plane_n = (long long)nx * ny;
  const df r12d[3] = {d2df_bits(g.r12h[0]), d2df_bits(g.r12h[1]), d2df_bits(g.r12h[2])};
  const df rhd[3] = {d2df_bits(g.rh[0]), d2df_bits(g.rh[1]), d2df_bits(g.rh[2])};
  const int tid = threadIdx.x, tx = tid % VT_X, ty = tid / VT_X;
  constexpr int NPOS = (VT_PLANE + ST_THREADS - 1) / ST_THREADS;
  df wmax{0.0f, 0.0f};
  double sum[NSUM];
#pragma unroll
  for (int m = 0; m < NSUM; ++m) sum[m] = 0.0;
  df klo{0.0f, 0.0f}, elo{0.0f, 0.0f};  // low words of the kinetic energy and the enstrophy
  long long rmin = DKEY_PINF, pmin = DKEY_PINF;
  auto ld = [](const float2* P, int i) { const float2 v = P[i]; return df{v.x, v.y}; };
  auto add_lo = [](df& s, float x) {  // compensated
    const df t = two_sum(s.hi, x);
    s = df{t.hi, __fadd_rn(s.lo, t.lo)};
  };
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int x0 = (int)(t % ntx) * VT_X;
    const long long rest = t / ntx;
    const int y0 = (int)(rest % nty) * VT_Y, z0 = (int)(rest / nty) * cz;
    const int z1 = min(z0 + cz, nz);
    auto slot = [&](int zz) { return ring + ((zz - z0 + 2) % VT_RING) * 3 * VT_PLANE; };
    int xy[NPOS];
#pragma unroll
    for (int k = 0; k < NPOS; ++k) {
      const int pos = tid + k * ST_THREADS;
      const int hy = pos / VT_HX, hx = pos - hy * VT_HX;
      xy[k] = wrap_idx(y0 - 2 + hy, ny) * nx + wrap_idx(x0 - 2 + hx, nx);
    }
    auto load_plane = [&](int zz) {
      const long long zoff = (long long)wrap_idx(zz, nz) * plane_n;
      float2* R = slot(zz);
#pragma unroll
      for (int k = 0; k < NPOS; ++k) {
        const int pos = tid + k * ST_THREADS;
        if (pos >= VT_PLANE) break;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const df v = d2df_bits(__ldg(pm + (long long)q * N + zoff + xy[k]));
          R[q * VT_PLANE + pos] = make_float2(v.hi, v.lo);
        }
      }
    };
    __syncthreads();  // the previous tile's last reads of the ring
    for (int zz = z0 - 2; zz < z0 + 2; ++zz) load_plane(zz);
    for (int z = z0; z < z1; ++z) {
      load_plane(z + 2);
      __syncthreads();
      if (x0 + tx < nx && y0 + ty < ny) {
        const long long p = (long long)z * plane_n + (long long)(y0 + ty) * nx + (x0 + tx);
        const int c = (ty + 2) * VT_HX + (tx + 2);
        const float2 *Zm2 = slot(z - 2), *Zm1 = slot(z - 1), *Z0 = slot(z), *Zp1 = slot(z + 1), *Zp2 = slot(z + 2);
        const double rho = __ldg(u + p);
        const double pr = __ldg(pm + PM_P * N + p);
        sum[0] += rho;
        sum[1] += __ldg(u + N + p);
        sum[2] += __ldg(u + 2 * N + p);
        sum[3] += __ldg(u + 3 * N + p);
        sum[4] += __ldg(u + 4 * N + p);
        const df rd = d2df_bits(rho);
        const df rh2{0.5f * rd.hi, 0.5f * rd.lo};  // rho / 2, exact
        const df vd[3] = {ld(Z0, c), ld(Z0 + VT_PLANE, c), ld(Z0 + 2 * VT_PLANE, c)};
        const df ke = df_mul_u(rh2, df_add_pos_u(df_sqr_u(vd[0]), df_add_pos_u(df_sqr_u(vd[1]), df_sqr_u(vd[2]))));
        sum[5] += f2d_bits(ke.hi);
        add_lo(klo, ke.lo);
        // vorticity: dv_m/dx_d for m != d
        auto gx = [&](int m) {
          const float2* P = Z0 + m * VT_PLANE;
          return d4_dfv(ld(P, c - 2), ld(P, c - 1), ld(P, c + 1), ld(P, c + 2), r12d[0]);
        };
        auto gy = [&](int m) {
          const float2* P = Z0 + m * VT_PLANE;
          return d4_dfv(ld(P, c - 2 * VT_HX), ld(P, c - VT_HX), ld(P, c + VT_HX), ld(P, c + 2 * VT_HX), r12d[1]);
        };
        auto gz = [&](int m) {
          const int o = m * VT_PLANE + c;
          return d4_dfv(ld(Zm2, o), ld(Zm1, o), ld(Zp1, o), ld(Zp2, o), r12d[2]);
        };
        const df wx = df_add_fast(gy(2), df_neg(gz(1)));
        const df wy = df_add_fast(gz(0), df_neg(gx(2)));
        const df wz = df_add_fast(gx(1), df_neg(gy(0)));
        const df en = df_mul_u(rh2, df_add_pos_u(df_sqr_u(wx), df_add_pos_u(df_sqr_u(wy), df_sqr_u(wz))));
        sum[6] += f2d_bits(en.hi);
        add_lo(elo, en.lo);
        key_min(rmin, rho);
        key_min(pmin, pr);
        const df cs = df_sqrt(DFT ? load_df(pm + PM_T * N + p) : d2df_bits(__ldg(pm + PM_T * N + p)));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const df w = df_mul(df_add_pos(df_abs(vd[d]), cs), rhd[d]);
          if (df_lt(wmax, w)) wmax = w;
        }
      }
      __syncthreads();  // the slot of plane z - 2 takes plane z + 3 next
    }
  }
  // the block's fold: quantity q of every thread side by side in shared memory, then one warp each
  double* sh = reinterpret_cast<double*>(ring);  // [NRED][ST_THREADS]
  sum[5] += f2d_bits(klo.hi) + f2d_bits(klo.lo);
  sum[6] += f2d_bits(elo.hi) + f2d_bits(elo.lo);
#pragma unroll
  for (int m = 0; m < NSUM; ++m) sh[m * ST_THREADS + tid] = sum[m];
  sh[7 * ST_THREADS + tid] = __longlong_as_double(rmin ^ (long long)((unsigned long long)(rmin >> 63) >> 1));
  sh[8 * ST_THREADS + tid] = __longlong_as_double(pmin ^ (long long)((unsigned long long)(pmin >> 63) >> 1));
  sh[9 * ST_THREADS + tid] = f2d_bits(wmax.hi) + f2d_bits(wmax.lo);
  __syncthreads();
  for (int q = tid / 32; q < NRED; q += ST_THREADS / 32) {
    const double r = fold_column(q, sh + q * ST_THREADS, ST_THREADS, tid & 31);
    if ((tid & 31) == 0) partials[(long long)q * gridDim.x + blockIdx.x] = r;
  }
}

// partials [NRED][nblocks] of k_stats_tiled -> the statistics; one warp folds each quantity.
__global__ void __launch_bounds__(ST_FINAL_THREADS) k_stats_final(const double* __restrict__ partials, int nblocks,
                                                                  const int* __restrict__ status, double vol,
                                                                  double inv_n, double* __restrict__ out) {
  const int q = threadIdx.x / 32, lane = threadIdx.x & 31;
  const double r = fold_column(q, partials + (long long)q * nblocks, nblocks, lane);
  if (lane == 0) out[q] = (q < 5) ? r * vol : (q < NSUM) ? r * inv_n : r;
  if (threadIdx.x == 0) {
    out[10] = (double)(*status);
    out[11] = 0.0;
  }
}

}  // namespace

cudaError_t launch_prim(const Grid& g, const double* u, double* pm, double gamma, int* status, cudaStream_t s,
                        int df, long long p0, long long p1) {
  if (p1 < 0) p1 = g.N;
  if (p0 < 0 || p1 > g.N || p0 >= p1) return p0 == p1 ? cudaSuccess : cudaErrorInvalidValue;
  const int grid = grid_for(p1 - p0, PW_THREADS);
  if (df)
    k_prim<true><<<grid, PW_THREADS, 0, s>>>(u, pm, g.N, p0, p1, gamma, status);
  else
    k_prim<false><<<grid, PW_THREADS, 0, s>>>(u, pm, g.N, p0, p1, gamma, status);
  return cudaGetLastError();
}

// Planes per CTA of the tiled viscous kernels over nz planes of g, with `slots` CTAs resident at
// once: the chunk for which the rounds of resident CTAs times the planes a CTA walks (its chunk
// and 4 halo planes, which only load: counted half) are fewest, the longest of equals.  A fixed
// chunk of 16 left 32^3 with 8 CTAs of 20 serial planes, 64^3 with 64, and 128^3 with 512 CTAs on
// 456 slots, a second round for 56 of them.  Per launch (ncu): 32^3 43 -> 7 us, 64^3 44 -> 22 us,
// 128^3 115 -> 97 us, 256^3 685 -> 672 us.
static int visc_chunk(const Grid& g, int nz, int slots) {
  const long long nxy = (long long)((g.n[0] + VT_X - 1) / VT_X) * ((g.n[1] + VT_Y - 1) / VT_Y);
  long long best = -1;
  int chunk = 1;
  for (int cz = std::min(nz, 64); cz >= 1; --cz) {
    const long long ctas = nxy * ((nz + cz - 1) / cz);
    const long long cost = ((ctas + slots - 1) / slots) * (cz + 2);
    if (best < 0 || cost < best) {
      best = cost;
      chunk = cz;
    }
  }
  return chunk;
}

cudaError_t launch_visc(const Grid& g, const double* pm, double* fv, double mu, double kappa, cudaStream_t s,
                        int only_d, int df, int z0, int z1) {
  const double rx = g.r12h[0], ry = g.r12h[1], rz = g.r12h[2];
  const int nz = g.n[2];
  if (z1 < 0) z1 = nz;
  if (z0 < 0 || z1 > nz || z0 > z1) return cudaErrorInvalidValue;
  if (z0 == z1) return cudaSuccess;
  if (df) {
    const int cz = visc_chunk(g, z1 - z0, 3 * 152);
    const dim3 grid((g.n[0] + VT_X - 1) / VT_X, (g.n[1] + VT_Y - 1) / VT_Y, (z1 - z0 + cz - 1) / cz);
    k_visc_tiled<<<grid, VT_X * VT_Y, VT_SMEM, s>>>(pm, fv, g, mu, kappa, only_d, z0, z1, cz);
  } else {
    dim3 grid = plane_grid(g);
    grid.z = z1 - z0;
    k_visc<<<grid, PW_THREADS, 0, s>>>(pm, fv, g.n[0], g.n[1], nz, rx, ry, rz, mu, kappa, only_d, z0);
  }
  return cudaGetLastError();
}

cudaError_t prepare_visc_kernels() {
  cudaError_t e = cudaFuncSetAttribute(k_visc_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize, VT_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stats_tiled<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SR_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_stats_tiled<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SR_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_visc32t, cudaFuncAttributeMaxDynamicSharedMemorySize, V32_SMEM);
  return e;
}

cudaError_t launch_visc32(const Grid& g, const double* u, float* fv, double gamma, double mu, double kappa,
                          cudaStream_t s, int only_d) {
  const int cz = visc_chunk(g, g.n[2], 5 * 152);
  const dim3 grid((g.n[0] + VT_X - 1) / VT_X, (g.n[1] + VT_Y - 1) / VT_Y, (g.n[2] + cz - 1) / cz);
  k_visc32t<<<grid, VT_X * VT_Y, V32_SMEM, s>>>(u, fv, g, (float)gamma, (float)mu, (float)kappa, only_d, cz);
  return cudaGetLastError();
}

// Tiles of the statistics kernel: cz planes each, chosen so that the rounds of ST_SLOTS resident
// blocks times a tile's planes (cz to fold and 4 halo planes, which only load: counted half) are
// fewest.  256^3: 37 planes in 3 rounds where 16 take 7; small grids get short tiles (32^3: one
// plane) so that more SMs share the serial plane loop.
struct StatsPlan {
  int cz, ntx, nty, blocks;
  long long ntiles;
};
static StatsPlan stats_plan(const Grid& g) {
  StatsPlan p;
  p.ntx = (g.n[0] + VT_X - 1) / VT_X;
  p.nty = (g.n[1] + VT_Y - 1) / VT_Y;
  long long best = -1;
  for (int cz = std::min(g.n[2], 64); cz >= 1; --cz) {
    const long long tiles = (long long)p.ntx * p.nty * ((g.n[2] + cz - 1) / cz);
    const long long cost = ((tiles + ST_SLOTS - 1) / ST_SLOTS) * (cz + 2);
    if (best < 0 || cost < best) {
      best = cost;
      p.cz = cz;
      p.ntiles = tiles;
    }
  }
  p.blocks = (int)std::min<long long>(p.ntiles, ST_SLOTS);
  return p;
}

int stats_num_blocks(const Grid& g) { return stats_plan(g).blocks; }

cudaError_t launch_stats(const Grid& g, const double* u, const double* pm, double gamma, double* partials,
                         cudaStream_t s, int df) {
  (void)gamma;
  const StatsPlan p = stats_plan(g);
  if (df)
    k_stats_tiled<true><<<p.blocks, ST_THREADS, SR_SMEM, s>>>(u, pm, g, partials, p.ntx, p.nty, p.ntiles, p.cz);
  else
    k_stats_tiled<false><<<p.blocks, ST_THREADS, SR_SMEM, s>>>(u, pm, g, partials, p.ntx, p.nty, p.ntiles, p.cz);
  return cudaGetLastError();
}

cudaError_t launch_stats_final(const Grid& g, const double* partials, int nblocks, const int* status, double* out,
                               cudaStream_t s) {
  k_stats_final<<<1, ST_FINAL_THREADS, 0, s>>>(partials, nblocks, status, g.h[0] * g.h[1] * g.h[2],
                                               1.0 / (double)g.N, out);
  return cudaGetLastError();
}

}  // namespace ns3d
