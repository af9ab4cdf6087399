// Pieces shared by the direction passes (k_dir.cu: FP64 modes, k_dir32.cu:
// FP32-bulk mode): tile indexing and the accumulation / Runge-Kutta epilogue.
#pragma once

#include "ns3d_internal.cuh"

namespace ns3d {

// Shared-memory index of (position along the pencil, line) in a tile of W lines:
// position-major for y/z lines (consecutive threads = consecutive x lines),
// line-major for x lines (consecutive threads = consecutive x points).
template <int D, int W>
__device__ __forceinline__ int tile_idx(int pos, int line, int npos) {
  return D == 0 ? line * npos + pos : pos * W + line;
}
template <int D, int W>
__device__ __forceinline__ void tile_split(int item, int npos, int& pos, int& line) {
  if (D == 0) {
    pos = item % npos;
    line = item / npos;
  } else {
    line = item % W;
    pos = item / W;
  }
}

// ---- balanced tiles -----------------------------------------------------------------
// A pencil of n points is cut into nt = ceil(n / TP) tiles of nearly equal length (at most TP)
// instead of full tiles and a remainder, and a tile computes no more than its own points and
// halo.  Lengths are whole units of points: 4 along x, so that the tiles' rows start on 32-byte
// sectors, 1 along y and z.  Tile t covers tile_unit * [t u + min(t, r), ...) with
// u = units / nt, r = units % nt (the first r tiles are one unit longer).
__host__ __device__ constexpr int tile_unit(int d) { return d == 0 ? 4 : 1; }
__host__ __device__ __forceinline__ void tile_split_units(int d, int n, int nt, int& u, int& r) {
  const int units = (n + tile_unit(d) - 1) / tile_unit(d);
  u = units / nt;
  r = units - u * nt;
}
// First point and number of points of tile t.
__host__ __device__ __forceinline__ void tile_span(int d, int n, int u, int r, int t, int& s0, int& len) {
  s0 = tile_unit(d) * (t * u + (t < r ? t : r));
  const int end = s0 + tile_unit(d) * (u + (t < r ? 1 : 0));
  len = (end < n ? end : n) - s0;
}

// ceil(2^20 / d): i / d = (i * c_rcp20[d]) >> 20 for the item numbers of a tile (i d < 2^20, and the
// product below 2^32), d a run-time extent of the tile.
struct Rcp20 {
  unsigned v[64];
  constexpr Rcp20() : v() {
    for (unsigned d = 1; d < 64; ++d) v[d] = ((1u << 20) + d - 1) / d;
  }
};
static __constant__ const Rcp20 c_rcp20 = Rcp20();

// Item numbers of a phase over (scalar m, position < npos, line < W): the order of tile_idx with the
// run-time extent npos (rcp = c_rcp20.v[npos]).
template <int D, int W>
__device__ __forceinline__ void item_split(int item, int npos, unsigned rcp, int& m, int& pos, int& line) {
  if (D == 0) {
    const int ml = (int)(((unsigned)item * rcp) >> 20);
    pos = item - ml * npos;
    m = ml / W;
    line = ml % W;
  } else {
    const int mp = item / W;
    line = item % W;
    m = (int)(((unsigned)mp * rcp) >> 20);
    pos = mp - m * npos;
  }
}
// The same without the scalar.
template <int D, int W>
__device__ __forceinline__ void item_split(int item, int npos, unsigned rcp, int& pos, int& line) {
  if (D == 0) {
    line = (int)(((unsigned)item * rcp) >> 20);
    pos = item - line * npos;
  } else {
    line = item % W;
    pos = item / W;
  }
}

// Flat grid index of pencil coordinate c on line la of the tile row bz.
template <int D>
__device__ __forceinline__ long long tile_flat(const Grid& g, int c, int la, int bz) {
  constexpr int AX = (D == 0) ? 1 : 0;
  constexpr int BX = (D == 2) ? 1 : 2;
  int idx[3];
  idx[D] = c;
  idx[AX] = la;
  idx[BX] = bz;
  return ((long long)idx[2] * g.n[1] + idx[1]) * g.n[0] + idx[0];
}

// Number of FP64 operands per point the epilogue reads (k, then U_n, then acc or the stage input).
__host__ __device__ __forceinline__ int epilogue_operands(int epi) {
  switch (epi) {
    case EPI_ACC_WRITE: return 0;
    case EPI_ACC_ADD:
    case EPI_RHS_OUT: return 5;
    case EPI_RK4_FIRST:
    case EPI_SSP_1: return 10;
    default: return 15;
  }
}

// Asynchronous 8-byte global -> shared copy (cp.async, cached at all levels).
__device__ __forceinline__ void cp_async8(double* dst_smem, const double* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned), L2 only.
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
// One double (PAIR false), or two adjacent ones from 16-byte aligned addresses.
template <bool PAIR>
__device__ __forceinline__ void cp_async_d(double* dst_smem, const double* src) {
  if (PAIR) cp_async16(dst_smem, src);
  else cp_async8(dst_smem, src);
}

// Start fetching the epilogue operands of point p (PAIR: of p and p + 1) into pre[v * TS],
// v < epilogue_operands(a.epi), and the y contribution, if it is apart, into v = 15 .. 19.
template <bool PAIR, int TS>
__device__ __forceinline__ void epilogue_prefetch(const DirArgs& a, long long p, double* pre) {
  const long long N = a.g.N;
  const int n = epilogue_operands(a.epi);
  if (n == 0) return;
#pragma unroll
  for (int v = 0; v < 5; ++v) cp_async_d<PAIR>(pre + v * TS, a.k + v * N + p);
  if (n >= 10) {
#pragma unroll
    for (int v = 0; v < 5; ++v) cp_async_d<PAIR>(pre + (5 + v) * TS, a.un + v * N + p);
  }
  if (n == 15) {
    const double* third = (a.epi == EPI_SSP_2 || a.epi == EPI_SSP_3) ? a.u : a.acc;
#pragma unroll
    for (int v = 0; v < 5; ++v) cp_async_d<PAIR>(pre + (10 + v) * TS, third + v * N + p);
  }
  if (a.k2 != nullptr) {
#pragma unroll
    for (int v = 0; v < 5; ++v) cp_async_d<PAIR>(pre + (15 + v) * TS, a.k2 + v * N + p);
  }
}

// Accumulate this direction's contribution cv[5] at point p, or finish the RHS / RK stage (last
// direction), according to a.epi; the operands in pre[v * TS] (filled by epilogue_prefetch).
template <int TS>
__device__ __forceinline__ void dir_epilogue_pre(const DirArgs& a, long long p, const double cv[5],
                                                 const double* pre) {
  const long long N = a.g.N;
  auto kxy = [&](int v) { return a.k2 != nullptr ? pre[v * TS] + pre[(15 + v) * TS] : pre[v * TS]; };
  switch (a.epi) {
    case EPI_ACC_WRITE:
#pragma unroll
      for (int v = 0; v < 5; ++v) a.k[v * N + p] = cv[v];
      break;
    case EPI_ACC_ADD:
#pragma unroll
      for (int v = 0; v < 5; ++v) a.k[v * N + p] = pre[v * TS] + cv[v];
      break;
    case EPI_RHS_OUT:
#pragma unroll
      for (int v = 0; v < 5; ++v) a.out[v * N + p] = kxy(v) + cv[v];
      break;
    case EPI_RK4_FIRST:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = fma(a.a, K, pre[(5 + v) * TS]);
        a.acc[v * N + p] = K;
      }
      break;
    case EPI_RK4_MID:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = fma(a.a, K, pre[(5 + v) * TS]);
        a.acc[v * N + p] = fma(2.0, K, pre[(10 + v) * TS]);
      }
      break;
    case EPI_RK4_LAST:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = fma(a.a, pre[(10 + v) * TS] + K, pre[(5 + v) * TS]);
      }
      break;
    case EPI_SSP_1:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = fma(a.a, K, pre[(5 + v) * TS]);
      }
      break;
    case EPI_SSP_2:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = 0.75 * pre[(5 + v) * TS] + 0.25 * fma(a.a, K, pre[(10 + v) * TS]);
      }
      break;
    case EPI_SSP_3:
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double K = kxy(v) + cv[v];
        a.out[v * N + p] = (1.0 / 3.0) * pre[(5 + v) * TS] + (2.0 / 3.0) * fma(a.a, K, pre[(10 + v) * TS]);
      }
      break;
    default:
      break;
  }
}

}  // namespace ns3d
