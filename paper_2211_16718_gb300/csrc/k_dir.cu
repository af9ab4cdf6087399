// Standalone launches of the fused direction pass (one tile per CTA); the tile
// computation itself is dir_tile in k_dir_impl.cuh.  Tile shapes (points along the
// pencil, at most, x lines; the pencil is cut into tiles of equal length) are template variants: a context uses the one set by
// ns3d_set_variant (default 0); an ensemble's autotuner picks one per grid size.
//   MODE 0 (all FP64):              32 x 4
//   MODE 1 (FP64 + double-float):   variant 0: 24 x 4, 1: 16 x 4, 2: 40 x 2
// All variants compute bitwise identical results (the per-interface arithmetic
// does not depend on the tiling).
#include "k_dir_impl.cuh"

namespace ns3d {

namespace {

template <int D, int MODE, int TP, int W>
__global__ void __launch_bounds__(Plan<MODE, TP, W>::THREADS, Plan<MODE, TP, W>::MIN_CTAS) k_dir(const DirArgs a) {
  extern __shared__ __align__(16) double sm[];
  const bool swap = (D == 2 && a.zorder);
  const int tile = (swap ? blockIdx.y : blockIdx.x) + (D == 2 ? a.t0 : 0);
  int s0, len;
  tile_span(D, a.g.n[D], a.tile_u, a.tile_r, tile, s0, len);
  dir_tile<D, MODE, TP, W>(a, sm, s0, len, swap ? blockIdx.x : blockIdx.y, blockIdx.z + (D == 2 ? 0 : a.t0));
}

// The x pass (blocks below nbx) and the y pass side by side in one launch: neither reads what the
// other writes.  It fills the second pass's launch gap and the last, partly filled round of CTAs:
// 40x25x18 right-hand side 34.8 -> 30.2 us, 32^3 RK4 step 240 -> 215 us, 64^3 passes 115 -> 112 us,
// 96^3 all-FP64 step 8.97 -> 8.91 ms, but 128^3 passes 805 -> 816 us (why was not measured), so only
// grids of up to 2^20 points (dir_xy_merged).
template <int MODE, int TP, int W>
__global__ void __launch_bounds__(Plan<MODE, TP, W>::THREADS, Plan<MODE, TP, W>::MIN_CTAS) k_dir_xy(const DirArgs ax,
                                                                                                const DirArgs ay,
                                                                                                int nbx) {
  extern __shared__ __align__(16) double sm[];
  int s0, len;
  if ((int)blockIdx.x < nbx) {
    const int nt = (ax.g.n[0] + TP - 1) / TP, nl = (ax.g.n[1] + W - 1) / W;
    const int r = blockIdx.x / nt, bz = r / nl;
    tile_span(0, ax.g.n[0], ax.tile_u, ax.tile_r, blockIdx.x - r * nt, s0, len);
    dir_tile<0, MODE, TP, W>(ax, sm, s0, len, r - bz * nl, bz);
  } else {
    const int b = blockIdx.x - nbx;
    const int nt = (ay.g.n[1] + TP - 1) / TP, nl = (ay.g.n[0] + W - 1) / W;
    const int r = b / nt, bz = r / nl;
    tile_span(1, ay.g.n[1], ay.tile_u, ay.tile_r, b - r * nt, s0, len);
    dir_tile<1, MODE, TP, W>(ay, sm, s0, len, r - bz * nl, bz);
  }
}

template <int MODE, int TP, int W>
cudaError_t launch_xy(const DirArgs& a, double* k2, cudaStream_t s) {
  using PL = Plan<MODE, TP, W>;
  const int* n = a.g.n;
  const int nx = (n[0] + TP - 1) / TP, ny = (n[1] + TP - 1) / TP;
  const long long nbx = (long long)nx * ((n[1] + W - 1) / W) * n[2], nby = (long long)ny * ((n[0] + W - 1) / W) * n[2];
  if (nbx + nby > 0x7fffffffLL) return cudaErrorInvalidValue;
  DirArgs x = a, y = a;
  x.epi = y.epi = EPI_ACC_WRITE;
  x.t0 = y.t0 = 0;
  y.k = k2;
  tile_split_units(0, n[0], nx, x.tile_u, x.tile_r);
  tile_split_units(1, n[1], ny, y.tile_u, y.tile_r);
  k_dir_xy<MODE, TP, W><<<(unsigned)(nbx + nby), PL::THREADS, PL::BYTES, s>>>(x, y, (int)nbx);
  return cudaGetLastError();
}

// Tiles [lo, hi) along the range axis (hi < 0: all): the tiles along z for D = 2 (blockIdx.x, or
// blockIdx.y with a.zorder), blockIdx.z (planes z) for D = 0, 1.
template <int D, int MODE, int TP, int W>
cudaError_t launch_t(const DirArgs& a, cudaStream_t s, int lo = 0, int hi = -1) {
  using PL = Plan<MODE, TP, W>;
  constexpr int AX = (D == 0) ? 1 : 0;
  constexpr int BX = (D == 2) ? 1 : 2;
  dim3 grid((a.g.n[D] + TP - 1) / TP, (a.g.n[AX] + W - 1) / W, a.g.n[BX]);
  if (D == 2 && a.zorder) {
    const unsigned t = grid.x;
    grid.x = grid.y;
    grid.y = t;
  }
  unsigned& ext = (D == 2) ? (a.zorder ? grid.y : grid.x) : grid.z;
  if (hi < 0) hi = (int)ext;
  if (lo < 0 || hi > (int)ext || lo > hi) return cudaErrorInvalidValue;
  if (lo == hi) return cudaSuccess;
  ext = (unsigned)(hi - lo);
  DirArgs r = a;
  r.t0 = lo;
  tile_split_units(D, a.g.n[D], (a.g.n[D] + TP - 1) / TP, r.tile_u, r.tile_r);
  k_dir<D, MODE, TP, W><<<grid, PL::THREADS, PL::BYTES, s>>>(r);
  return cudaGetLastError();
}

// Dynamic shared memory of the tile plan, and the largest shared-memory carveout so that
// Plan::MIN_CTAS tiles fit on an SM (the rest of the unified L1 stays cache).
template <typename K>
cudaError_t set_func_attr(K* kernel, int bytes) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

template <int MODE, int TP, int W>
cudaError_t set_attr() {
  const int bytes = Plan<MODE, TP, W>::BYTES;
  cudaError_t e = set_func_attr(k_dir<0, MODE, TP, W>, bytes);
  if (e == cudaSuccess) e = set_func_attr(k_dir<1, MODE, TP, W>, bytes);
  if (e == cudaSuccess) e = set_func_attr(k_dir<2, MODE, TP, W>, bytes);
  if (e == cudaSuccess) e = set_func_attr(k_dir_xy<MODE, TP, W>, bytes);
  return e;
}

template <int MODE, int TP, int W>
cudaError_t launch_dirs(int d, const DirArgs& a, cudaStream_t s, int lo = 0, int hi = -1) {
  switch (d) {
    case 0: return launch_t<0, MODE, TP, W>(a, s, lo, hi);
    case 1: return launch_t<1, MODE, TP, W>(a, s, lo, hi);
    default: return launch_t<2, MODE, TP, W>(a, s, lo, hi);
  }
}

}  // namespace

cudaError_t prepare_dir_kernels() {
  cudaError_t e = set_attr<0, 32, 4>();
  if (e == cudaSuccess) e = set_attr<1, 24, 4>();
  if (e == cudaSuccess) e = set_attr<1, 16, 4>();
  if (e == cudaSuccess) e = set_attr<1, 40, 2>();
  if (e == cudaSuccess) e = prepare_dir32_kernels();
  if (e == cudaSuccess) e = prepare_visc_kernels();
  return e;
}

// With the tiles along z fastest, the CTAs resident at one time cover every z-plane of a few
// line groups, i.e. one 32-byte piece of each of ~30 planes of ~30 arrays per tile.  On a 1024^3
// grid (8 MB between planes) that z pass took 2.8x the time of the x pass; walking the line
// groups of one z-tile row first (CTAs resident at once within a few tile rows) brought it to
// 1.26x.  On 256^3 the tiles-along-z order is 0.5 % faster overall, so the switch is by size:
// line groups first from 2^28 points (2 GB per array) up.
int dir_zorder(const Grid& g) { return g.N >= (1LL << 28) ? 1 : 0; }

void dir_tile_shape(int mode, int variant, int* tp, int* w) {
  if (mode == 0) {
    *tp = 32;
    *w = 4;
  } else if (mode == 1 && variant == 1) {
    *tp = 16;
    *w = 4;
  } else if (mode == 1 && variant == 2) {
    *tp = 40;
    *w = 2;
  } else if (mode == 1) {
    *tp = 24;
    *w = 4;
  } else {  // FP32 bulk
    *tp = 32;
    *w = 4;
  }
}

int dir_tile_start(const Grid& g, int d, int mode, int variant, int t) {
  int tp = 0, w = 0, u = 0, r = 0, s0 = 0, len = 0;
  dir_tile_shape(mode, variant, &tp, &w);
  const int nt = (g.n[d] + tp - 1) / tp;
  if (t >= nt) return g.n[d];
  tile_split_units(d, g.n[d], nt, u, r);
  tile_span(d, g.n[d], u, r, t, s0, len);
  return s0;
}

cudaError_t launch_dir(int d, const DirArgs& a, cudaStream_t s) {
  if (a.mode == 2) return launch_dir32(d, a, s);
  return launch_dir_range(d, a, s, 0, -1);
}

cudaError_t launch_dir_xy(const DirArgs& a, double* k2, cudaStream_t s) {
  if (a.mode == 2 || (a.fv != nullptr && a.fv_dstride == 0)) return cudaErrorInvalidValue;
  if (a.mode == 0) return launch_xy<0, 32, 4>(a, k2, s);
  switch (a.variant) {
    case 1: return launch_xy<1, 16, 4>(a, k2, s);
    case 2: return launch_xy<1, 40, 2>(a, k2, s);
    default: return launch_xy<1, 24, 4>(a, k2, s);
  }
}

cudaError_t launch_dir_range(int d, const DirArgs& a, cudaStream_t s, int lo, int hi) {
  if (a.mode == 2) return cudaErrorInvalidValue;
  if (a.mode == 0) return launch_dirs<0, 32, 4>(d, a, s, lo, hi);
  switch (a.variant) {
    case 1: return launch_dirs<1, 16, 4>(d, a, s, lo, hi);
    case 2: return launch_dirs<1, 40, 2>(d, a, s, lo, hi);
    default: return launch_dirs<1, 24, 4>(d, a, s, lo, hi);
  }
}

}  // namespace ns3d
