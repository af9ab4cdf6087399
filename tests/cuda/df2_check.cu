// Test-only CUDA source (built by tests/test_gpu_df2.py, not part of libns3d.so): compares the
// two-lane double-float operations of df2.cuh with the scalar ones of df.cuh bit for bit, lane
// by lane, on pseudo-random inputs generated on the device.  The division and square root of
// df2.cuh take the error term of their last step from the exact product (fma form); their
// scalar references below are written out in that form.
#include <cuda_runtime.h>
#include <stdint.h>

#include "df.cuh"
#include "df2.cuh"
#include "k_dir_impl.cuh"

using namespace ns3d;

namespace {

constexpr int NOPS = 19;

__device__ uint64_t mix64(uint64_t z) {  // SplitMix64 finaliser
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// A double-float with |hi| in [2^-40, 2^20), a random sign unless pos, lo of a few ulp(hi) or less.
__device__ df rand_df(uint64_t key, bool pos) {
  const uint64_t r = mix64(key);
  const float m = 1.0f + (float)(r & 0xffffff) * 0x1p-24f;
  const int e = (int)((r >> 24) % 60) - 40;
  float hi = ldexpf(m, e);
  if (!pos && ((r >> 40) & 1)) hi = -hi;
  const float frac = ((float)((r >> 41) & 0xffff) * 0x1p-16f - 0.5f) * 0x1p-23f;
  return df{hi, hi * frac};
}

__device__ bool same(df a, df b) {
  return __float_as_uint(a.hi) == __float_as_uint(b.hi) && __float_as_uint(a.lo) == __float_as_uint(b.lo);
}

// scalar reference of df2_div (last step in the fma form)
__device__ df ref_div(df x, df y) {
  const float r = rcp_seed(y.hi);
  const float q1 = __fmul_rn(x.hi, r);
  const df p = two_prod(q1, y.hi);
  float rem = __fsub_rn(x.hi, p.hi);
  rem = __fsub_rn(rem, p.lo);
  rem = __fadd_rn(rem, x.lo);
  rem = __fmaf_rn(-q1, y.lo, rem);
  const float s = __fadd_rn(q1, __fmul_rn(rem, r));
  return df{s, __fmaf_rn(rem, r, -__fsub_rn(s, q1))};
}

// scalar references of df2_div_ru and df2_rcp_ru (unnormalised results)
__device__ df ref_div_ru(df x, df y) {
  float r = rcp_seed(y.hi);
  r = __fmaf_rn(r, __fmaf_rn(-y.hi, r, 1.0f), r);
  const float q1 = __fmul_rn(x.hi, r);
  const df p = two_prod(q1, y.hi);
  float rem = __fsub_rn(x.hi, p.hi);
  rem = __fsub_rn(rem, p.lo);
  rem = __fadd_rn(rem, x.lo);
  rem = __fmaf_rn(-q1, y.lo, rem);
  return df{q1, __fmul_rn(rem, r)};
}
__device__ df ref_rcp_ru(df y) {
  float r = rcp_seed(y.hi);
  r = __fmaf_rn(r, __fmaf_rn(-y.hi, r, 1.0f), r);
  const df p = two_prod(r, y.hi);
  const float rem = __fmaf_rn(-r, y.lo, __fsub_rn(__fsub_rn(1.0f, p.hi), p.lo));
  return df{r, __fmul_rn(rem, r)};
}

// scalar reference of df2_offset3 (the WENO5 offset of the direction pass)
__device__ df ref_offset3(bool scale, df B1, df B2, df B3, df ta6, df tb6) {
  if (scale) {
    const int e1 = exponent_of(B1.hi), e2 = exponent_of(B2.hi), e3 = exponent_of(B3.hi);
    const float sc = pow2f(-min(min(max(e1, max(e2, e3)), min(e1, min(e2, e3)) + 96), 126));
    df* B[3] = {&B1, &B2, &B3};
    for (int k = 0; k < 3; ++k) {
      *B[k] = df{B[k]->hi * sc, B[k]->lo * sc};
      if (B[k]->hi >= 2.0f) *B[k] = df{2.0f, 0.0f};
    }
  }
  const df b1 = df_mul_f_u(B1, 3.0f), b3 = df_twice(B3);
  const df den = df_add_pos_u(df_mul_u(B2, B3), df_mul_u(b1, df_add_pos_u(b3, B2)));
  const df num = df_mul(B2, df_add_fast(df_mul_u(b3, ta6), df_mul_u(b1, tb6)));
  return ref_div_ru(num, fast_two_sum(den.hi, den.lo));
}

// scalar reference of the squared indicators of phase B of the direction pass
__device__ void ref_indicators(df dgm, df dgp, df c133, df eps4, df& B1, df& B2, df& B3) {
  const df ds = df_add_fast(dgp, df_neg(dgm));
  const df s2 = df_sqr_u(ds);
  const df aa = df_add_pos_u(df_mul_u(s2, c133), eps4);
  const df u2 = df_add_fast(dgm, dgp);
  const df b2 = df_add_pos_u(df_sqr_u(u2), aa);
  const df pq = df_add_ordered_u(b2, df_twice(df_twice(s2)));
  const df r4 = df_twice(df_twice(df_mul_u(u2, ds)));
  B1 = df_sqr_u(df_add_ordered(pq, r4));
  B2 = df_sqr_u(b2);
  B3 = df_sqr_u(df_add_ordered(pq, df_neg(r4)));
}
__device__ void new_indicators(df2 dgm, df2 dgp, df2 c133, df2 eps4, df2& B1, df2& B2, df2& B3) {
  const df2 ds = df2_add_fast(dgp, df2_neg(dgm));
  const df2 s2 = df2_sqr_u(ds);
  const df2 aa = df2_add_pos_u(df2_mul_u(s2, c133), eps4);
  const df2 u2 = df2_add_fast(dgm, dgp);
  const df2 b2 = df2_add_pos_u(df2_sqr_u(u2), aa);
  const df2 pq = df2_add_ordered_u(b2, df2_twice(df2_twice(s2)));
  const df2 r4 = df2_twice(df2_twice(df2_mul_u(u2, ds)));
  B1 = df2_sqr_u(df2_add_ordered(pq, r4));
  B2 = df2_sqr_u(b2);
  B3 = df2_sqr_u(df2_add_ordered(pq, df2_neg(r4)));
}

__global__ void k_check(int n, uint64_t seed, int* bad) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  df a[2][6];
  for (int l = 0; l < 2; ++l)
    for (int j = 0; j < 6; ++j) a[l][j] = rand_df(seed + 12ull * (uint64_t)t + 6ull * l + j, j >= 2 && j <= 4);
  df2 p[6];
  for (int j = 0; j < 6; ++j) p[j] = df2_pack(a[0][j], a[1][j]);
  const df c133{4.3333335f, -3.9736431e-08f}, eps4{4e-06f, 1e-13f};
  df2 r2[NOPS];
  df r[2][NOPS];
  r2[0] = df2_add_fast(p[0], p[1]);
  r2[1] = df2_add_fast(p[0], df2_neg(p[1]));
  r2[2] = df2_mul_u(p[0], p[1]);
  r2[3] = df2_mul(p[0], p[1]);
  r2[4] = df2_sqr_u(p[0]);
  r2[5] = df2_mul_f_u(p[0], 6.0f);
  r2[6] = df2_add_pos_u(p[2], p[3]);
  r2[7] = df2_add_ordered_u(p[2], p[3]);
  r2[8] = df2_add_ordered(p[2], p[3]);
  r2[9] = df2_twice(p[1]);
  r2[10] = two_prod2(p[0].hi, p[1].hi);
  r2[11] = df2_div(p[0], p[2]);
  r2[12] = df2_offset3<false>(p[2], p[3], p[4], p[0], p[1]);
  new_indicators(p[0], p[1], df2_splat(c133), df2_splat(eps4), r2[13], r2[14], r2[15]);
  // the rescaled form: indicators of their own powers of two in [2^-90, 2^118), so that the lanes'
  // scales differ and about a third of the triples is cut
  df b[2][3];
  for (int l = 0; l < 2; ++l)
    for (int j = 0; j < 3; ++j) {
      const int e = (int)(mix64(~seed + 12ull * (uint64_t)t + 6ull * l + j) % 148) - 50;
      b[l][j] = df{ldexpf(a[l][2 + j].hi, e), ldexpf(a[l][2 + j].lo, e)};
    }
  r2[16] = df2_offset3<true>(df2_pack(b[0][0], b[1][0]), df2_pack(b[0][1], b[1][1]), df2_pack(b[0][2], b[1][2]), p[0],
                             p[1]);
  r2[17] = df2_div_ru(p[0], p[2]);
  r2[18] = df2_rcp_ru(p[2]);
  for (int l = 0; l < 2; ++l) {
    const df* x = a[l];
    r[l][0] = df_add_fast(x[0], x[1]);
    r[l][1] = df_add_fast(x[0], df_neg(x[1]));
    r[l][2] = df_mul_u(x[0], x[1]);
    r[l][3] = df_mul(x[0], x[1]);
    r[l][4] = df_sqr_u(x[0]);
    r[l][5] = df_mul_f_u(x[0], 6.0f);
    r[l][6] = df_add_pos_u(x[2], x[3]);
    r[l][7] = df_add_ordered_u(x[2], x[3]);
    r[l][8] = df_add_ordered(x[2], x[3]);
    r[l][9] = df_twice(x[1]);
    r[l][10] = two_prod(x[0].hi, x[1].hi);
    r[l][11] = ref_div(x[0], x[2]);
    r[l][12] = ref_offset3(false, x[2], x[3], x[4], x[0], x[1]);
    ref_indicators(x[0], x[1], c133, eps4, r[l][13], r[l][14], r[l][15]);
    r[l][16] = ref_offset3(true, b[l][0], b[l][1], b[l][2], x[0], x[1]);
    r[l][17] = ref_div_ru(x[0], x[2]);
    r[l][18] = ref_rcp_ru(x[2]);
  }
  for (int o = 0; o < NOPS; ++o)
    if (!same(df2_lane0(r2[o]), r[0][o]) || !same(df2_lane1(r2[o]), r[1][o])) atomicAdd(&bad[o], 1);
}

// Relative errors of the divisions and square roots on normalised random operands, against FP64, in
// units of 2^-48: the largest (1e-3 units) and the sum (for the mean) of df_div, df2_div, df_div_r,
// df2_div_ru, df2_rcp_ru, df_sqrt, df_sqrt_r.
constexpr int NERR = 7;
__global__ void k_check_errors(int n, uint64_t seed, int* emax, double* esum) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  auto norm = [](df x) { return fast_two_sum(x.hi, x.lo); };
  const df x = norm(rand_df(seed + 2ull * (uint64_t)t, false)), y = norm(rand_df(seed + 2ull * (uint64_t)t + 1, true));
  auto val = [](df q) { return (double)q.hi + (double)q.lo; };
  auto lane = [](df2 q) { return df2_lane1(q); };
  const df2 x2 = df2_splat(x), y2 = df2_splat(y);
  const double vx = val(x), vy = val(y);
  const df got[NERR] = {df_div(x, y), lane(df2_div(x2, y2)), df_div_r(x, y), lane(df2_div_ru(x2, y2)),
                        lane(df2_rcp_ru(y2)), df_sqrt(y), df_sqrt_r(y)};
  const double ref[NERR] = {vx / vy, vx / vy, vx / vy, vx / vy, 1.0 / vy, sqrt(vy), sqrt(vy)};
  for (int o = 0; o < NERR; ++o) {
    const double e = fabs(val(got[o]) / ref[o] - 1.0) * 0x1p48;
    atomicMax(&emax[o], e < 1e6 ? (int)(e * 1e3) : 1000000000);
    atomicAdd(&esum[o], e);
  }
}

// rcp_cubic (what = 0) and rsqrt_cubic (1) at the positive doubles of biased exponent
// e11 = blockIdx.x and a pseudo-random mantissa per thread (thread 0: zero, so 0, powers of two and
// infinity; thread 1: all ones): where both operand and IEEE result are normal, the error in ulps of
// the result into *ulp (as an integer of 1e-6 ulp); elsewhere the bits of the IEEE operations, counted
// in *bad where they differ.
__global__ void k_check_cubic(int what, uint64_t seed, int* ulp, int* bad) {
  const uint64_t key = seed + blockIdx.x * 4096ull + threadIdx.x;
  const uint64_t m = threadIdx.x == 0 ? 0 : threadIdx.x == 1 ? 0xfffffffffffffull : mix64(key) >> 12;
  const double x = __longlong_as_double(((long long)blockIdx.x << 52) | (long long)m);
  const double r = what ? rsqrt_cubic(x) : rcp_cubic(x);
  const double ref = what ? 1.0 / sqrt(x) : 1.0 / x;
  const int er = (int)((__double_as_longlong(ref) >> 52) & 0x7ff);
  if (blockIdx.x == 0 || blockIdx.x == 0x7ff || er == 0 || er == 0x7ff) {
    if (!(r == ref || (isnan(r) && isnan(ref)))) atomicAdd(bad, 1);
    return;
  }
  // relative error: 1 - x r exactly; (1 - x r^2)/2 with x r as a sum of two doubles
  const double p = x * r, pe = fma(x, r, -p);
  const double rel = what ? 0.5 * fma(-pe, r, fma(-p, r, 1.0)) : fma(-x, r, 1.0);
  const double mant = __longlong_as_double((__double_as_longlong(ref) & 0xfffffffffffffll) | (1023ll << 52));
  const double err = fabs(rel) * mant * 0x1p52 * 1e6;
  if (!(err < 2e9)) atomicAdd(bad, 1);
  else atomicMax(ulp, (int)err);
}

}  // namespace

// Runs n lane pairs; bad_host receives NOPS mismatch counts (add_fast, sub, mul_u, mul, sqr_u,
// mul_f_u, add_pos_u, add_ordered_u, add_ordered, twice, two_prod, div, offset, indicator
// B1, B2, B3, rescaled offset, div_ru, rcp_ru).  Returns a cudaError_t.
extern "C" int df2_check(int n, unsigned long long seed, int* bad_host) {
  int* bad = nullptr;
  cudaError_t e = cudaMalloc(&bad, sizeof(int) * NOPS);
  if (e != cudaSuccess) return (int)e;
  cudaMemset(bad, 0, sizeof(int) * NOPS);
  k_check<<<(n + 255) / 256, 256>>>(n, seed, bad);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(bad_host, bad, sizeof(int) * NOPS, cudaMemcpyDeviceToHost);
  cudaFree(bad);
  return (int)e;
}

extern "C" int df2_check_nops() { return NOPS; }

// Largest error (1e-6 ulp) of rcp_cubic (what = 0) or rsqrt_cubic (1) over all exponents, and the number
// of wrong special values.  Returns a cudaError_t.
extern "C" int cubic_check(int what, unsigned long long seed, int* ulp_host, int* bad_host) {
  int* d = nullptr;
  cudaError_t e = cudaMalloc(&d, 2 * sizeof(int));
  if (e != cudaSuccess) return (int)e;
  cudaMemset(d, 0, 2 * sizeof(int));
  k_check_cubic<<<2048, 1024>>>(what, seed, d, d + 1);
  e = cudaGetLastError();
  int h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  *ulp_host = h[0];
  *bad_host = h[1];
  return (int)e;
}

// Largest and mean relative error (units of 2^-48) of the operations of k_check_errors over n operand
// pairs: NERR doubles each.  Returns a cudaError_t.
extern "C" int error_check(int n, unsigned long long seed, double* max_host, double* mean_host) {
  double* d = nullptr;  // NERR sums, then NERR ints
  cudaError_t e = cudaMalloc(&d, 2 * NERR * sizeof(double));
  if (e != cudaSuccess) return (int)e;
  cudaMemset(d, 0, 2 * NERR * sizeof(double));
  int* m = reinterpret_cast<int*>(d + NERR);
  k_check_errors<<<(n + 255) / 256, 256>>>(n, seed, m, d);
  e = cudaGetLastError();
  double sum[NERR];
  int mx[NERR];
  if (e == cudaSuccess) e = cudaMemcpy(sum, d, sizeof(sum), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(mx, m, sizeof(mx), cudaMemcpyDeviceToHost);
  cudaFree(d);
  for (int o = 0; o < NERR && e == cudaSuccess; ++o) {
    max_host[o] = mx[o] * 1e-3;
    mean_host[o] = sum[o] / n;
  }
  return (int)e;
}

extern "C" int error_check_nops() { return NERR; }
