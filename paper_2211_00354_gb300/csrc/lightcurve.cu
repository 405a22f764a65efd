// lightcurve.cu -- Gaussian-source light curve as a ray sum and its gradient
// with respect to the mapped rays.  A source of profile
// G(s) = exp(-|s|^2 / (2 sigma^2)) / (2 pi sigma^2) (the Gaussian source of
// Sec. 2.5) centred at s_k has magnification F_k = sum_r w_ray G(y_r - s_k)
// when every ray carries the image-plane area w_ray; sampling s_k along a
// track gives a light curve (Sec. 3.3).  Pairs with |y_r - s_k| > trunc sigma
// are left out.  L = sum_k (F_k - T_k)^2 gives
//   dL/dy_r = sum_k 2 (F_k - T_k) w_ray G(y_r - s_k) (-(y_r - s_k) / sigma^2).
// Samples are bucketed on a uniform grid of cell >= trunc*sigma, the rays near
// them on the same grid (one cell wider), each cell in up to 4 x 4 parts.  The
// forward pass gives each sample a block that sums over the rays of the parts
// its cut reaches (no atomics); the gradient gives each of these rays, in the
// order of the parts, a thread that sums over the samples of the 3 x 3 cells
// around it, the samples stored in cell order with their coefficients.  A pair's difference, cut test, Gaussian and sums
// are float-float (pairs of float32, ~48 bits) on the float32 pipe -- GB300's
// float64 pipe is 1/74 of float32 -- and a plain float32 test with a margin
// for its rounding skips the pairs clearly beyond the cut.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "cx.cuh"
#include "lens_internal.h"

namespace lens {
namespace {

constexpr int kLcThreads = 256;

// exp(x), x <= 0, in float-float by the table-driven method of Tang ("Table-
// driven implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15(2), 1989): x = (64 m + j) ln2/64 + r with
// |r| <= ln2/128, exp(x) = 2^m 2^(j/64) exp(r); 2^(j/64) from a float-float
// table, exp(r) from its Taylor series, 1 + r + r^2/2 in float-float and the
// terms from r^3/6 (< 3e-8) on in float32.  ln2/64 is split as L1 + L2 + L3,
// L1 with 11 significant bits, so that k L1 is exact for |k| < 2^13.  Below
// x = -87 (2^m under the float32 normal range) the result is 0.
struct ExpTab {
  float thi[64], tlo[64];  // 2^(j/64)
  float l1, l2, l3;        // ln2/64
};
// The table in shared memory: the lanes of a warp read different entries, which
// the constant bank of the kernel's arguments would serve one by one.
struct ExpShared {
  const float2* t;
  float l1, l2, l3;
};
__device__ __forceinline__ ExpShared stage_exp(const ExpTab& T, float2* sh) {
  for (int j = threadIdx.x; j < 64; j += blockDim.x) sh[j] = make_float2(T.thi[j], T.tlo[j]);
  __syncthreads();
  return ExpShared{sh, T.l1, T.l2, T.l3};
}

ExpTab make_exp_tab() {
  ExpTab t{};
  for (int j = 0; j < 64; ++j) {
    const double v = std::exp2(j / 64.0);
    t.thi[j] = (float)v;
    t.tlo[j] = (float)(v - (double)t.thi[j]);
  }
  const double L = std::log(2.0) / 64.0;
  const double l1 = std::ldexp(std::nearbyint(std::ldexp(L, 17)), -17);  // 11 bits
  t.l1 = (float)l1;
  t.l2 = (float)(L - l1);
  t.l3 = (float)(L - l1 - (double)t.l2);
  return t;
}

__device__ __forceinline__ ff ff_exp_neg(ff x, const ExpShared& T) {
  if (!(x.hi > -87.0f)) return ff{0.f, 0.f};
  const float kf = rintf(x.hi * 92.33248261689366f);  // 64 / ln2
  const int k = (int)kf;
  const int m = k >> 6, j = k - (m << 6);
  // r = x - k ln2/64: x.hi - k L1 is exact (Sterbenz), -k L2 an exact product
  const float a = fmaf(-kf, T.l1, x.hi);
  const float p = -kf * T.l2;
  const float pe = fmaf(-kf, T.l2, -p);
  float s, e;
  two_sum(a, p, s, e);
  e += pe + x.lo - kf * T.l3;
  const ff r = ff_norm(s, e);
  // 1 + r + r^2/2 + r^3/6 + ... + r^6/720: the heads of the first three terms,
  // each below the sum so far, by two fast two-sums, everything else (< 2^-24) in
  // float32
  const float r2h = r.hi * r.hi;
  const float r2l = fmaf(r.hi, r.hi, -r2h) + 2.f * r.hi * r.lo;
  const float tail =
      r2h * r.hi * fmaf(r.hi, fmaf(r.hi, fmaf(r.hi, 1.f / 720.f, 1.f / 120.f), 1.f / 24.f), 1.f / 6.f);
  const float h1 = 1.f + r.hi, e1 = r.hi - (h1 - 1.f);
  const float q2 = 0.5f * r2h;
  const float h2 = h1 + q2, e2 = q2 - (h2 - h1);
  ff E = ff_norm(h2, (e1 + e2) + (fmaf(0.5f, r2l, r.lo) + tail));
  const float2 t2 = T.t[j];
  E = ff_mul(E, ff{t2.x, t2.y});
  const float sc = __int_as_float((127 + m) << 23);  // 2^m, m >= -126
  return ff{E.hi * sc, E.lo * sc};
}

__device__ __forceinline__ bool ff_gt(ff a, ff b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }

// Positions are kept as a cell of the sample grid (a side of three significant
// bits, origin a multiple of it) and the offset from that cell's origin, exact in float64
// (|offset| < 2 cells) and then float-float: the difference of two points is
// (a - b) + (cell_a - cell_b) * side, to ~2^-48 of a cell whatever the
// coordinates' size.
struct Pos {
  float4 o;  // offset: x hi, x lo, y hi, y lo
  int2 c;    // cell
};
// An offset moved by whole cells, |hi + shift| < 2 cells: exact, the head's error kept
// apart (in the tail it would be the same rounding for every pair of the point).
struct Shifted {
  float hi, lo, mid;
};
__device__ __forceinline__ Shifted shifted(float hi, float lo, float shift) {
  Shifted r;
  two_sum(hi, shift, r.hi, r.mid);
  r.lo = lo;
  return r;
}
// a - b, and (a + mid) - b
__device__ __forceinline__ ff minus(float ahi, float alo, float bhi, float blo, float mid) {
  float s, e;
  two_sum(ahi, -bhi, s, e);
  return ff_norm(s, e + ((alo - blo) + mid));
}
__device__ __forceinline__ Pos make_pos(double x, double y, int cx, int cy, double x0, double y0,
                                        double side) {
  const ff a = ff_of(x - (x0 + cx * side)), b = ff_of(y - (y0 + cy * side));
  return Pos{make_float4(a.hi, a.lo, b.hi, b.lo), make_int2(cx, cy)};
}

// The Gaussian of a pair, G = exp(-|d|^2 / (2 sigma^2)) with d = a - b (two points
// in one cell's frame), in float-float; false beyond the cut (q = |d|^2 > cut2).
// A float32 test first: the heads are within 2^-23 of 2 cells of the truth,
// so a margin of 2^-21 cells (in near2, the square of the widened cut)
// covers their rounding and that of d and q; it rejects only pairs surely
// beyond the cut.
struct Cut {
  ff ninv2s2, cut2;
  float near2;
};
__device__ __forceinline__ float near_cut2(float cutf, float side) {
  const float c = cutf * 1.00001f + 4.8e-7f * side;
  return c * c;
}
__device__ __forceinline__ ff sq(ff d) {  // normalised
  const float p = d.hi * d.hi;
  return ff{p, fmaf(d.hi + d.hi, d.lo, fmaf(d.hi, d.hi, -p))};
}
// a and b: offsets (x hi, x lo, y hi, y lo); mid1, mid2: what their heads leave out
__device__ __forceinline__ bool pair_gauss(float4 a, float4 b, float mid1, float mid2, const Cut& C,
                                           const ExpShared& T, ff& d1, ff& d2, ff& G) {
  const float e1 = a.x - b.x, e2 = a.z - b.z;
  if (fmaf(e1, e1, e2 * e2) > C.near2) return false;
  d1 = minus(a.x, a.y, b.x, b.y, mid1);
  d2 = minus(a.z, a.w, b.z, b.w, mid2);
  const ff q1 = sq(d1), q2 = sq(d2);
  float s, e;
  two_sum(q1.hi, q2.hi, s, e);
  const ff q = ff_norm(s, e + (q1.lo + q2.lo));
  if (ff_gt(q, C.cut2)) return false;
  G = ff_exp_neg(ff_mul(q, C.ninv2s2), T);
  return true;
}
struct SampleGrid {
  double x0, y0, cell;
  int nx, ny;
  const int64_t* off;  // [nx*ny + 1]
  const int* idx;    // sample ids bucketed by cell
};

__global__ void k_lc_bounds(const double* s, int64_t ns, double* out) {
  // one block: min/max of the samples
  __shared__ double sh[4][256];
  double a = INFINITY, b = -INFINITY, c = INFINITY, d = -INFINITY;
  for (int64_t k = threadIdx.x; k < ns; k += blockDim.x) {
    a = fmin(a, s[2 * k]); b = fmax(b, s[2 * k]);
    c = fmin(c, s[2 * k + 1]); d = fmax(d, s[2 * k + 1]);
  }
  sh[0][threadIdx.x] = a; sh[1][threadIdx.x] = b; sh[2][threadIdx.x] = c; sh[3][threadIdx.x] = d;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] = fmin(sh[0][threadIdx.x], sh[0][threadIdx.x + o]);
      sh[1][threadIdx.x] = fmax(sh[1][threadIdx.x], sh[1][threadIdx.x + o]);
      sh[2][threadIdx.x] = fmin(sh[2][threadIdx.x], sh[2][threadIdx.x + o]);
      sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 4) out[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_lc_count(const double* s, int64_t ns, double x0, double y0, double cell, int nx,
                           int ny, unsigned long long* cnt, int* cellof) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= ns) return;
  int cx = (int)floor((s[2 * k] - x0) / cell), cy = (int)floor((s[2 * k + 1] - y0) / cell);
  cx = min(max(cx, 0), nx - 1);
  cy = min(max(cy, 0), ny - 1);
  const int c = cy * nx + cx;
  cellof[k] = c;
  atomicAdd(&cnt[c], 1ull);
}

__global__ void k_lc_fill(int64_t ns, const int* cellof, const int64_t* off,
                          unsigned long long* cur, int* idx) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= ns) return;
  const int c = cellof[k];
  idx[off[c] + (int64_t)atomicAdd(&cur[c], 1ull)] = (int)k;
}

// warp-aggregated atomicAdd of 1 (lanes with the same counter combine)
__device__ __forceinline__ unsigned long long agg_inc(unsigned long long* p, int key) {
  const unsigned grp = __match_any_sync(__activemask(), key);
  const int lane = threadIdx.x & 31, leader = __ffs(grp) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(p, (unsigned long long)__popc(grp));
  base = __shfl_sync(grp, base, leader);
  return base + __popc(grp & ((1u << lane) - 1u));
}

// The rays near the samples: within one cell of the sample grid, bucketed over the
// parts of the grid widened by one cell on every side, (nx + 2) sub by (ny + 2) sub
// parts, row by row.  sub is 4, less for a very large grid.
struct RayGrid {
  double icell;   // 1 / cell
  float xf, yf, icf, slack;  // origin and 1 / cell in float32; its rounding, in cells
  float fsc;      // parts per unit length
  int sub;
};

// Cell c (-1 .. n) and offset of x from its origin: c = floor((x - x0) / cell), from
// the rounded product with 1 / cell and put right by the sign of the offset, which
// is formed anyway.  False for the rest, infinities and NaN included.  Four
// float64 operations; with the division, floor, comparisons and conversions on
// the float64 pipe, 22.
__device__ __forceinline__ bool locate(double x, double x0, double cell, double icell, int n,
                                       int& c, double& off) {
  const double t = (x - x0) * icell;
  const int H = __double2hiint(t);
  if (((unsigned)H & 0x7fffffffu) >= (1047u << 20)) return false;  // |t| >= 2^24, inf, NaN
  unsigned q;
  floor_u32(__hiloint2double(H & 0x7fffffff, __double2loint(t)), q);
  c = H < 0 ? -(int)q - 1 : (int)q;
  if (c < -2 || c > n + 1) return false;
  off = x - fma(f2d((float)c), cell, x0);
  const int step = __double2hiint(off) < 0 ? -1
                   : __double_as_longlong(off) >= __double_as_longlong(cell) ? 1 : 0;
  if (step != 0) {
    c += step;
    off = x - fma(f2d((float)c), cell, x0);
  }
  return c >= -1 && c <= n;
}

// surely beyond [-1, n + 1) cells, in float32 (the coordinate's and the origin's
// roundings and the subtraction's are covered by slack and 2^-21 of |x|)
__device__ __forceinline__ bool surely_out(double x, float x0, float icf, float slack, int n) {
  const float xf = d2f(x);
  const float t = (xf - x0) * icf, e = slack + fabsf(xf * icf) * 4.8e-7f;
  return t < -1.f - e || t > (float)(n + 1) + e;
}

// the ray's part, -1 for a ray that is not near; its position
__device__ __forceinline__ int ray_part(const SampleGrid& G, const RayGrid& R, double x, double y, Pos& p) {
  if (surely_out(x, R.xf, R.icf, R.slack, G.nx) || surely_out(y, R.yf, R.icf, R.slack, G.ny)) return -1;
  int cx, cy;
  double ox, oy;
  if (!locate(x, G.x0, G.cell, R.icell, G.nx, cx, ox) || !locate(y, G.y0, G.cell, R.icell, G.ny, cy, oy))
    return -1;
  const ff a = ff_of(ox), b = ff_of(oy);
  p = Pos{make_float4(a.hi, a.lo, b.hi, b.lo), make_int2(cx, cy)};
  const int fx = min(max((int)(a.hi * R.fsc), 0), R.sub - 1);
  const int fy = min(max((int)(b.hi * R.fsc), 0), R.sub - 1);
  return ((cy + 1) * R.sub + fy) * ((G.nx + 2) * R.sub) + (cx + 1) * R.sub + fx;
}

__global__ void k_lc_ray_cell(const double* __restrict__ y, int64_t m, SampleGrid G, RayGrid R,
                              int* __restrict__ partof, unsigned long long* __restrict__ cnt) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= m) return;
  Pos p;
  const int c = ray_part(G, R, y[2 * r], y[2 * r + 1], p);
  partof[r] = c;
  if (c >= 0) agg_inc(&cnt[c], c);
}

// positions (and ray numbers, where they are asked for) in the order of the parts
__global__ void k_lc_ray_fill(const double* __restrict__ y, int64_t m, const int* __restrict__ partof,
                              const int64_t* __restrict__ off, unsigned long long* __restrict__ cur,
                              SampleGrid G, RayGrid R, Pos* __restrict__ yp, int64_t* __restrict__ num) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= m) return;
  const int c = partof[r];
  if (c < 0) return;
  const int64_t pos = off[c] + (int64_t)agg_inc(&cur[c], c);
  Pos p;
  ray_part(G, R, y[2 * r], y[2 * r + 1], p);
  yp[pos] = p;
  if (num) num[pos] = r;
}

// F_k: one block per sample over the rays of the parts within the cut, row by row of
// parts (a row's parts are contiguous); the rows' rays are spread over the threads.
// Bound by instruction issue: a pair within the cut takes ~100 float32 operations,
// and a warp with one such pair issues them, so what the candidates beyond the cut
// cost counts: two thirds of them over 3 x 3 whole cells, one quarter over
// the parts.  3e6 rays (1.4e6 near), 2048 samples: 620 -> 305 us.
constexpr int kMaxSub = 4, kPartRows = 2 * kMaxSub + 4;

__global__ void __launch_bounds__(kLcThreads)
k_lc_fwd(const double* __restrict__ s, int64_t ns, SampleGrid G, RayGrid R,
         const int64_t* __restrict__ roff, const Pos* __restrict__ yp, ExpTab T, ff ninv2s2, ff cut2,
         float cutf, double norm, double* __restrict__ F) {
  __shared__ double red[kLcThreads / 32];
  __shared__ float2 sh_exp[64];
  __shared__ int64_t beg[kPartRows], incl[kPartRows];
  __shared__ float2 sx[3];
  const int64_t k = blockIdx.x;
  const double s1 = s[2 * k], s2 = s[2 * k + 1];
  int cx = (int)floor((s1 - G.x0) / G.cell), cy = (int)floor((s2 - G.y0) / G.cell);
  cx = min(max(cx, 0), G.nx - 1);
  cy = min(max(cy, 0), G.ny - 1);
  const Pos sp = make_pos(s1, s2, cx, cy, G.x0, G.y0, G.cell);
  const float side = (float)G.cell;
  // the cut's rows of parts, numbered from the sample's cell; every bound a
  // hundredth of a part wide of the float32 rounding (< 1e-5 parts)
  const float px = sp.o.x * R.fsc, py = sp.o.z * R.fsc;
  const float cu = cutf * R.fsc * 1.0001f + 0.01f;
  // (and within the sample's 3 x 3 cells, all of them in the widened grid)
  const int lo = max((int)floorf(py - cu), -R.sub);
  const int hi = min((int)floorf(py + cu), 2 * R.sub - 1);
  const int nrow = min(hi - lo + 1, kPartRows);
  if ((int)threadIdx.x < nrow) {
    const int j = lo + (int)threadIdx.x;
    const float dy = fmaxf(fmaxf((float)j - py, py - (float)(j + 1)) - 0.01f, 0.f);
    const float w = sqrtf(fmaxf(cu * cu - dy * dy, 0.f)) + 0.01f;
    const int xa = max((int)floorf(px - w), -R.sub);
    const int xb = min((int)floorf(px + w), 2 * R.sub - 1);
    const int row = ((cy + 1) * R.sub + j) * ((G.nx + 2) * R.sub) + (cx + 1) * R.sub;
    const int64_t b = roff[row + xa];
    beg[threadIdx.x] = b;
    incl[threadIdx.x] = xb >= xa ? roff[row + xb + 1] - b : 0;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int i = 1; i < nrow; ++i) incl[i] += incl[i - 1];
  // the sample in the frames of the three columns of cells
  if (threadIdx.x < 3) {
    const Shifted f = shifted(sp.o.x, sp.o.y, (1.f - (float)threadIdx.x) * side);
    sx[threadIdx.x] = make_float2(f.hi, f.mid);
  }
  const ExpShared X = stage_exp(T, sh_exp);
  const Cut C{ninv2s2, cut2, near_cut2(cutf, side)};
  ff acc{0.f, 0.f};
  const int64_t tot = nrow > 0 ? incl[nrow - 1] : 0;
  int row = 0;
  int64_t before = 0;  // rays of the rows ahead of `row`
  for (int64_t q = threadIdx.x; q < tot; q += kLcThreads) {
    while (incl[row] <= q) before = incl[row++];
    const Pos y = yp[beg[row] + (q - before)];
    const int ox = y.c.x - cx, oy = y.c.y - cy;  // -1 .. 1
    const float2 bx = sx[ox + 1];
    const Shifted by = shifted(sp.o.z, sp.o.w, (float)-oy * side);
    ff d1, d2, g;
    if (pair_gauss(y.o, make_float4(bx.x, sp.o.y, by.hi, by.lo), -bx.y, -by.mid, C, X, d1, d2, g))
      acc = ff_add(acc, g);
  }
  double a = ff_to_double(acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int w = 0; w < kLcThreads / 32; ++w) sum += red[w];
    F[k] = norm * sum;
  }
}

// samples in cell order: offsets and the gradient coefficient
// 2 (F_k - T_k) norm (-1 / sigma^2) (float-float)
__global__ void k_lc_sample_coef(const double* __restrict__ s, const int* __restrict__ idx, int64_t ns,
                                 SampleGrid G, const double* __restrict__ F,
                                 const double* __restrict__ T, double coef0, float4* __restrict__ so,
                                 float2* __restrict__ coef) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= ns) return;
  const int k = idx[t];
  const double s1 = s[2 * k], s2 = s[2 * k + 1];
  int cx = (int)floor((s1 - G.x0) / G.cell), cy = (int)floor((s2 - G.y0) / G.cell);
  cx = min(max(cx, 0), G.nx - 1);
  cy = min(max(cy, 0), G.ny - 1);
  so[t] = make_pos(s1, s2, cx, cy, G.x0, G.y0, G.cell).o;
  const ff c = ff_of(2.0 * (F[k] - T[k]) * coef0);
  coef[t] = make_float2(c.hi, c.lo);
}

// dL/dy_r of the rays near the samples, one thread per ray in the order of the parts
// (the rays of a warp see the same samples and mostly agree on the cut), over the
// samples of the 3 x 3 cells around it.  Bound by instruction issue, as the forward pass.
// In the order of the rays, with every ray's cell by divisions: 1140 us for 3e6 rays and
// 2048 samples (1.4e6 of them near), now 458.
// Not ORDERED: all m rays as they come, their positions formed here.
constexpr int kGradThreads = 128;
template <bool ORDERED>
__global__ void __launch_bounds__(kGradThreads)
k_lc_grad(const Pos* __restrict__ yp, const int64_t* __restrict__ num, const double* __restrict__ rays,
          int64_t m, SampleGrid G, RayGrid R, const float4* __restrict__ so,
          const float2* __restrict__ coef, ExpTab T, ff ninv2s2, ff cut2, float cutf,
          double* __restrict__ gy) {
  __shared__ float2 sh_exp[64];
  const ExpShared X = stage_exp(T, sh_exp);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= m) return;
  Pos y;
  if (ORDERED) {
    y = yp[i];
  } else if (ray_part(G, R, rays[2 * i], rays[2 * i + 1], y) < 0) {
    gy[2 * i] = 0.0;
    gy[2 * i + 1] = 0.0;
    return;
  }
  const float side = (float)G.cell;
  ff g1{0.f, 0.f}, g2{0.f, 0.f};
  const Cut C{ninv2s2, cut2, near_cut2(cutf, side)};
  for (int oy = -1; oy <= 1; ++oy) {
    const int yy = y.c.y + oy;
    if (yy < 0 || yy >= G.ny) continue;
    const Shifted ay = shifted(y.o.z, y.o.w, (float)-oy * side);  // in the frame of row yy
    for (int ox = -1; ox <= 1; ++ox) {
      const int xx = y.c.x + ox;
      if (xx < 0 || xx >= G.nx) continue;
      const Shifted ax = shifted(y.o.x, y.o.y, (float)-ox * side);
      const float4 a = make_float4(ax.hi, ax.lo, ay.hi, ay.lo);
      const int64_t t1 = G.off[yy * G.nx + xx + 1];
      for (int64_t t = G.off[yy * G.nx + xx]; t < t1; ++t) {
        ff d1, d2, g;
        if (!pair_gauss(a, so[t], ax.mid, ay.mid, C, X, d1, d2, g)) continue;
        const float2 c = coef[t];
        const ff c2 = ff_mul(ff{c.x, c.y}, g);
        g1 = ff_add(g1, ff_mul(c2, d1));
        g2 = ff_add(g2, ff_mul(c2, d2));
      }
    }
  }
  const int64_t r = ORDERED ? num[i] : i;
  gy[2 * r] = ff_to_double(g1);
  gy[2 * r + 1] = ff_to_double(g2);
}

struct GridHolder {
  SampleGrid G;
  Scratch off, idx;
};

void build_sample_grid(const double* smp, int64_t ns, double sigma, double trunc, DeviceAlloc& da,
                       cudaStream_t s, GridHolder& H) {
  Scratch bb(&da, sizeof(double) * 4);
  k_lc_bounds<<<1, 256, 0, s>>>(smp, ns, bb.as<double>());
  LENS_LAUNCHED("k_lc_bounds");
  double hb[4];
  int64_t hw[4];
  read_words(bb.as<int64_t>(), 4, hw, s);
  std::memcpy(hb, hw, sizeof(hb));
  if (!(std::isfinite(hb[0]) && std::isfinite(hb[1]) && std::isfinite(hb[2]) && std::isfinite(hb[3])))
    fail(LENS_EINVAL, "non-finite light-curve sample");
  // side: the least k 2^e (k = 4 .. 8, three significant bits) at or above
  // trunc sigma; origin: a multiple of it.  Then a cell's origin x0 + i side
  // is exact in float64, and so is a point's offset from it.
  int ex = 0;
  std::frexp(trunc * sigma, &ex);  // trunc sigma in [2^(ex-1), 2^ex)
  const double unit = std::ldexp(1.0, ex - 3);
  double cell = std::ceil(trunc * sigma / unit) * unit;
  double x0 = 0, y0 = 0;
  int nx = 0, ny = 0;
  for (;;) {
    x0 = std::floor(hb[0] / cell) * cell;
    y0 = std::floor(hb[2] / cell) * cell;
    nx = (int)std::ceil((hb[1] - x0) / cell) + 1;
    ny = (int)std::ceil((hb[3] - y0) / cell) + 1;
    if ((int64_t)nx * ny <= (1 << 22)) break;
    cell *= 2.0;
  }
  const int nc = nx * ny;
  Scratch cellof(&da, sizeof(int) * ns);
  Scratch cnt(&da, sizeof(int64_t) * 2 * (size_t)nc);  // counts, cursors
  H.off = Scratch(&da, sizeof(int64_t) * (size_t)(nc + 1));
  H.idx = Scratch(&da, sizeof(int) * ns);
  LENS_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes, s));
  unsigned long long* c = cnt.as<unsigned long long>();
  k_lc_count<<<grid_for(ns, 256), 256, 0, s>>>(smp, ns, x0, y0, cell, nx, ny, c, cellof.as<int>());
  LENS_LAUNCHED("k_lc_count");
  const ScanJob job{cnt.as<int64_t>(), H.off.as<int64_t>()};
  exclusive_scans(&job, 1, nc, da, s);
  k_lc_fill<<<grid_for(ns, 256), 256, 0, s>>>(ns, cellof.as<int>(), H.off.as<int64_t>(), c + nc,
                                              H.idx.as<int>());
  LENS_LAUNCHED("k_lc_fill");
  H.G = SampleGrid{x0, y0, cell, nx, ny, H.off.as<int64_t>(), H.idx.as<int>()};
}

// the rays near the samples, in the order of the parts
struct RayParts {
  RayGrid R;
  Scratch off, yp, num;
  int64_t near = 0;
};

// The gradient takes the rays as they come where there are few of them, few samples for a
// ray to look at (9 cells' worth, on average over the grid), or few pairs of both: the
// counting, its scan and read-back cost more than the order saves.  Random rays, as they come
// and in order: 3e6 and 1 sample a ray 255 and 966 us, 3 samples 298 and 344, 13 samples
// 618 and 358; 5000 and 64 samples 177 and 186, 256 samples 370 and 284; 3e4 and 16 samples
// 131 and 171.
constexpr int64_t kFewRays = 1 << 12;
constexpr double kFewSamples = 8.0, kFewPairs = 1e6;

RayGrid ray_grid(const SampleGrid& G, int sub) {
  const double icell = 1.0 / G.cell;
  return RayGrid{icell, (float)G.x0, (float)G.y0, (float)icell,
                 (float)(1e-3 + 4.8e-7 * (std::max(std::fabs(G.x0), std::fabs(G.y0)) * icell +
                                          std::max(G.nx, G.ny))),
                 (float)(sub * icell), sub};
}

void bucket_near_rays(const double* y, int64_t m, const SampleGrid& G, int sub, bool numbers,
                      DeviceAlloc& da, cudaStream_t s, RayParts& B) {
  const int64_t nce = (int64_t)(G.nx + 2) * (G.ny + 2);
  while (sub > 1 && nce * sub * sub > (1 << 22)) sub /= 2;
  const int64_t np = nce * sub * sub;
  B.R = ray_grid(G, sub);
  Scratch partof(&da, sizeof(int) * (size_t)m);
  Scratch cnt(&da, sizeof(int64_t) * 2 * (size_t)np);  // counts, cursors
  B.off = Scratch(&da, sizeof(int64_t) * (size_t)(np + 1));
  LENS_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes, s));
  unsigned long long* c = cnt.as<unsigned long long>();
  k_lc_ray_cell<<<grid_for(m, 256), 256, 0, s>>>(y, m, G, B.R, partof.as<int>(), c);
  LENS_LAUNCHED("k_lc_ray_cell");
  const ScanJob job{cnt.as<int64_t>(), B.off.as<int64_t>()};
  exclusive_scans(&job, 1, np, da, s);
  const int64_t* addr[1] = {B.off.as<int64_t>() + np};
  read_i64(addr, 1, &B.near, s);
  if (B.near == 0) return;
  B.yp = Scratch(&da, sizeof(Pos) * (size_t)B.near);
  if (numbers) B.num = Scratch(&da, sizeof(int64_t) * (size_t)B.near);
  k_lc_ray_fill<<<grid_for(m, 256), 256, 0, s>>>(y, m, partof.as<int>(), B.off.as<int64_t>(), c + np,
                                                 G, B.R, B.yp.as<Pos>(),
                                                 numbers ? B.num.as<int64_t>() : nullptr);
  LENS_LAUNCHED("k_lc_ray_fill");
}

}  // namespace

void light_curve(const double* y, int64_t m, double w, const double* smp, int64_t ns,
                 double sigma, double trunc, double* F, cudaStream_t s) {
  DeviceAlloc da;
  da.stream = s;
  LENS_CUDA(cudaMemsetAsync(F, 0, sizeof(double) * ns, s));
  if (m == 0 || ns == 0) return;
  GridHolder H;
  build_sample_grid(smp, ns, sigma, trunc, da, s, H);
  const SampleGrid& G = H.G;
  RayParts B;
  try {
    bucket_near_rays(y, m, G, kMaxSub, false, da, s, B);
  } catch (const Error& e) {
    if (e.status != LENS_ENOMEM) throw;
    B = RayParts{};  // whole cells: a sixteenth of the counters
    bucket_near_rays(y, m, G, 1, false, da, s, B);
  }
  if (ns > (int64_t)INT32_MAX) fail(LENS_EINVAL, "too many light-curve samples");
  static const ExpTab kExp = make_exp_tab();
  k_lc_fwd<<<(unsigned)ns, kLcThreads, 0, s>>>(smp, ns, G, B.R, B.off.as<int64_t>(), B.yp.as<Pos>(), kExp,
                                               ff_of(-1.0 / (2.0 * sigma * sigma)),
                                               ff_of(trunc * trunc * sigma * sigma),
                                               (float)(trunc * sigma),
                                               w / (2.0 * M_PI * sigma * sigma), F);
  LENS_LAUNCHED("k_lc_fwd");
  LENS_CUDA(cudaStreamSynchronize(s));
}

void light_curve_grad(const double* y, int64_t m, double w, const double* smp, int64_t ns,
                      double sigma, double trunc, const double* F, const double* T, double* gy,
                      cudaStream_t s) {
  DeviceAlloc da;
  da.stream = s;
  if (ns == 0) {
    LENS_CUDA(cudaMemsetAsync(gy, 0, sizeof(double) * 2 * m, s));
    return;
  }
  if (m == 0) return;
  GridHolder H;
  build_sample_grid(smp, ns, sigma, trunc, da, s, H);
  const double inv2s2 = 1.0 / (2.0 * sigma * sigma);
  const double norm = w / (2.0 * M_PI * sigma * sigma);
  Scratch so(&da, sizeof(float4) * (size_t)ns);
  Scratch coef(&da, sizeof(float2) * (size_t)ns);
  k_lc_sample_coef<<<grid_for(ns, 256), 256, 0, s>>>(smp, H.G.idx, ns, H.G, F, T,
                                                      norm * (-2.0 * inv2s2), so.as<float4>(),
                                                      coef.as<float2>());
  LENS_LAUNCHED("k_lc_sample_coef");
  static const ExpTab kExp = make_exp_tab();
  const double seen = std::min((double)ns, 9.0 * ns / ((double)H.G.nx * H.G.ny));
  bool ordered = m > kFewRays && seen > kFewSamples && seen * m > kFewPairs;
  RayParts B;
  try {
    if (ordered) bucket_near_rays(y, m, H.G, kMaxSub, true, da, s, B);
  } catch (const Error& e) {
    if (e.status != LENS_ENOMEM) throw;
    ordered = false;
    B = RayParts{};
  }
  if (ordered) {
    LENS_CUDA(cudaMemsetAsync(gy, 0, sizeof(double) * 2 * m, s));
  } else {
    B.R = ray_grid(H.G, 1);
    B.near = m;
  }
  if (B.near > 0) {
    const auto kernel = ordered ? k_lc_grad<true> : k_lc_grad<false>;
    kernel<<<grid_for(B.near, kGradThreads), kGradThreads, 0, s>>>(
        B.yp.as<Pos>(), B.num.as<int64_t>(), y, B.near, H.G, B.R, so.as<float4>(), coef.as<float2>(), kExp,
        ff_of(-inv2s2), ff_of(trunc * trunc * sigma * sigma), (float)(trunc * sigma), gy);
    LENS_LAUNCHED("k_lc_grad");
  }
  LENS_CUDA(cudaStreamSynchronize(s));
}

}  // namespace lens
