// mapops.cu -- consumers of a magnification map (Sec. 3: magnification
// histograms of finite sources, light curves along source tracks).
//  * finite Gaussian source: the map seen by a circular Gaussian source of
//    sigma pixels whose profile is cut at the isophote |d| = trunc sigma,
//    renormalised to the part of the profile inside the map.  The disk is a
//    stack of row segments |dx| <= r(dy); the weight exp(-|d|^2 / 2 s^2) is
//    g(dx) g(dy).  Two-pass form: the row sums over |dx| <= r of every map row
//    for all half-widths r by one chain, then a sum over dy per output pixel.
//    One-pass form (very wide disks): each output pixel sums, per dy >= 0, the
//    two map rows y + dy and y - dy (added once into shared memory) against
//    g(dx) over |dx| <= r(dy), folded as g(0) T[x] + sum_k g(k) (T[x+k] + T[x-k]).
//    The normalisation is the same stack of segments over the all-ones map
//    (one constant for the pixels at least R from every edge).  The map and g
//    are taken as float-float (pairs of float32, ~48 bits) and the sums run on
//    the float32 pipe (GB300's float64 pipe is ~1/74 of it), the normalisation
//    in float64;
//  * histogram: equal bins of the value or of log10(value), counts kept per
//    block in shared memory, then one atomic per bin and block;
//  * track: the map bilinear between pixel centres at source positions.
#include <algorithm>
#include <cmath>

#include "cx.cuh"
#include "lens_internal.h"

namespace lens {
namespace {

constexpr int kMaxSourceRadius = 1024;  // pixels
constexpr int kSourceThreads = 256;

// the map as float-float
__global__ void k_map_ff(const double* __restrict__ map, int64_t n, float2* __restrict__ mf) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ff v = ff_of(map[i]);
  mf[i] = make_float2(v.hi, v.lo);
}

// tab: g[0..R] (g[k] = exp(-k^2 / 2 s^2)), G[0..R] (G[k] = g[0] + .. + g[k]),
// then r[0..R] as ints (r[dy]: largest |dx| with dx^2 + dy^2 <= (trunc s)^2,
// -1 if none).  dfull: the normalisation of a pixel at least R from every
// edge.  Shared memory: g as float-float, then the folded row T (256 + 2 R).
__global__ void __launch_bounds__(kSourceThreads)
k_source_disk(const float2* __restrict__ mf, int npx, int npy, int R,
              const double* __restrict__ tab, double dfull, double* __restrict__ out) {
  extern __shared__ float2 smf[];
  float2* gf = smf;
  float2* T = smf + (R + 1);
  const double* G = tab + (R + 1);
  const int* rt = reinterpret_cast<const int*>(tab + 2 * (R + 1));
  const int t = threadIdx.x;
  const int blocks_x = (npx + kSourceThreads - 1) / kSourceThreads;
  const int py = blockIdx.x / blocks_x;
  const int x0 = (blockIdx.x - py * blocks_x) * kSourceThreads;
  const int px = x0 + t;
  for (int k = t; k <= R; k += kSourceThreads) {
    const ff v = ff_of(tab[k]);
    gf[k] = make_float2(v.hi, v.lo);
  }
  // every pixel of the block at least R from every edge: one normalisation
  const bool interior = x0 >= R && x0 + kSourceThreads - 1 <= npx - 1 - R && py >= R &&
                        py <= npy - 1 - R;
  ff num{0.f, 0.f};
  double den = 0.0;
  for (int dy = 0; dy <= R; ++dy) {
    const int r = rt[dy];
    const int ya = py + dy, yb = py - dy;
    const bool ina = ya < npy, inb = dy > 0 && yb >= 0;
    if (r < 0 || !(ina || inb)) continue;  // uniform over the block
    __syncthreads();  // the previous segment's readers of T are done
    const int nt = kSourceThreads + 2 * r;
    for (int i = t; i < nt; i += kSourceThreads) {
      const int x = x0 - r + i;
      ff v{0.f, 0.f};
      if (x >= 0 && x < npx) {
        if (ina) { const float2 a = mf[(int64_t)ya * npx + x]; v = ff{a.x, a.y}; }
        if (inb) { const float2 b = mf[(int64_t)yb * npx + x]; v = ff_add(v, ff{b.x, b.y}); }
      }
      T[i] = make_float2(v.hi, v.lo);
    }
    __syncthreads();
    if (px < npx) {
      const int c = t + r;
      ff acc = ff_mul(ff{gf[0].x, gf[0].y}, ff{T[c].x, T[c].y});
      for (int k = 1; k <= r; ++k) {
        const ff pair = ff_add(ff{T[c + k].x, T[c + k].y}, ff{T[c - k].x, T[c - k].y});
        acc = ff_add(acc, ff_mul(ff{gf[k].x, gf[k].y}, pair));
      }
      num = ff_add(num, ff_mul(ff{gf[dy].x, gf[dy].y}, acc));
      if (!interior) {
        // in-map weight of this segment: columns px - min(r, px) .. px + min(r, npx-1-px)
        const double seg = G[min(r, px)] + G[min(r, npx - 1 - px)] - tab[0];
        den = fma(tab[dy] * ((ina ? 1.0 : 0.0) + (inb ? 1.0 : 0.0)), seg, den);
      }
    }
  }
  if (px < npx) out[(int64_t)py * npx + px] = ff_to_double(num) / (interior ? dfull : den);
}

// The same sum in two passes over rows.  The row sums C_r[x] = sum_{|k| <= r} g(k)
// m[x + k] of one map row for every half-width r come from one chain (C_r =
// C_{r-1} + g(r) (m[x+r] + m[x-r])), and an output pixel is sum_dy g(dy)
// (C_{r(dy)} of row y + dy + C_{r(dy)} of row y - dy): R steps and R + 1 terms a
// pixel instead of one sum per segment, ~pi R^2 / 4 (30 and 31 against 707 at R =
// 30).  The row sums of the distinct half-widths go through a ring of map rows
// of bounded size.  Two neighbouring columns a thread, in the
// two-lane float32 instructions, float-float as above.  A 2000^2 map, R = 30: 3416
// -> 404 us (row sums 140, output rows 200; bound by load latency and issue), the
// error against 64 bits 6.9e-15 both times; 400^2, R = 2: 51 -> 47 us.
constexpr int kRowThreads = 64;
constexpr int kRowCols = 2 * kRowThreads;
constexpr int kRowStep = 4;  // steps of the chain whose pair sums are formed together

// a += g (h + l) for both columns, g the same in both: g4 = hi, hi, lo, lo
__device__ __forceinline__ void ff2_mac(ff2& a, float4 g4, float2 h, float2 l) {
  const float2 gh = make_float2(g4.x, g4.y), gl = make_float2(g4.z, g4.w);
  const float2 np = __fmul2_rn(make_float2(-g4.x, -g4.y), h);  // -round(g h)
  float2 pe = __ffma2_rn(gh, h, np);
  pe = __ffma2_rn(gh, l, __ffma2_rn(gl, h, pe));
  float2 s, e;
  two_diff2(a.hi, np, s, e);
  a = ff2_norm(s, __fadd2_rn(e, __fadd2_rn(a.lo, pe)));
}
// The tables come ready in float-float (a float64 instruction, a conversion
// included, costs a warp ~77 cycles of its sub-partition: the float64 loop over
// dy for the normalisation near the map's edges alone took 300 us as a tail of
// the launches, a float64 quotient a pixel 150): g4[k] = g(k) as hi, hi, lo, lo; qd[dy] the number of r(dy) among the distinct
// half-widths (counted from dy = R), qk[k] that number by half-width (-1: none).
// ring: [row mod nring][q][pair of columns], hi, hi, lo, lo.
struct RowPass {
  int npx, npy, R, pairs, nq, nring;
  int dlast;  // the last dy with r(dy) >= 0 (R but for rounding)
  int steps;  // R rounded up to whole groups of kRowStep, plus one
  const float4* g4;   // [steps]
  const int* qk;      // [steps]
  const int* qd;      // [R + 1]
  const double* Q;    // [R + 1][R + 1] in-map weights, see k_source_rows
  float4* ring;
};

// Row sums of map rows row0 + blockIdx.y.  The row is staged twice over (hi, lo;
// then the same shifted by one column), so that the columns c + k, c + k + 1 are
// one aligned load for odd k as well.
__global__ void __launch_bounds__(kRowThreads)
k_row_sums(const double* __restrict__ map, RowPass A, int row0) {
  extern __shared__ float4 sm4[];
  const int R = A.R, steps = A.steps;
  const int pad = (steps + 1) & ~1, nt = kRowCols + 2 * pad;
  float4* gk = sm4;                                 // [steps]
  float* T = reinterpret_cast<float*>(gk + steps);  // [hi, lo, shifted hi, lo][nt]
  int* qk = reinterpret_cast<int*>(T + 4 * nt);     // [steps]
  const int t = threadIdx.x, c = 2 * t + pad;
  const int x0 = blockIdx.x * kRowCols, row = row0 + blockIdx.y;
  for (int k = t; k < steps; k += kRowThreads) {
    gk[k] = A.g4[k];
    qk[k] = A.qk[k];
  }
  for (int i = t; i < nt; i += kRowThreads) {
    const int x = x0 - pad + i;
    const ff v = ff_of(x >= 0 && x < A.npx ? map[(int64_t)row * A.npx + x] : 0.0);
    T[i] = v.hi;
    T[nt + i] = v.lo;
    if (i > 0) {
      T[2 * nt + i - 1] = v.hi;
      T[3 * nt + i - 1] = v.lo;
    }
  }
  __syncthreads();
  const int pair = blockIdx.x * kRowThreads + t;
  if (pair >= A.pairs) return;
  float4* out = A.ring + (int64_t)(row % A.nring) * A.nq * A.pairs + pair;
  const float* Tc = T + c;
  const auto at = [](const float* q) { return *reinterpret_cast<const float2*>(q); };
  ff2 C{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const auto keep = [&](int k) {
    const int q = qk[k];
    if (q >= 0) out[(int64_t)q * A.pairs] = make_float4(C.hi.x, C.hi.y, C.lo.x, C.lo.y);
  };
  ff2_mac(C, gk[0], at(Tc), at(Tc + nt));
  keep(0);
  for (int k = 1; k <= R; k += kRowStep) {
    float2 s[kRowStep], e[kRowStep];
#pragma unroll
    for (int j = 0; j < kRowStep; ++j) {
      const float* Tj = Tc + (j & 1 ? 0 : 2 * nt - 1);  // k + j is odd for even j
      const float *ta = Tj + (k + j), *tb = Tj - (k + j);
      two_sum2(at(ta), at(tb), s[j], e[j]);
      e[j] = __fadd2_rn(e[j], __fadd2_rn(at(ta + nt), at(tb + nt)));
    }
#pragma unroll
    for (int j = 0; j < kRowStep; ++j) {
      ff2_mac(C, gk[k + j], s[j], e[j]);
      keep(k + j);
    }
  }
}

// Output rows y0 + blockIdx.y from the ring.
__global__ void __launch_bounds__(kRowThreads)
k_source_rows(RowPass A, int y0, double inv_full, double* __restrict__ out) {
  extern __shared__ float4 sm4[];
  const int R = A.R, npx = A.npx, npy = A.npy;
  float4* gd = sm4;                             // [R + 1]
  int* qd = reinterpret_cast<int*>(gd + R + 1);  // [R + 1]
  const int t = threadIdx.x;
  for (int k = t; k <= R; k += kRowThreads) {
    gd[k] = A.g4[k];
    qd[k] = A.qd[k];
  }
  __syncthreads();
  const int pair = blockIdx.x * kRowThreads + t, py = y0 + blockIdx.y;
  if (pair >= A.pairs) return;
  const float4* ring = A.ring + pair;
  const int64_t ld = (int64_t)A.nq * A.pairs;
  const uint32_t pr = (uint32_t)A.pairs;
  const auto both = [](float4 v) { return ff2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; };
  const auto load = [&](int row, int dy) {  // row: a ring slot after any number of wraps
    row = row < 0 ? row + A.nring : row >= A.nring ? row - A.nring : row;
    return ring[(uint64_t)row * ld + (uint32_t)qd[dy] * pr];
  };
  const int r0 = py % A.nring;  // R < nring, so row py + dy is at most one wrap away
  ff2 acc{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  {
    const ff2 p = both(load(r0, 0));
    ff2_mac(acc, gd[0], p.hi, p.lo);
  }
  int dy = 1;
  if (py >= A.dlast && py + A.dlast < npy) {  // uniform over the block
    for (; dy + kRowStep - 1 <= A.dlast; dy += kRowStep) {
      float4 u[kRowStep], v[kRowStep];
#pragma unroll
      for (int j = 0; j < kRowStep; ++j) {
        u[j] = load(r0 + dy + j, dy + j);
        v[j] = load(r0 - dy - j, dy + j);
      }
#pragma unroll
      for (int j = 0; j < kRowStep; ++j) {
        const ff2 p = ff2_add(both(u[j]), both(v[j]));
        ff2_mac(acc, gd[dy + j], p.hi, p.lo);
      }
    }
  }
  for (; dy <= A.dlast; ++dy) {
    ff2 p{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (py + dy < npy) p = both(load(r0 + dy, dy));
    if (py >= dy) p = ff2_add(p, both(load(r0 - dy, dy)));
    ff2_mac(acc, gd[dy], p.hi, p.lo);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int px = 2 * pair + q;
    if (px >= npx) break;
    const ff num = q ? ff{acc.hi.y, acc.lo.y} : ff{acc.hi.x, acc.lo.x};
    double w = inv_full;
    if (px < R || px > npx - 1 - R || py < R || py > npy - 1 - R) {
      // in-map weight: with Q[e][n] = sum_{dy <= n} g(dy) G[min(r(dy), e)], the
      // segments' parts on either side of the column and of the row
      const double* Ql = A.Q + (int64_t)min(px, R) * (R + 1);
      const double* Qr = A.Q + (int64_t)min(npx - 1 - px, R) * (R + 1);
      const int na = min(npy - 1 - py, R), nb = min(py, R);
      const double den = (Ql[na] + Qr[na] - A.Q[na]) + (Ql[nb] + Qr[nb] - A.Q[nb]) -
                         (Ql[0] + Qr[0] - A.Q[0]);
      w = 1.0 / den;
    }
    out[(int64_t)py * npx + px] = ff_to_double(num) * w;
  }
}

__global__ void k_histogram(const double* __restrict__ v, int64_t n, double lo, double hi,
                            int nbins, int log_bins, unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned int hb[];  // nbins + 2
  for (int b = threadIdx.x; b < nbins + 2; b += blockDim.x) hb[b] = 0;
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double x = v[i];
    int b;
    if (log_bins && !(x > 0.0)) {
      b = 0;
    } else {
      if (log_bins) x = log10(x);
      if (x < lo) b = 0;
      else if (x >= hi) b = nbins + 1;
      else b = 1 + min((int)floor((x - lo) / (hi - lo) * nbins), nbins - 1);
    }
    atomicAdd(&hb[b], 1u);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins + 2; b += blockDim.x)
    if (hb[b]) atomicAdd(&counts[b], (unsigned long long)hb[b]);
}

__global__ void k_track(const double* __restrict__ map, int npx, int npy, double u0, double v0,
                        double du, double dv, const double2* __restrict__ s, int64_t ns,
                        double* __restrict__ out) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= ns) return;
  double x = (s[k].x - u0) / du - 0.5, y = (s[k].y - v0) / dv - 0.5;
  x = fmin(fmax(x, 0.0), (double)(npx - 1));
  y = fmin(fmax(y, 0.0), (double)(npy - 1));
  int ix = (int)floor(x), iy = (int)floor(y);
  if (ix > npx - 2) ix = npx > 1 ? npx - 2 : 0;
  if (iy > npy - 2) iy = npy > 1 ? npy - 2 : 0;
  const double fx = npx > 1 ? x - ix : 0.0, fy = npy > 1 ? y - iy : 0.0;
  const int ix1 = npx > 1 ? ix + 1 : ix, iy1 = npy > 1 ? iy + 1 : iy;
  const double m00 = map[(int64_t)iy * npx + ix], m10 = map[(int64_t)iy * npx + ix1];
  const double m01 = map[(int64_t)iy1 * npx + ix], m11 = map[(int64_t)iy1 * npx + ix1];
  out[k] = (1 - fy) * ((1 - fx) * m00 + fx * m10) + fy * ((1 - fx) * m01 + fx * m11);
}

// The two-pass form keeps a ring of 2 R + some map rows of row sums.  Few long
// launches beat a ring that fits L2: 80 MB 589 us, 200 MB 478, 384 MB 404 (2000^2, R =
// 30).  Wide disks on wide maps may take up to kRingMax; beyond that, beyond
// kTwoPassMaxR, or where the memory is not to be had, the one-pass kernel runs
// (401 x 333 pixels, R = 240: 9168 us against 306).
constexpr size_t kRingBytes = (size_t)384 << 20, kRingMax = (size_t)512 << 20;
constexpr int kRingMinRows = 32;  // output rows a launch
// a few terms a pixel of a small map are less than a second launch: one pass there (64^2
// px, R 1: 35 us against 38; R 12: 50 against 43; 1000^2 px, R 1: 76 against 56)
constexpr int kOnePassR = 4;
constexpr int64_t kOnePassPixels = 1 << 16;
constexpr int kTwoPassMaxR = 256;  // (R + 1)^2 in-map weights are formed on the host

bool source_two_pass(const double* map, RowPass A, double dfull, double* out, DeviceAlloc& da,
                     cudaStream_t s) {
  const int npy = A.npy, R = A.R, nq = A.nq;
  const size_t row = sizeof(float4) * (size_t)A.pairs * nq;
  const int64_t fit = (int64_t)(kRingBytes / row) - 2 * R;
  const int rows = (int)std::min<int64_t>(npy, std::max<int64_t>(kRingMinRows, fit));
  A.nring = (int)std::min<int64_t>(npy, (int64_t)rows + 2 * R);
  if (row * (size_t)A.nring > kRingMax) return false;
  Scratch ring;
  try {
    ring = Scratch(&da, row * (size_t)A.nring);
  } catch (const Error& e) {
    if (e.status != LENS_ENOMEM) throw;
    return false;
  }
  A.ring = ring.as<float4>();
  const int steps = A.steps, pad = (steps + 1) & ~1;
  const size_t sm1 = (sizeof(float4) + sizeof(int)) * (size_t)steps +
                     sizeof(float) * 4 * ((size_t)kRowCols + 2 * pad);
  const size_t sm2 = (sizeof(float4) + sizeof(int)) * ((size_t)R + 1);
  if (sm1 > 48 * 1024)
    LENS_CUDA(cudaFuncSetAttribute(k_row_sums, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm1));
  const unsigned bx = (unsigned)((A.pairs + kRowThreads - 1) / kRowThreads);
  int done = 0;  // map rows summed so far
  for (int y0 = 0; y0 < npy; y0 += rows) {
    const int ny = std::min(rows, npy - y0), need = std::min(npy, y0 + ny + R);
    for (; done < need;) {  // at most 65535 rows a launch
      const int n = std::min(need - done, 65535);
      k_row_sums<<<dim3(bx, (unsigned)n), kRowThreads, sm1, s>>>(map, A, done);
      LENS_LAUNCHED("k_row_sums");
      done += n;
    }
    for (int y = y0; y < y0 + ny; y += 65535) {
      const int n = std::min(y0 + ny - y, 65535);
      k_source_rows<<<dim3(bx, (unsigned)n), kRowThreads, sm2, s>>>(A, y, 1.0 / dfull, out);
      LENS_LAUNCHED("k_source_rows");
    }
  }
  return true;
}

void source_one_pass(const double* map, int npx, int npy, int R, const double* tab, double dfull,
                     double* out, DeviceAlloc& da, cudaStream_t s) {
  const int64_t npix = (int64_t)npx * npy;
  const int blocks_x = (npx + kSourceThreads - 1) / kSourceThreads;
  const int64_t blocks = (int64_t)blocks_x * npy;
  if (blocks > INT32_MAX) fail(LENS_EINVAL, "map too large");
  Scratch mf(&da, sizeof(float2) * (size_t)npix);
  k_map_ff<<<grid_for(npix, 256), 256, 0, s>>>(map, npix, mf.as<float2>());
  LENS_LAUNCHED("k_map_ff");
  const size_t smem = sizeof(float2) * ((size_t)R + 1 + kSourceThreads + 2 * (size_t)R);
  if (smem > 48 * 1024)
    LENS_CUDA(cudaFuncSetAttribute(k_source_disk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)smem));
  k_source_disk<<<(unsigned)blocks, kSourceThreads, smem, s>>>(mf.as<float2>(), npx, npy, R, tab,
                                                               dfull, out);
  LENS_LAUNCHED("k_source_disk");
}

}  // namespace

void map_source(const double* map, int npx, int npy, double sigma_px, double trunc, double* out,
                DeviceAlloc& da, cudaStream_t s) {
  const int R = (int)std::floor(trunc * sigma_px);
  if (R > kMaxSourceRadius) fail(LENS_EINVAL, "source radius above 1024 pixels");
  // the disk: integer offsets with dx^2 + dy^2 <= (trunc sigma)^2 (the same
  // products in the same order as the definition, so the same offsets)
  const double cut2 = trunc * trunc * sigma_px * sigma_px;
  const double inv2s2 = 1.0 / (2.0 * sigma_px * sigma_px);
  const size_t n1 = (size_t)R + 1;
  const int steps = (R + kRowStep - 1) / kRowStep * kRowStep + 1;
  // one host block: g, G, r(dy) (float64 slots), then the float-float tables of
  // the two-pass form on a 16-byte boundary, its ints and its in-map weights
  const bool two = R <= kTwoPassMaxR && (R > kOnePassR || (int64_t)npx * npy > kOnePassPixels);
  const size_t nf = (3 * n1 + 1) / 2 * 2, ni = (size_t)steps + n1;
  const size_t nq0 = nf + 2 * (size_t)steps + (ni + 1) / 2;
  std::vector<double> tab(nq0 + (two ? n1 * n1 : 0), 0.0);
  double acc = 0.0;
  for (int d = 0; d <= R; ++d) {
    tab[(size_t)d] = std::exp(-(double)d * d * inv2s2);
    acc += tab[(size_t)d];
    tab[n1 + (size_t)d] = acc;
  }
  int* rt = reinterpret_cast<int*>(tab.data() + 2 * n1);
  for (int dy = 0; dy <= R; ++dy) {
    int r = -1;
    while (r < R && (double)(r + 1) * (r + 1) + (double)dy * dy <= cut2) ++r;
    rt[dy] = r;
  }
  // the normalisation of an interior pixel, in the kernels' order
  double dfull = 0.0;
  for (int dy = 0; dy <= R; ++dy) {
    if (rt[dy] < 0) continue;
    const double seg = tab[n1 + (size_t)rt[dy]] + tab[n1 + (size_t)rt[dy]] - tab[0];
    dfull = std::fma(tab[(size_t)dy] * (dy > 0 ? 2.0 : 1.0), seg, dfull);
  }
  float* g4 = reinterpret_cast<float*>(tab.data() + nf);
  int* qk = reinterpret_cast<int*>(g4 + 4 * (size_t)steps);
  int* qd = qk + steps;
  RowPass A{};
  A.npx = npx; A.npy = npy; A.R = R; A.pairs = (npx + 1) / 2; A.steps = steps;
  for (int k = 0; k <= R; ++k) {
    const ff v = ff_of(tab[(size_t)k]);
    g4[4 * k] = g4[4 * k + 1] = v.hi;
    g4[4 * k + 2] = g4[4 * k + 3] = v.lo;
  }
  std::fill(qk, qk + steps, -1);
  for (int dy = R; dy >= 0; --dy) {
    qd[dy] = -1;
    if (rt[dy] < 0) continue;
    A.dlast = std::max(A.dlast, dy);
    if (qk[rt[dy]] < 0) qk[rt[dy]] = A.nq++;
    qd[dy] = qk[rt[dy]];
  }
  for (size_t e = 0; two && e < n1; ++e) {
    double q = 0.0;
    for (size_t dy = 0; dy < n1; ++dy) {
      if (rt[dy] >= 0) q = std::fma(tab[dy], tab[n1 + std::min((size_t)rt[dy], e)], q);
      tab[nq0 + e * n1 + dy] = q;
    }
  }
  Scratch dt(&da, sizeof(double) * tab.size());
  LENS_CUDA(cudaMemcpyAsync(dt.p, tab.data(), sizeof(double) * tab.size(), cudaMemcpyHostToDevice,
                            s));
  A.g4 = reinterpret_cast<const float4*>(dt.as<double>() + nf);
  A.Q = dt.as<double>() + nq0;
  A.qk = reinterpret_cast<const int*>(A.g4 + steps);
  A.qd = A.qk + steps;
  if (!two || !source_two_pass(map, A, dfull, out, da, s))
    source_one_pass(map, npx, npy, R, dt.as<double>(), dfull, out, da, s);
  // the host table must outlive the copy
  LENS_CUDA(cudaStreamSynchronize(s));
}

void map_histogram(const double* v, int64_t n, double lo, double hi, int nbins, int log_bins,
                   int64_t* counts, cudaStream_t s) {
  LENS_CUDA(cudaMemsetAsync(counts, 0, sizeof(int64_t) * (size_t)(nbins + 2), s));
  if (n == 0) return;
  const size_t smem = sizeof(unsigned int) * (size_t)(nbins + 2);
  k_histogram<<<grid_for(n, 256, 152 * 8), 256, smem, s>>>(
      v, n, lo, hi, nbins, log_bins, reinterpret_cast<unsigned long long*>(counts));
  LENS_LAUNCHED("k_histogram");
}

void map_track(const double* map, int npx, int npy, const double box[4], const double* pos,
               int64_t ns, double* out, cudaStream_t s) {
  if (ns == 0) return;
  const double du = (box[1] - box[0]) / npx, dv = (box[3] - box[2]) / npy;
  k_track<<<grid_for(ns, 256), 256, 0, s>>>(map, npx, npy, box[0], box[2], du, dv,
                                            reinterpret_cast<const double2*>(pos), ns, out);
  LENS_LAUNCHED("k_track");
}

}  // namespace lens
