// ipm.cu -- first-order Inverse Polygon Mapping (Sec. 2.3; step 4 of the
// FMM-IPM algorithm of Sec. 2.4).  Each image-plane cell (i, j) of a grid
// chunk has corners y[j][i], y[j][i+1], y[j+1][i+1], y[j+1][i]
// (counter-clockwise in the image plane); its source-plane quadrilateral P
// receives the cell area h^2, apportioned over the map pixels by the signed
// overlap fraction a_pix / A_P, and
//     map[pix] += (h^2 / S*) * a_pix / A_P.
//
// Corners arrive in pixel coordinates u = (y1 - u0)/du, v = (y2 - v0)/dv,
// split as (floor, float fraction) by the deflection epilogue, so no step
// needs float64.  One warp takes 32 consecutive cells
// (k_ipm_cells): single-pixel cells add their whole area; cells with a pixel
// box up to 4 x 4 get one overlap per pixel; larger cells are swept row band
// by row band, whole-pixel runs going to a per-row difference array and
// only the pixels an edge crosses getting an overlap; all three kinds of
// work are spread evenly over the warp's lanes.  Ill-conditioned cells
// (|A_P| small against the box) are queued for float-float (k_ipm_ext).
// Overlaps come from Green's theorem, edge by edge (the apportioning rule of
// Sec. 2.3): the result is the winding-number-weighted area, so inverted and
// self-intersecting (critical) cells are handled "naively", as the
// first-order IPM does.
// Ledger per chunk: area_in_map, area_outside, area_dropped (bbox larger
// than the cap, or a corner beyond 2^30 pixels), area_degenerate
// (|A_P| <= 1e-14 h^2).
#include "cx.cuh"
#include "ipm_warp.cuh"
#include "lens_internal.h"

namespace lens {
namespace {

constexpr int kIpmThreads = 256;
// 32-cell chunks per fetch of the chunk counter: at most 8 (a single address serves all
// warps, ~2 ns a fetch: a fetch per chunk made it the bound of a pass without B and C work),
// fewer where that would leave a resident warp under 8 fetches: with 8 always, the 900
// chunks of a refinement level went to 112 of 4864 warps (308 us of a 200^2-pixel window's
// map) and the 7.8e3 chunks of a 500^2 grid to 976.
constexpr int kMaxGrab = 8, kFetches = 8;
// A pass of kDense cells a map pixel or more: 3 fetches a warp are enough (cells of a pixel
// or two each: 4e6 of them 340 us, with 8 fetches 498), and they are dealt out to strips of the
// cells, 16 for fetches of 8 chunks and more for shorter ones (kSpread chunks in all), so that
// the resident warps work in many places: next to each other they queue up at the same
// pixels where a map is strongly compressed (4000^2 cells of a field at high magnification on
// 100^2 pixels: 15.5 ms in one strip, 9.4 so).  Sparser passes go in order (4e6 cells, the
// tenth of them that falls on the map's 4e6 pixels 10 pixels long: 160 us, in strips 265),
// and so do those of more than kStripCells cells, whose corners do not stay in L2 (critical-
// curve map: 643 ms, in strips 744).
constexpr int kFetchesDense = 3, kSpread = 128;
constexpr double kDense = 1.5;
constexpr int64_t kStripCells = 6 << 20;
// Cells per chunk: 32, fewer (down to kMinLanes lanes with a cell) while that leaves fewer
// than kChunksPerWarp chunks for a resident warp.  Most of a round's work is pixels and rows,
// spread over all lanes whoever holds the cells, so short rounds cost little and a
// refinement level or a small grid reaches all the warps: 2.9e4 sub-cells of a window map
// 79 -> 29 us (2 chunks a warp the same, 4: a 500^2 grid 35 -> 46 us).
constexpr int kMinLanes = 4, kChunksPerWarp = 1;
constexpr int kBlocksPerSm = 4;

constexpr int kWarps = kIpmThreads / 32;

// c / nx for a cell id c < 2^30: with L = ceil(log2 nx) and M = floor(2^(30+L)
// / nx) + 1 < 2^32, M nx - 2^(30+L) <= nx <= 2^L, so c M / 2^(30+L) exceeds c / nx by
// less than 1 / nx and the floors agree (a 32-bit division takes ~20 instructions
// of the ~350 that a round of single-pixel cells has).
__device__ __forceinline__ int64_t cell_row(const IpmArgs& A, uint32_t c) {
  return (int64_t)(((uint64_t)c * A.div_m) >> A.div_s);
}

// One warp per round of up to 32 cells of a grid chunk (or of a cell list, or of
// sub-cells given as four corners each), rounds handed out by a counter.
template <bool QUADS, bool LIST = false>
__global__ void __launch_bounds__(kIpmThreads, kBlocksPerSm) k_ipm_cells(IpmArgs A) {
  __shared__ WarpCells sh[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int lanes = A.lanes;
  const int64_t nchunks = (A.ncells + lanes - 1) / lanes;
  const int64_t W = A.nx + 1;
  Ledger led;
  // Chunks of A.lanes cells are handed out by a counter (qcount[1]), so the
  // warps of a block finish together however the large cells fall; one
  // fetch takes A.grab chunks.
  unsigned* next = reinterpret_cast<unsigned*>(A.qcount) + 1;
  // (the first fetch is the warp's number)
  const unsigned warps = gridDim.x * kWarps;
  unsigned g_u = blockIdx.x * kWarps + w;
  for (;;) {
    const unsigned f = __shfl_sync(0xffffffffu, g_u, 0), pos = f >> A.strips;
    if (pos >= A.per) break;
    // the following grab is fetched while this one is processed
    if (lane == 0) g_u = warps + atomicAdd(next, 1u);
    int64_t ch = ((int64_t)(f - (pos << A.strips)) * A.per + pos) * A.grab;
    const int64_t end = min64(ch + A.grab, nchunks);
    for (; ch < end; ++ch) {
      const int64_t idx = ch * lanes + lane;
      const bool has = lane < lanes && idx < A.ncells;
      int64_t c = idx;
      PixCorner q4[4];
      if (has) {
        if (LIST) c = A.cell_list[idx];
        if (QUADS) {
#pragma unroll
          for (int k = 0; k < 4; ++k) q4[k] = A.yc[4 * c + k];
        } else {
          const int64_t j = cell_row(A, (uint32_t)c);
          const PixCorner* y0 = A.yc + (c + j);  // j W + i = c + j
          q4[0] = y0[0];
          q4[1] = y0[1];
          q4[2] = y0[W + 1];
          q4[3] = y0[W];
        }
      }
      ipm_round<false>(A, sh[w], lane, has, c, q4, led);
      __syncwarp();  // the next chunk overwrites this one's staging
    }
  }
  block_add_stats<kWarps>(A.stats, led, A.wcell);
}

// Ill-conditioned cells queued by k_ipm_cells, up to 32 a warp.  Bound by instruction issue, the float-float arithmetic of the cut pixels.  A
// cell a warp: 4096^2 map of a clustered field 123 us, 2000^2 at high magnification
// 220, a critical-curve map of 21 bands 17.4 ms; now 23 us, 42 us, 1.3 ms.
template <bool QUADS>
__global__ void __launch_bounds__(kIpmThreads) k_ipm_ext(IpmArgs A) {
  __shared__ int cut_x[kWarps][64], cut_y[kWarps][64];
  __shared__ ExtCells sh[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t wg = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nq = *A.qcount;
  Ledger led;
  ExtSum sum;
  // a warp's cells are nwarps apart: neighbours have boxes of one size
  for (int64_t t0 = wg; t0 < nq; t0 += nwarps * 32) {
    const int64_t t = t0 + nwarps * lane;
    const bool has = t < nq;
    PixCorner q4[4];
    if (has) {
      const int64_t c = A.queue[t];
      if (QUADS) {
#pragma unroll
        for (int k = 0; k < 4; ++k) q4[k] = A.yc[4 * c + k];
      } else {
        const int64_t j = cell_row(A, (uint32_t)c), W = A.nx + 1;
        const PixCorner* y0 = A.yc + (c + j);
        q4[0] = y0[0];
        q4[1] = y0[1];
        q4[2] = y0[W + 1];
        q4[3] = y0[W];
      }
    }
    const bool large = ext_round(A, sh[w], lane, has, q4, led, sum);
    for (unsigned m = __ballot_sync(0xffffffffu, large); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      PixCorner qq[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        qq[k].iu = __shfl_sync(0xffffffffu, q4[k].iu, src);
        qq[k].fu = __shfl_sync(0xffffffffu, q4[k].fu, src);
        qq[k].iv = __shfl_sync(0xffffffffu, q4[k].iv, src);
        qq[k].fv = __shfl_sync(0xffffffffu, q4[k].fv, src);
      }
      ext_cell_call(A, qq, cut_x[w], cut_y[w], lane, led);
    }
  }
  ext_close(sum, lane, led);
  block_add_stats<kWarps>(A.stats, led, A.wcell);
}

}  // namespace

std::pair<cudaEvent_t, cudaEvent_t> event_pair_begin(cudaStream_t s) {
  std::pair<cudaEvent_t, cudaEvent_t> e;
  LENS_CUDA(cudaEventCreate(&e.first));
  LENS_CUDA(cudaEventCreate(&e.second));
  LENS_CUDA(cudaEventRecord(e.first, s));
  return e;
}
void event_pair_end(std::pair<cudaEvent_t, cudaEvent_t>& e, cudaStream_t s) {
  LENS_CUDA(cudaEventRecord(e.second, s));
}

// thresholds and the float32 map increment of a launch (from ip and wcell)
void ipm_prepare(IpmArgs& A) {
  A.thr_area = (float)(1e-13 * A.ip.a_cell / A.ip.s_star);
  A.thr_degen = (float)(1e-14 * A.ip.a_cell / A.ip.s_star);
  A.scale_f = (float)(A.ip.scale * A.wcell);
}

namespace {
void ipm_launch(IpmArgs& A, bool quads, int* qcount, cudaStream_t s,
                std::vector<std::pair<cudaEvent_t, cudaEvent_t>>* ev) {
  ipm_prepare(A);
  // qcount[0]: float-float queue length; qcount[1]: chunk counter of k_ipm_cells
  LENS_CUDA(cudaMemsetAsync(qcount, 0, 2 * sizeof(int), s));
  std::pair<cudaEvent_t, cudaEvent_t> e;
  if (ev) e = event_pair_begin(s);
  int dev = 0, sms = 152;
  LENS_CUDA(cudaGetDevice(&dev));
  LENS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  A.lanes = 32;
  const int64_t warps = (int64_t)sms * kBlocksPerSm * kWarps;
  while (A.lanes > kMinLanes && A.ncells / A.lanes < kChunksPerWarp * warps) A.lanes /= 2;
  const int64_t chunk_blocks = (A.ncells + A.lanes * kWarps - 1) / (A.lanes * kWarps);
  const unsigned g = (unsigned)std::min<int64_t>(chunk_blocks, (int64_t)sms * kBlocksPerSm);
  int L = 0;
  while ((1ll << L) < A.nx) ++L;
  A.div_s = 30 + L;
  A.div_m = A.nx > 0 ? (uint32_t)((1ull << A.div_s) / (uint64_t)A.nx + 1) : 0;
  const bool dense = (double)A.ncells >= kDense * A.ip.npx * A.ip.npy;
  A.grab = (int)std::max<int64_t>(
      1, std::min<int64_t>(kMaxGrab, A.ncells / A.lanes / (warps * (dense ? kFetchesDense : kFetches))));
  const int64_t fetches = (A.ncells + (int64_t)A.lanes * A.grab - 1) / ((int64_t)A.lanes * A.grab);
  A.strips = 0;
  if (dense && A.ncells <= kStripCells)
    while (A.grab << A.strips < kSpread && fetches >> A.strips >= 8) ++A.strips;
  A.per = (unsigned)((fetches + (1 << A.strips) - 1) >> A.strips);
  if (quads) k_ipm_cells<true><<<g, kIpmThreads, 0, s>>>(A);
  else if (A.cell_list) k_ipm_cells<false, true><<<g, kIpmThreads, 0, s>>>(A);
  else k_ipm_cells<false><<<g, kIpmThreads, 0, s>>>(A);
  LENS_LAUNCHED("k_ipm_cells");
  if (quads) k_ipm_ext<true><<<sms * 2, kIpmThreads, 0, s>>>(A);
  else k_ipm_ext<false><<<sms * 2, kIpmThreads, 0, s>>>(A);
  LENS_LAUNCHED("k_ipm_ext");
  if (ev) {
    event_pair_end(e, s);
    ev->push_back(e);
  }
}

// Refinement, step 1: for each queued cell, its 3 x 3 corner grid of half
// spacing (the rays to deflect) and the lower-left corners of its 2 x 2
// sub-cells.  A queued cell is a grid cell (origin from the grid) at the first
// level, a sub-cell of the previous level (origin from org_in) after that.
__global__ void k_refine_points(const int* __restrict__ parents, int64_t np,
                                const double2* __restrict__ org_in, double gx0, double gy0,
                                int64_t grow0, int64_t gnx, double h, double2* __restrict__ rays,
                                double2* __restrict__ org_out) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= np) return;
  const int64_t c = parents[k];
  double xl, yl;
  if (org_in) {
    xl = org_in[c].x; yl = org_in[c].y;
  } else {
    // the expression the grid's corners use: x0 + i h, y0 + j h
    const int64_t j = c / gnx, i = c - j * gnx;
    xl = gx0 + (double)i * h; yl = gy0 + (double)(grow0 + j) * h;
  }
  const double g = 0.5 * h;
  const double xs[3] = {xl, xl + g, xl + h}, ys[3] = {yl, yl + g, yl + h};
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a) rays[9 * k + 3 * b + a] = make_double2(xs[a], ys[b]);
#pragma unroll
  for (int b = 0; b < 2; ++b)
#pragma unroll
    for (int a = 0; a < 2; ++a) org_out[4 * k + 2 * b + a] = make_double2(xs[a], ys[b]);
}

// Refinement, step 2: the deflected 3 x 3 grids in pixel coordinates, four
// corners (c00, c10, c11, c01) per sub-cell, sub-cell 4k + 2b + a.
__global__ void k_refine_quads(const double2* __restrict__ y, int64_t np, IpmParams ip,
                               PixCorner* __restrict__ quads) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= np * 16) return;
  const int64_t k = t >> 4;
  const int q = (int)(t & 15), sub = q >> 2, corner = q & 3;
  const int a = sub & 1, b = sub >> 1;
  // corner order c00, c10, c11, c01 of the sub-cell at (a, b)
  const int ca = a + (corner == 1 || corner == 2), cb = b + (corner >= 2);
  const double2 p = y[9 * k + 3 * cb + ca];
  const double u = (p.x - ip.u0) * ip.inv_du, v = (p.y - ip.v0) * ip.inv_dv;
  PixCorner pc;
  if (!(fabs(u) < 5.0e8) || !(fabs(v) < 5.0e8)) {
    pc.iu = kFar; pc.fu = 0.f; pc.iv = kFar; pc.fv = 0.f;
  } else {
    const double fu = floor(u), fv = floor(v);
    pc.iu = (int)fu; pc.fu = (float)(u - fu);
    pc.iv = (int)fv; pc.fv = (float)(v - fv);
    // a fraction that rounds up to 1 moves to the next pixel
    if (pc.fu >= 1.f) { pc.iu += 1; pc.fu = 0.f; }
    if (pc.fv >= 1.f) { pc.iv += 1; pc.fv = 0.f; }
  }
  quads[4 * (4 * k + sub) + corner] = pc;
}
}  // namespace

void ipm_accumulate(const PixCorner* yc, int64_t nx, int64_t nrows_cells, const IpmParams& ip,
                    float* map, float* rowdiff, double* stats_dev, int* queue, int* qcount,
                    int* rq, int* rqcount, cudaStream_t s,
                    std::vector<std::pair<cudaEvent_t, cudaEvent_t>>* ev) {
  const int64_t ncells = nx * nrows_cells;
  if (ncells <= 0) return;
  IpmArgs A{};
  A.yc = yc; A.nx = nx; A.ncells = ncells; A.map = map; A.stats = stats_dev;
  A.D = rowdiff; A.ldd = (int64_t)ip.npx + 1;
  A.queue = queue; A.qcount = qcount; A.ip = ip;
  A.wcell = 1.f;
  A.rq = rq; A.rqcount = rqcount;
  ipm_launch(A, false, qcount, s, ev);
}

void ipm_accumulate_list(const PixCorner* yc, int64_t nx, const int* list, int64_t n,
                         const IpmParams& ip, float* map, float* rowdiff, double* stats_dev,
                         int* queue, int* qcount, int* rq, int* rqcount, cudaStream_t s,
                         std::vector<std::pair<cudaEvent_t, cudaEvent_t>>* ev) {
  if (n <= 0) return;
  IpmArgs A{};
  A.yc = yc; A.nx = nx; A.ncells = n; A.cell_list = list; A.map = map; A.stats = stats_dev;
  A.D = rowdiff; A.ldd = (int64_t)ip.npx + 1;
  A.queue = queue; A.qcount = qcount; A.ip = ip;
  A.wcell = 1.f;
  A.rq = rq; A.rqcount = rqcount;
  ipm_launch(A, false, qcount, s, ev);
}

int64_t ipm_refine(Plan& P, const int* parents, int64_t np, const double2* org_in, double gx0,
                   double gy0, int64_t grow0, int64_t gnx, double h, int level,
                   const IpmParams& ip, float* map,
                   float* rowdiff, double* stats_dev, int* rq_next, int* rqcount_next,
                   double2* org_out, cudaStream_t s,
                   std::vector<std::pair<cudaEvent_t, cudaEvent_t>>* ev) {
  if (np <= 0) return 0;
  Scratch rays(&P.da, sizeof(double2) * 9 * (size_t)np);
  Scratch y(&P.da, sizeof(double2) * 9 * (size_t)np);
  Scratch quads(&P.da, sizeof(PixCorner) * 16 * (size_t)np);
  Scratch queue(&P.da, sizeof(int) * 4 * (size_t)np + sizeof(int) * 2);
  k_refine_points<<<grid_for(np, 128), 128, 0, s>>>(parents, np, org_in, gx0, gy0, grow0, gnx,
                                                     h, rays.as<double2>(), org_out);
  LENS_LAUNCHED("k_refine_points");
  evaluate_rays(P, rays.as<double>(), 9 * np, y.as<double>(), nullptr, s);
  k_refine_quads<<<grid_for(16 * np, 256), 256, 0, s>>>(y.as<double2>(), np, ip,
                                                         quads.as<PixCorner>());
  LENS_LAUNCHED("k_refine_quads");
  IpmArgs A{};
  A.yc = quads.as<PixCorner>(); A.nx = 0; A.ncells = 4 * np; A.map = map; A.stats = stats_dev;
  A.D = rowdiff; A.ldd = (int64_t)ip.npx + 1;
  A.queue = queue.as<int>(); A.qcount = queue.as<int>() + 4 * np; A.ip = ip;
  A.wcell = (float)std::ldexp(1.0, -2 * level);
  A.rq = rq_next; A.rqcount = rqcount_next;
  ipm_launch(A, true, A.qcount, s, ev);
  return 4 * np;
}

}  // namespace lens
