// adjoint.cu -- transposed FMM: gradient of a loss through Eq. 1 with respect
// to the star positions, masses, kappa_s and gamma (not in the paper; the
// forward operators are those of Appendix A, run backwards on the same tree).
//
// With f(z) = sum_j m_j/(z - z_j), alpha = conj(f) and g = dL/dy at every ray,
// dL/dalpha = -g, so dL = Re sum_r c_r df_r with the ray charge
// c_r = -(g1 + i g2).  Every forward step is complex-linear in its input, so
// its adjoint is its plain transpose (dL = Re sum_l Lhat_l dB_l):
//   L2P^T  Lhat_B,l   += sum_{r in B} c_r w_r^l           (w = (z_r - c_B)/r_B)
//   M2P^T  Mhat_C,k   += sum_{r} c_r q_r^k / (z_r - c_C)   (q = r_C/(z_r - c_C), W lists)
//   P2P^T  Phi_j      += c_r/(z_r - z_j),  Psi_j += c_r m_j/(z_r - z_j)^2   (U lists)
//   L2L^T  Lhat_P,l   += sum_{j<=l} S_q[j][l] Lhat_C,j      (children -> parent)
//   M2L^T  Mhat_C,k   += u^k sum_l C(k+l,k) (-1)^l u^(l+1) Lhat_B,l / r   (V lists)
//   P2L^T  Phi_j += sum_l Lhat_B,l (-q^l/(z_j-c)),  Psi_j += sum_l Lhat_B,l m_j (l+1) q^l/(z_j-c)^2  (X)
//   M2M^T  Mhat_C,k   += sum_{l>=k} T_q[l][k] Mhat_P,l     (parent -> children)
//   P2M^T  Phi_j += sum_k Mhat_k w_j^k,  Psi_j += m_j sum_k k Mhat_k w_j^(k-1)/r  (leaves)
// where Phi_j, Psi_j give dL/dm_j = Re Phi_j and dL/dz_j = Psi_j, i.e.
// dL/dx_j = Re Psi_j, dL/dy_j = -Im Psi_j.  The smooth field adds
// dL/dkappa_s = -sum_r (g1 x1 + g2 x2), dL/dgamma = sum_r (-g1 x1 + g2 x2).
// For float64 plans everything here is float64; float32-bulk plans run the
// per-ray and per-pair operators in float32 (below).  Deterministic up to the
// order of atomic adds.
#include <cmath>

#include "cx.cuh"
#include "lens_internal.h"

namespace lens {
namespace {

constexpr int kAdjTile = 128;  // rays per tile
// float32-bulk plans: twice that once the rays give the chip several blocks an SM all
// the same (a star's offsets and sums are formed once a tile).  P2P^T and moments at 3e6
// rays on 16 leaves 384 + 72 us (tiles of 128: 420 + 91; plain sums), at 5e5 rays 69 + 18
// (73 + 15), at 1.3e5 26 + 15 (24 + 10): the line is where the two meet.
constexpr int kAdjTile32 = 256;
constexpr int64_t kAdjLarge = 1 << 19;
constexpr int kAdjU = 64;      // U-list leaves staged at a time by k_adj_p2p32

__device__ __forceinline__ void atomic_add2(double2* p, double2 v) {
  atomicAdd(&p->x, v.x);
  atomicAdd(&p->y, v.y);
}

struct AdjArgs {
  const double* rays; const double* gy;
  const int* perm; const int64_t* ray_off; const int2* tile_leaf; int tile;
  const int* leaves; const int* aidx; const int* level; const int* ix; const int* iy;
  const int* start; const int* count; const int* child; const int* parent;
  const int64_t* U_off; const int* U_list; const int64_t* W_off; const int* W_list;
  const int64_t* V_off; const int* V_list; const int64_t* X_off; const int* X_list;
  const double2* spos; const double* smass;
  FmmTables tab;
  double lo_x, lo_y, size, isize;  // isize = 1 / size
  int p;
  double2* Lh; double2* Mh;   // adjoints of L (by box) and M (by box)
  double2* Phi; double2* Psi; // per sorted star
  double* gkg;                // [2]
};

// A box's half side, its inverse and its centre, without a division or a conversion
// on the float64 pipe (a block of few rays formed them at ~40 operations there).
__device__ __forceinline__ double box_r(const AdjArgs& A, int b) {
  return box_half(A.size, A.level[b]);
}
__device__ __forceinline__ double box_ir(const AdjArgs& A, int b) {
  return box_inv_half(A.isize, A.level[b]);
}
__device__ __forceinline__ double2 box_c(const AdjArgs& A, int b, double r) {
  return make_double2(box_centre(A.lo_x, A.ix[b], r), box_centre(A.lo_y, A.iy[b], r));
}

// One warp per (leaf, tile): L2P^T moments of the tile's rays and M2P^T for
// every W entry, accumulated per lane in shared memory, reduced, and added
// atomically (tiles of one leaf share Lhat_B).
__global__ void __launch_bounds__(32) k_adj_leaf_moments(AdjArgs A) {
  extern __shared__ double2 acc[];  // [(p+1)][32]
  const int lane = threadIdx.x;
  const int2 kt = A.tile_leaf[blockIdx.x];
  if (kt.x < 0) return;
  const int64_t k = kt.x;
  const int B = A.leaves[k];
  const int a = A.aidx[B];
  const int64_t tile = kt.y;
  const int64_t n = A.ray_off[k + 1] - A.ray_off[k];
  const int64_t r0 = tile * kAdjTile;
  const int64_t r1 = min64(n, r0 + kAdjTile);
  const int p = A.p;
  const double rB = box_r(A, B);
  const double2 cB = box_c(A, B, rB);
  const double irB = box_ir(A, B);
  // pass 0: L2P^T; pass e >= 1: M2P^T of W entry e-1
  const int64_t nW = A.W_off[a + 1] - A.W_off[a];
  for (int64_t pass = 0; pass <= nW; ++pass) {
    for (int l = 0; l <= p; ++l) acc[l * 32 + lane] = make_double2(0.0, 0.0);
    int C = -1;
    double rC = 0;
    double2 cC = make_double2(0, 0);
    if (pass > 0) {
      C = A.W_list[A.W_off[a] + pass - 1];
      rC = box_r(A, C);
      cC = box_c(A, C, rC);
    }
    for (int64_t t = r0 + lane; t < r1; t += 32) {
      const int64_t ridx = A.perm[A.ray_off[k] + t];
      const double2 z = make_double2(A.rays[2 * ridx], A.rays[2 * ridx + 1]);
      const double2 c = make_double2(-A.gy[2 * ridx], -A.gy[2 * ridx + 1]);
      double2 pw, w;
      if (pass == 0) {
        w = make_double2((z.x - cB.x) * irB, (z.y - cB.y) * irB);
        pw = c;
      } else {
        const double2 inv = cinv(make_double2(z.x - cC.x, z.y - cC.y));
        w = make_double2(inv.x * rC, inv.y * rC);
        pw = cmul(c, inv);
      }
      for (int l = 0; l <= p; ++l) {
        acc[l * 32 + lane] = acc[l * 32 + lane] + pw;
        pw = cmul(pw, w);
      }
    }
    __syncwarp();
    double2* dst = pass == 0 ? A.Lh + (int64_t)B * (p + 1) : A.Mh + (int64_t)C * (p + 1);
    for (int l = 0; l <= p; ++l) {
      double2 v = acc[l * 32 + lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      }
      if (lane == 0 && (v.x != 0.0 || v.y != 0.0)) atomic_add2(dst + l, v);
    }
    __syncwarp();
  }
}

// The stars of a leaf's U list, flattened over the block's threads (a leaf's own
// count is often below the block size): up to kAdjU leaves at a time, their first
// star and inclusive star counts in shared memory.  f(sj, h) is called for every
// star of the list by S neighbouring lanes, h = 0 .. S - 1.
struct UStage {
  int start[kAdjU], incl[kAdjU];
};
template <int S, typename F>
__device__ __forceinline__ void for_u_stars(const AdjArgs& A, int a, UStage& su, F f) {
  const int64_t u0 = A.U_off[a], nu = A.U_off[a + 1] - u0;
  for (int64_t ub = 0; ub < nu; ub += kAdjU) {
    const int nub = (int)min64(kAdjU, nu - ub);
    __syncthreads();  // the previous group's readers are done (and the caller's staging)
    if (threadIdx.x < nub) {
      const int C = A.U_list[u0 + ub + threadIdx.x];
      su.start[threadIdx.x] = A.start[C];
      su.incl[threadIdx.x] = A.count[C];
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int i = 1; i < nub; ++i) su.incl[i] += su.incl[i - 1];
    __syncthreads();
    const int tot = su.incl[nub - 1];
    for (int qs = threadIdx.x; qs < tot * S; qs += blockDim.x) {
      const int q = qs / S;
      // the group's leaf holding flattened star q: the first with incl > q
      int lo = 0, hi = nub - 1;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (su.incl[mid] > q) hi = mid; else lo = mid + 1;
      }
      f(su.start[lo] + q - (lo ? su.incl[lo - 1] : 0), qs % S);
    }
  }
}

// P2P^T in float64: threads over the U-list stars of the tile's leaf, the tile's
// rays staged in shared memory.  Bound by the float64 pipe: 21 operations a pair
// (with a division and comparisons with 0 on that pipe, ~30), a warp
// instruction for up to 32 stars (one leaf at a time, ~11).  1.26e5 rays, 2e4
// stars, leaves of 16: 1781 -> 306 us.
__global__ void __launch_bounds__(128) k_adj_p2p(AdjArgs A) {
  __shared__ double2 sz[kAdjTile], sc[kAdjTile];
  __shared__ UStage su;
  const int2 kt = A.tile_leaf[blockIdx.x];
  if (kt.x < 0) return;
  const int64_t k = kt.x;
  const int a = A.aidx[A.leaves[k]];
  const int64_t tile = kt.y;
  const int64_t n = A.ray_off[k + 1] - A.ray_off[k];
  const int64_t r0 = tile * kAdjTile;
  const int nr = (int)min64(kAdjTile, n - r0);
  for (int t = threadIdx.x; t < nr; t += blockDim.x) {
    const int64_t ridx = A.perm[A.ray_off[k] + r0 + t];
    sz[t] = make_double2(A.rays[2 * ridx], A.rays[2 * ridx + 1]);
    sc[t] = make_double2(-A.gy[2 * ridx], -A.gy[2 * ridx + 1]);
  }
  for_u_stars<1>(A, a, su, [&](int sj, int) {
    const double2 zj = A.spos[sj];
    double2 F = make_double2(0, 0), G = make_double2(0, 0);
#pragma unroll 2
    for (int t = 0; t < nr; ++t) {
      const double2 d = make_double2(sz[t].x - zj.x, sz[t].y - zj.y);
      const double r2 = d.x * d.x + d.y * d.y;
      double w;
      if (rcp_in_range(r2)) w = rcp_newton(r2);
      else if (r2 == 0.0) continue;  // self-interaction, whatever the charge
      else w = 1.0 / r2;
      const double2 inv = make_double2(d.x * w, -d.y * w);
      const double2 ci = cmul(sc[t], inv);
      F = F + ci;
      G = cfma(ci, inv, G);
    }
    const double mj = A.smass[sj];
    atomic_add2(A.Phi + sj, F);
    atomic_add2(A.Psi + sj, make_double2(mj * G.x, mj * G.y));
  });
}

// ---- float32 bulk (plans of precision LENS_FP32_BULK) ------------------------
// The per-ray and per-pair parts of the adjoint in float32, as the forward
// pass evaluates them: P2P^T on float-float offsets from the leaf centre
// (each pair's difference exact to float32 rounding however close a ray is
// to a star), partial sums compensated; L2P^T / M2P^T moments with the
// scaled offsets w rounded once to float32 (|w| <= ~1.5: no cancellation),
// summed per lane and across lanes compensated.  The transposed
// translations (L2L^T, M2L^T, P2L^T, M2M^T, P2M^T) stay float64.

// P2P^T: block per (leaf, tile of rays), four lanes a star over the U-list stars, each
// with every fourth pair of the tile's rays, staged as float-float offsets from
// the leaf centre with their float32 charges; two rays an instruction (paired
// float32), the four lanes' sums combined in float-float.  Bound by the FMA
// pipe and issue: 12 products and differences and 28 operations of compensated
// sums a pair of points.  A lane a star left a third of the lanes idle at ~70 stars a
// list: 3e6 rays, p 24, leaves of 16: 530 -> 420 us,
// tiles of 256 rays 384.
constexpr int kStarLanes = 4;

__device__ __forceinline__ ff lanes_sum(const fcomp2& a) {
  ff u, v;
  two_sum(a.hi.x, a.lo.x, u.hi, u.lo);
  two_sum(a.hi.y, a.lo.y, v.hi, v.lo);
  return ff_add(u, v);
}
__device__ __forceinline__ ff ff_shfl_xor(unsigned mask, ff a, int o) {
  return ff{__shfl_xor_sync(mask, a.hi, o), __shfl_xor_sync(mask, a.lo, o)};
}

__global__ void __launch_bounds__(128) k_adj_p2p32(AdjArgs A) {
  // pairs of rays: x, x, -y, -y (high and low parts), charges, -c.y
  __shared__ float4 szh[kAdjTile32 / 2], szl[kAdjTile32 / 2], sc[kAdjTile32 / 2];
  __shared__ float2 snc[kAdjTile32 / 2];
  const int2 kt = A.tile_leaf[blockIdx.x];
  if (kt.x < 0) return;
  const int64_t k = kt.x;
  const int B = A.leaves[k];
  const int a = A.aidx[B];
  const int64_t tile = kt.y;
  const int64_t n = A.ray_off[k + 1] - A.ray_off[k];
  const int64_t r0 = tile * A.tile;
  const int nr = (int)min64(A.tile, n - r0);
  const int np = (nr + 2 * kStarLanes - 1) / (2 * kStarLanes) * kStarLanes;  // pairs, whole rounds
  const double rB = box_r(A, B);
  const double2 cB = box_c(A, B, rB);
  for (int t = threadIdx.x; t < 2 * np; t += blockDim.x) {
    ff ox{1e18f, 0.f}, oy{1e18f, 0.f};  // beyond the tile: far, no charge
    float c1 = 0.f, c2 = 0.f;
    if (t < nr) {
      const int64_t ridx = A.perm[A.ray_off[k] + r0 + t];
      ox = ff_of(A.rays[2 * ridx] - cB.x);
      oy = ff_of(A.rays[2 * ridx + 1] - cB.y);
      c1 = -d2f(A.gy[2 * ridx]);
      c2 = -d2f(A.gy[2 * ridx + 1]);
    }
    float* h = reinterpret_cast<float*>(szh + (t >> 1)) + (t & 1);
    float* l = reinterpret_cast<float*>(szl + (t >> 1)) + (t & 1);
    float* c = reinterpret_cast<float*>(sc + (t >> 1)) + (t & 1);
    h[0] = ox.hi; h[2] = -oy.hi;
    l[0] = ox.lo; l[2] = -oy.lo;
    c[0] = c1; c[2] = c2;
    reinterpret_cast<float*>(snc + (t >> 1))[t & 1] = -c2;
  }
  __shared__ UStage su;
  for_u_stars<kStarLanes>(A, a, su, [&](int sj, int h) {
    const double2 zj = A.spos[sj];
    const ff sx = ff_of(zj.x - cB.x), sy = ff_of(zj.y - cB.y);
    const float2 xh = make_float2(-sx.hi, -sx.hi), xl = make_float2(-sx.lo, -sx.lo);
    const float2 yh = make_float2(sy.hi, sy.hi), yl = make_float2(sy.lo, sy.lo);
    const float2 tiny = make_float2(1e-30f, 1e-30f), m1 = make_float2(-1.f, -1.f);
    const float2 zero = make_float2(0.f, 0.f);
    fcomp2 F1{zero, zero}, F2{zero, zero}, G1{zero, zero}, G2{zero, zero};
    for (int i = h; i < np; i += kStarLanes) {
      const float4 zh = szh[i], zl = szl[i], c4 = sc[i];
      const float2 cx = make_float2(c4.x, c4.y), cy = make_float2(c4.z, c4.w), ncy = snc[i];
      // d = z_r - z_j; 1/d = conj(d) / |d|^2 (a star exactly at the ray adds
      // nothing: d = 0 makes both terms 0 under the floor on |d|^2)
      const float2 d1 = __fadd2_rn(__fadd2_rn(make_float2(zh.x, zh.y), xh),
                                   __fadd2_rn(make_float2(zl.x, zl.y), xl));
      const float2 n2 = __fadd2_rn(__fadd2_rn(make_float2(zh.z, zh.w), yh),  // -d2
                                   __fadd2_rn(make_float2(zl.z, zl.w), yl));
      const float2 q = __ffma2_rn(d1, d1, __ffma2_rn(n2, n2, tiny));
      const float2 w = make_float2(frcp_fast(q.x), frcp_fast(q.y));
      const float2 i1 = __fmul2_rn(d1, w), i2 = __fmul2_rn(n2, w), mi2 = __fmul2_rn(i2, m1);
      const float2 c1 = __ffma2_rn(cx, i1, __fmul2_rn(ncy, i2));  // c / d
      const float2 c2 = __ffma2_rn(cx, i2, __fmul2_rn(cy, i1));
      F1.add(c1); F2.add(c2);
      G1.add(__ffma2_rn(c1, i1, __fmul2_rn(c2, mi2)));            // c / d^2
      G2.add(__ffma2_rn(c1, i2, __fmul2_rn(c2, i1)));
    }
    // lane h ends with one of F1, G1, F2, G2 (its bits: G, second component)
    const unsigned mask = 0xfu << (threadIdx.x & 28u);
    const ff f1 = lanes_sum(F1), f2s = lanes_sum(F2), g1 = lanes_sum(G1), g2 = lanes_sum(G2);
    const bool bg = h & 1, b2 = h & 2;
    const ff k0 = ff_add(bg ? g1 : f1, ff_shfl_xor(mask, bg ? f1 : g1, 1));
    const ff k1 = ff_add(bg ? g2 : f2s, ff_shfl_xor(mask, bg ? f2s : g2, 1));
    const ff v = ff_add(b2 ? k1 : k0, ff_shfl_xor(mask, b2 ? k0 : k1, 2));
    double2* dst = (bg ? A.Psi : A.Phi) + sj;
    double x = ff_to_double(v);
    if (bg) x *= A.smass[sj];
    atomicAdd(b2 ? &dst->y : &dst->x, x);
  });
}

// a b, each component's fused product fixed: the same bits wherever it is inlined
__device__ __forceinline__ float2 cmul_fixed(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.y, b.x, __fmul_rn(a.x, b.y)));
}

// L2P^T and M2P^T moments in float32: one warp per (leaf, tile), as
// k_adj_leaf_moments.  A lane takes four rays at a time (a trip to shared memory per
// order and four rays) and compensates every sum: the terms of a tile cancel, so
// roundings of plain partial sums were most of the gradient's own spread
// (3e6 rays, p 24: 72 us with plain sums, 113 so).
constexpr int kMomRays = 4;
// a + b + c + d, the sum's head and its errors
__device__ __forceinline__ ff sum4(float a, float b, float c, float d) {
  float s, t, e, f, g, r;
  two_sum(a, b, s, e);
  two_sum(c, d, t, f);
  two_sum(s, t, r, g);
  return ff{r, g + (e + f)};
}
__global__ void __launch_bounds__(32) k_adj_leaf_moments32(AdjArgs A) {
  extern __shared__ float4 acc32[];  // [(p+1)][33]: lane partials (x, y, and their errors), padded
  const int lane = threadIdx.x;
  const int2 kt = A.tile_leaf[blockIdx.x];
  if (kt.x < 0) return;
  const int64_t k = kt.x;
  const int B = A.leaves[k];
  const int a = A.aidx[B];
  const int64_t tile = kt.y;
  const int64_t n = A.ray_off[k + 1] - A.ray_off[k];
  const int64_t r0 = tile * A.tile;
  const int64_t r1 = min64(n, r0 + A.tile);
  const int p = A.p;
  const double rB = box_r(A, B);
  const double2 cB = box_c(A, B, rB);
  const double irB = box_ir(A, B);
  const int64_t nW = A.W_off[a + 1] - A.W_off[a];
  for (int64_t pass = 0; pass <= nW; ++pass) {
    for (int l = 0; l <= p; ++l) acc32[l * 33 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    int C = -1;
    double rC = 0;
    double2 cC = make_double2(0, 0);
    if (pass > 0) {
      C = A.W_list[A.W_off[a] + pass - 1];
      rC = box_r(A, C);
      cC = box_c(A, C, rC);
    }
    for (int64_t t = r0 + lane; t < r1; t += 32 * kMomRays) {
      float2 pw[kMomRays], w[kMomRays];
#pragma unroll
      for (int q = 0; q < kMomRays; ++q) {
        pw[q] = w[q] = make_float2(0.f, 0.f);
        if (t + 32 * q >= r1) continue;
        const int64_t ridx = A.perm[A.ray_off[k] + t + 32 * q];
        const float2 c = make_float2(-d2f(A.gy[2 * ridx]), -d2f(A.gy[2 * ridx + 1]));
        if (pass == 0) {
          w[q] = make_float2(d2f((A.rays[2 * ridx] - cB.x) * irB),
                             d2f((A.rays[2 * ridx + 1] - cB.y) * irB));
          pw[q] = c;
        } else {
          const float2 inv = cinv(make_float2(d2f(A.rays[2 * ridx] - cC.x),
                                              d2f(A.rays[2 * ridx + 1] - cC.y)));
          w[q] = make_float2(inv.x * (float)rC, inv.y * (float)rC);
          pw[q] = cmul(c, inv);
        }
      }
      for (int l = 0; l <= p; ++l) {
        float4 a4 = acc32[l * 33 + lane];
        const ff x = sum4(pw[0].x, pw[1].x, pw[2].x, pw[3].x), y = sum4(pw[0].y, pw[1].y, pw[2].y, pw[3].y);
        float e1, e2;
        two_sum(a4.x, x.hi, a4.x, e1);
        two_sum(a4.y, y.hi, a4.y, e2);
        a4.z += e1 + x.lo;
        a4.w += e2 + y.lo;
        acc32[l * 33 + lane] = a4;
#pragma unroll
        for (int q = 0; q < kMomRays; ++q) pw[q] = cmul_fixed(pw[q], w[q]);
      }
    }
    __syncwarp();
    double2* dst = pass == 0 ? A.Lh + (int64_t)B * (p + 1) : A.Mh + (int64_t)C * (p + 1);
    // lane l sums order l's 32 lane partials, compensated (~48 bits): in
    // float64 the additions and conversions were most of the kernel's time
    // (3e6 rays, p 24: with the tile's box constants, 260 -> 91 us)
    for (int l = lane; l <= p; l += 32) {
      fcomp vx{0.f, 0.f}, vy{0.f, 0.f};
      for (int q = 0; q < 32; ++q) {
        const float4 vf = acc32[l * 33 + q];
        vx.add(vf.x);
        vy.add(vf.y);
        vx.lo += vf.z;
        vy.lo += vf.w;
      }
      const double2 v = make_double2(vx.value(), vy.value());
      if (v.x != 0.0 || v.y != 0.0) atomic_add2(dst + l, v);
    }
    __syncwarp();
  }
}

// L2L^T for one level: warp per active child box, adds into its parent.
__global__ void __launch_bounds__(128) k_adj_l2l(AdjArgs A, const int* active, int64_t a0, int64_t a1) {
  const int lane = threadIdx.x & 31;
  const int64_t ai = a0 + (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32;
  if (ai >= a1) return;
  const int C = active[ai];
  const int P = A.parent[C];
  const int q = C - A.child[P];
  const int P1 = A.p + 1;
  const double2* S = A.tab.l2l + (int64_t)q * P1 * P1;
  const double2* Lc = A.Lh + (int64_t)C * P1;
  for (int l = lane; l <= A.p; l += 32) {
    double2 v = make_double2(0, 0);
    for (int j = 0; j <= l; ++j) v = cfma(S[j * P1 + l], Lc[j], v);
    if (v.x != 0.0 || v.y != 0.0) atomic_add2(A.Lh + (int64_t)P * P1 + l, v);
  }
}

// M2L^T (V) and P2L^T (X): block per active box, its warps taking the V entries
// and the X stars in turn (a warp per box left a small target region, a few
// dozen boxes of ~27 entries each, on as many warps: 124 ->
// 30 us at p 24).
constexpr int kAdjM2lWarps = 8;
__global__ void __launch_bounds__(32 * kAdjM2lWarps)
k_adj_m2l(AdjArgs A, const int* active, int64_t na) {
  __shared__ double2 sbuf[kAdjM2lWarps][kMaxOrder + 2];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t ai = blockIdx.x;
  const int B = active[ai];
  const int p = A.p, P1 = p + 1;
  const double r = box_r(A, B);
  const double ir = 1.0 / r;
  const double2 cB = box_c(A, B, r);
  const double2* Lb = A.Lh + (int64_t)B * P1;
  double2* buf = sbuf[wib];
  for (int64_t e = A.V_off[ai] + wib; e < A.V_off[ai + 1]; e += kAdjM2lWarps) {
    const int C = A.V_list[e];
    const int dx = A.ix[C] - A.ix[B], dy = A.iy[C] - A.iy[B];
    const double2* up = A.tab.upow + (int64_t)((dy + 3) * 7 + (dx + 3)) * (p + 2);
    for (int l = lane; l <= p; l += 32) {
      double2 v = cmul(Lb[l], up[l + 1]);
      if (l & 1) v = make_double2(-v.x, -v.y);
      buf[l] = make_double2(v.x * ir, v.y * ir);
    }
    __syncwarp();
    for (int kk = lane; kk <= p; kk += 32) {
      double sx = 0, sy = 0;
      for (int l = 0; l <= p; ++l) {
        const double c = A.tab.binom[(int64_t)(kk + l) * A.tab.ldb + l];  // C(k+l, l)
        sx = fma(c, buf[l].x, sx);
        sy = fma(c, buf[l].y, sy);
      }
      const double2 v = cmul(up[kk], make_double2(sx, sy));
      if (v.x != 0.0 || v.y != 0.0) atomic_add2(A.Mh + (int64_t)C * P1 + kk, v);
    }
    __syncwarp();
  }
  for (int64_t e = A.X_off[ai]; e < A.X_off[ai + 1]; ++e) {
    const int C = A.X_list[e];
    for (int j = A.start[C] + wib; j < A.start[C] + A.count[C]; j += kAdjM2lWarps) {
      const double2 z = A.spos[j];
      const double m = A.smass[j];
      const double2 inv = cinv(make_double2(z.x - cB.x, z.y - cB.y));
      const double2 q = make_double2(inv.x * r, inv.y * r);
      double2 F = make_double2(0, 0), G = make_double2(0, 0);
      for (int l = lane; l <= p; l += 32) {
        double2 pw = make_double2(1.0, 0.0), bse = q;
        for (int e2 = l; e2 > 0; e2 >>= 1) {
          if (e2 & 1) pw = cmul(pw, bse);
          bse = cmul(bse, bse);
        }
        const double2 t = cmul(Lb[l], pw);
        F = F + t;
        G = G + make_double2((l + 1) * t.x, (l + 1) * t.y);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        F.x += __shfl_xor_sync(0xffffffffu, F.x, o); F.y += __shfl_xor_sync(0xffffffffu, F.y, o);
        G.x += __shfl_xor_sync(0xffffffffu, G.x, o); G.y += __shfl_xor_sync(0xffffffffu, G.y, o);
      }
      if (lane == 0) {
        const double2 Fj = cmul(F, inv);                 // sum Lhat q^l / (z - c)
        const double2 Gj = cmul(G, cmul(inv, inv));      // sum Lhat (l+1) q^l / (z - c)^2
        atomic_add2(A.Phi + j, make_double2(-Fj.x, -Fj.y));
        atomic_add2(A.Psi + j, make_double2(m * Gj.x, m * Gj.y));
      }
    }
  }
}

// M2M^T for one level, the children in groups of four, one thread per (parent,
// coefficient k).  The child offsets d_q = w i^m_q (w = (1+i)/2, m_q = 2, 3, 1, 0)
// enter through powers of i alone, as in the M2M:
//   Mhat_C,k += conj(w)^k sum_l i^(m (l-k)) C(l, k) w^l Mhat_P,l
//            = conj(w)^k sum_r i^(m r) G_r[k],  G_r[k] the terms with l - k = r mod 4,
// one real binomial sum and additions for four children.  Float64 pipe; with a
// complex matrix per child, a warp a box and half of its lanes past the
// triangle's edge: 1e5 stars, p 24: 172 -> 82 us.
constexpr int kAdjM2mThreads = 128;

__global__ void __launch_bounds__(kAdjM2mThreads)
k_adj_m2m(AdjArgs A, int64_t c0, int64_t ngroups) {
  extern __shared__ double2 Wp[];  // [parents per block][p+1], then the binomials
  const int p = A.p, P1 = p + 1;
  const int per = kAdjM2mThreads / P1;
  const int t = threadIdx.x, pb = t / P1, k = t - pb * P1;
  // C(l, k), k <= l, as [k][l - k]: row k from k (2 p + 3 - k) / 2
  double* cb = reinterpret_cast<double*>(Wp + (int64_t)per * P1);
  for (int i = t; i < P1 * P1; i += kAdjM2mThreads) {
    const int kk = i / P1, l = i - kk * P1;
    if (l >= kk) cb[kk * (2 * p + 3 - kk) / 2 + l - kk] = A.tab.binom[(int64_t)l * A.tab.ldb + kk];
  }
  const int64_t g = (int64_t)blockIdx.x * per + pb;
  const bool on = pb < per && g < ngroups;
  const int64_t c = c0 + 4 * g;  // first child of the group
  double2 w = make_double2(0.0, 0.0);
  if (on) {
    w = A.tab.wpow[k];
    Wp[pb * P1 + k] = cmul(w, A.Mh[(int64_t)A.parent[c] * P1 + k]);
  }
  __syncthreads();
  if (!on) return;
  const double* crow = cb + k * (2 * p + 3 - k) / 2;
  const double2* Wk = Wp + pb * P1 + k;
  double2 G[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) G[r] = make_double2(0.0, 0.0);
  for (int t0 = 0; t0 <= p - k; t0 += 4) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (t0 + r <= p - k) {
        G[r].x = fma(crow[t0 + r], Wk[t0 + r].x, G[r].x);
        G[r].y = fma(crow[t0 + r], Wk[t0 + r].y, G[r].y);
      }
    }
  }
  const double2 s02 = G[0] + G[2], d02 = G[0] - G[2], s13 = G[1] + G[3], d13 = G[1] - G[3];
  const double2 cw = make_double2(w.x, -w.y);
  // sum_r i^(m r) G_r for m = 2, 3, 1, 0
  const double2 f[4] = {s02 - s13, make_double2(d02.x + d13.y, d02.y - d13.x),
                        make_double2(d02.x - d13.y, d02.y + d13.x), s02 + s13};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (A.count[c + q] == 0) continue;
    double2* o = A.Mh + (c + q) * P1 + k;
    *o = *o + cmul(cw, f[q]);
  }
}

// P2M^T at the stars of every leaf, G lanes a leaf (a thread a leaf ran its stars
// one after another, ~25 dependent float64 steps each: 161 -> 29 us at 2e4
// stars, leaves of 16, p 24).  Horner's rule
// for the sum and its derivative side by side.
template <int G>
__global__ void __launch_bounds__(128) k_adj_p2m(AdjArgs A, int64_t nb) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t b = t / G;
  if (b >= nb || A.child[b] >= 0 || A.count[b] == 0) return;
  const int p = A.p, P1 = p + 1;
  const double r = box_r(A, (int)b);
  const double2 c = box_c(A, (int)b, r);
  const double ir = box_ir(A, (int)b);
  const double2* Mb = A.Mh + b * P1;
  const int s0 = A.start[b], s1 = s0 + A.count[b];
  for (int j = s0 + (int)(t % G); j < s1; j += G) {
    const double2 z = A.spos[j];
    const double m = A.smass[j];
    const double2 w = make_double2((z.x - c.x) * ir, (z.y - c.y) * ir);
    double2 F = Mb[p], D = make_double2(0.0, 0.0);  // sum, derivative in w
    for (int kk = p - 1; kk >= 0; --kk) {
      D = cfma(D, w, F);
      F = cfma(F, w, Mb[kk]);
    }
    A.Phi[j] = A.Phi[j] + F;
    A.Psi[j] = A.Psi[j] + make_double2(m * D.x * ir, m * D.y * ir);
  }
}

__global__ void k_adj_kg(const double* rays, const double* gy, int64_t m, const int64_t* bad,
                         double* gkg) {
  if (*bad) return;  // the call is refused
  __shared__ double sh[2][256];
  double sk = 0, sg = 0;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < m;
       r += (int64_t)gridDim.x * blockDim.x) {
    const double x1 = rays[2 * r], x2 = rays[2 * r + 1], g1 = gy[2 * r], g2 = gy[2 * r + 1];
    sk -= g1 * x1 + g2 * x2;
    sg += -g1 * x1 + g2 * x2;
  }
  sh[0][threadIdx.x] = sk; sh[1][threadIdx.x] = sg;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) { sh[0][threadIdx.x] += sh[0][threadIdx.x + o]; sh[1][threadIdx.x] += sh[1][threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { atomicAdd(&gkg[0], sh[0][0]); atomicAdd(&gkg[1], sh[1][0]); }
}

__global__ void k_adj_out(const double2* Phi, const double2* Psi, const uint32_t* sidx, int64_t n,
                          const int64_t* bad, double* gxy, double* gm) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n || *bad) return;
  const int64_t j = sidx[i];
  if (gm) gm[j] = Phi[i].x;
  if (gxy) { gxy[2 * j] = Psi[i].x; gxy[2 * j + 1] = -Psi[i].y; }
}

}  // namespace

void adjoint(Plan& P, const double* rays, int64_t m, const double* gy, double* gxy, double* gm,
             double* gkg, cudaStream_t s) {
  const int P1 = P.p + 1;
  wait_tree(P, s);  // the transposed operators need the tree, not the expansions
  if (gkg) LENS_CUDA(cudaMemsetAsync(gkg, 0, sizeof(double) * 2, s));
  if (m == 0) {
    if (gm) LENS_CUDA(cudaMemsetAsync(gm, 0, sizeof(double) * P.n, s));
    if (gxy) LENS_CUDA(cudaMemsetAsync(gxy, 0, sizeof(double) * 2 * P.n, s));
    return;
  }
  RayBuckets RB;
  const bool f32 = P.prec == LENS_FP32_BULK;
  const int tile = f32 && m >= kAdjLarge ? kAdjTile32 : kAdjTile;
  bucket_rays(P, rays, m, tile, RB, s);
  Scratch tl = tile_leaves(P, RB.toff, P.n_active_leaves, RB.tiles_max, s, RB.bad);
  Scratch Lh(&P.da, sizeof(double2) * (size_t)P.nb * P1);
  Scratch Mh(&P.da, sizeof(double2) * (size_t)P.nb * P1);
  Scratch Phi(&P.da, sizeof(double2) * (size_t)P.n), Psi(&P.da, sizeof(double2) * (size_t)P.n);
  LENS_CUDA(cudaMemsetAsync(Lh.p, 0, Lh.bytes, s));
  LENS_CUDA(cudaMemsetAsync(Mh.p, 0, Mh.bytes, s));
  LENS_CUDA(cudaMemsetAsync(Phi.p, 0, Phi.bytes, s));
  LENS_CUDA(cudaMemsetAsync(Psi.p, 0, Psi.bytes, s));
  AdjArgs A{};
  A.rays = rays; A.gy = gy;
  A.perm = RB.perm.as<int>(); A.ray_off = RB.off;
  A.tile_leaf = tl.as<int2>();
  A.tile = tile;
  A.leaves = P.active_leaves; A.aidx = P.box_aidx; A.level = P.box_level; A.ix = P.box_ix;
  A.iy = P.box_iy; A.start = P.box_start; A.count = P.box_count; A.child = P.box_child;
  A.parent = P.box_parent;
  A.U_off = P.U_off; A.U_list = P.U_list; A.W_off = P.W_off; A.W_list = P.W_list;
  A.V_off = P.V_off; A.V_list = P.V_list; A.X_off = P.X_off; A.X_list = P.X_list;
  A.spos = P.spos; A.smass = P.smass; A.tab = P.tab;
  A.lo_x = P.root_lo[0]; A.lo_y = P.root_lo[1]; A.size = P.root_size; A.isize = 1.0 / P.root_size; A.p = P.p;
  A.Lh = Lh.as<double2>(); A.Mh = Mh.as<double2>();
  A.Phi = Phi.as<double2>(); A.Psi = Psi.as<double2>();
  const unsigned tiles = (unsigned)RB.tiles_max;
  if (f32) {
    const size_t smem = sizeof(float4) * (size_t)P1 * 33;
    k_adj_leaf_moments32<<<tiles, 32, smem, s>>>(A);
    LENS_LAUNCHED("k_adj_leaf_moments32");
    k_adj_p2p32<<<tiles, 128, 0, s>>>(A);
    LENS_LAUNCHED("k_adj_p2p32");
  } else {
    const size_t smem = sizeof(double2) * (size_t)P1 * 32;
    if (smem > 48 * 1024)
      LENS_CUDA(cudaFuncSetAttribute(k_adj_leaf_moments, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    k_adj_leaf_moments<<<tiles, 32, smem, s>>>(A);
    LENS_LAUNCHED("k_adj_leaf_moments");
    k_adj_p2p<<<tiles, 128, 0, s>>>(A);
    LENS_LAUNCHED("k_adj_p2p");
  }
  // L2L^T, finest level first (levels >= 2 carry L2L)
  for (int l = P.nlevels - 1; l >= 2; --l) {
    const int64_t a0 = P.active_level_off[l], a1 = P.active_level_off[l + 1];
    if (a1 <= a0) continue;
    k_adj_l2l<<<grid_for((a1 - a0) * 32, 128), 128, 0, s>>>(A, P.active, a0, a1);
    LENS_LAUNCHED("k_adj_l2l");
  }
  if (P.n_active > 0) {
    k_adj_m2l<<<(unsigned)P.n_active, 32 * kAdjM2lWarps, 0, s>>>(A, P.active, P.n_active);
    LENS_LAUNCHED("k_adj_m2l");
  }
  // M2M^T, coarsest level first
  const int per = kAdjM2mThreads / P1;
  const size_t sm2 = sizeof(double2) * (size_t)per * P1 + sizeof(double) * (size_t)P1 * (P1 + 1) / 2;
  for (int l = 1; l < P.nlevels; ++l) {
    const int64_t b0 = P.level_off[l], ng = (P.level_off[l + 1] - b0) / 4;
    if (ng <= 0) continue;
    k_adj_m2m<<<grid_for(ng, per), kAdjM2mThreads, sm2, s>>>(A, b0, ng);
    LENS_LAUNCHED("k_adj_m2m");
  }
  if (P.leaf <= 8) k_adj_p2m<8><<<grid_for(P.nb * 8, 128), 128, 0, s>>>(A, P.nb);
  else if (P.leaf <= 16) k_adj_p2m<16><<<grid_for(P.nb * 16, 128), 128, 0, s>>>(A, P.nb);
  else k_adj_p2m<32><<<grid_for(P.nb * 32, 128), 128, 0, s>>>(A, P.nb);
  LENS_LAUNCHED("k_adj_p2m");
  if (gkg) {
    k_adj_kg<<<grid_for(m, 256, 1024), 256, 0, s>>>(rays, gy, m, RB.bad, gkg);
    LENS_LAUNCHED("k_adj_kg");
  }
  if (gxy || gm) {
    k_adj_out<<<grid_for(P.n, 256), 256, 0, s>>>(Phi.as<double2>(), Psi.as<double2>(), P.sidx, P.n,
                                                 RB.bad, gxy, gm);
    LENS_LAUNCHED("k_adj_out");
  }
  check_rays(RB);
}

}  // namespace lens
