// potential.cu -- the lensing potential psi(x) = sum_i m_i ln|x - x_i| +
// kappa_s |x|^2 / 2 + gamma (x1^2 - x2^2) / 2, whose gradient is x - y
// (Eq. 1 with its smooth field), through the plan's expansions (the
// potential of Sec. 2.5's lens; Appendix A's expansions of the complex
// logarithm, Greengard & Rokhlin 1987).
//
// With Phi(z) = sum_j m_j log(z - z_j), psi = Re Phi + smooth, and Phi' = f,
// the Cauchy sum the plan expands.  So the potential needs no new
// expansions, only their integrals and one real constant per box:
//   multipole  Phi(z) = a_0 log(z-c) - sum_{k>=1} a_k / (k (z-c)^k)
//   local      Phi(z) = c_B + sum_l b_l (z-c)^(l+1) / (l+1)
// (a_k, b_l the plan's field coefficients; stored scaled, A_k = a_k / r^k,
// B_l = b_l r^l).  The constant c_B = Re Phi_far(c_B) collects
//   M2L  over V:  a_0 ln|t| - Re sum_{k>=1} (A_k / k) u^k,  t = c_B - c_C, u = r / t
//   P2L  over X:  sum_j m_j ln|c_B - z_j|
//   L2L  from the parent P:  c_P + r_P Re sum_l B^P_l d^(l+1) / (l+1),
//        d = (c_B - c_P) / r_P = (+-1 +-i) / 2
// and a ray z in leaf B (half-side r, w = (z - c_B) / r) gets
//   L2P  c_B + r Re sum_l B_l w^(l+1) / (l+1)
//   P2P  over U (the leaf itself included): sum_j m_j ln|z - z_j| (a star
//        exactly at the ray contributes nothing)
//   M2P  over W:  a_0 ln|z - c_C| - Re sum_{k>=1} (A_k / k) (r_C / (z - c_C))^k
// All float64, so what counts is float64 operations (a warp-wide one takes a
// sub-partition ~77 cycles).  A thread takes a ray, the rays in leaf order
// (bucketed as the deflection's ray path does), so that the lanes of a warp share
// their leaf's lists and stars; the leaf's centre, scale, constant and
// integrated expansion are formed once per leaf.  With equal masses the near
// field's logarithms are one: the squared distances' exponents add up as
// integers and their mantissas multiply.  1e5 stars, leaves of 8, 2.6e5 rays: 1392
// -> 474 us a call (a logarithm per 8 stars, float64 range checks, divisions per ray
// and a launch per level for the constants before).  Not kept: a block per
// leaf and 128 of its rays with everything staged in shared memory (744 us
// against 635 for the same sums: partly filled warps cost as much as full ones).
// The constant c_B is formed as one increment per active box (its V and X
// lists and its parent's expansion at its centre), summed up the ancestors of
// each leaf.
#include "cx.cuh"
#include "potential.h"

namespace lens {
namespace {

struct PotArgs {
  int p;
  double lo_x, lo_y, size;
  const int* level; const int* ix; const int* iy; const int* parent; const int* child;
  const int* aidx; const int* start; const int* count; const int* active;
  const double2* spos; const double* smass;
  const double2* M; const double2* L;
  const int64_t* V_off; const int* V_list; const int64_t* X_off; const int* X_list;
  const int64_t* U_off; const int* U_list; const int64_t* W_off; const int* W_list;
  double* c0;  // per active box
  double ks, g;
  double m0;  // the mass of every star, if all are equal
};

__device__ __forceinline__ double half_side(const PotArgs& A, int level) {
  return A.size / (double)(2ull << level);
}
__device__ __forceinline__ double2 centre(const PotArgs& A, int b, double r) {
  return make_double2(A.lo_x + (2.0 * A.ix[b] + 1.0) * r, A.lo_y + (2.0 * A.iy[b] + 1.0) * r);
}
// 1/k for k = 0 .. n-1 in shared memory (1/0 unused); block-cooperative
constexpr int kPotInv = kMaxOrder + 2;
__device__ __forceinline__ void fill_inv(double* inv, int n) {
  for (int k = threadIdx.x; k < n; k += blockDim.x) inv[k] = k ? 1.0 / (double)k : 0.0;
  __syncthreads();
}

// sum of ln d2 over positive d2: exponents summed as integers, mantissas
// multiplied (each in [1, 2), so up to kLogRun of them stay in range); zeros are
// left out, subnormal and non-finite values take their own logarithm.  The sum of the
// exponents is kept as 2^16 e16 + e: a near field of millions of stars goes beyond 32
// bits, a run does not.
constexpr int kLogRun = 512;
struct LogSum {
  double prod = 1.0, rest = 0.0;
  int e16 = 0, e = 0, n = 0;
  __device__ __forceinline__ void add(double d2) {
    const int hi = __double2hiint(d2);
    if ((unsigned)hi - 0x00100000u < 0x7ff00000u - 0x00100000u) {
      e += (hi >> 20) - 1023;
      prod *= __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(d2));
      if (++n == kLogRun) fold();
    } else if (d2 > 0.0) {
      rest += log(d2);
    }
  }
  __device__ __forceinline__ void fold() {  // prod back to [1, 2)
    const int hi = __double2hiint(prod);
    e += (hi >> 20) - 1023;
    e16 += e >> 16;
    e &= 0xffff;
    n = 0;
    prod = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(prod));
  }
  __device__ __forceinline__ double value() const {
    return rest + fma((double)(65536ll * e16 + e), 0.69314718055994530942, log(prod));  // ln 2
  }
};

// increment of every active box (warp per box): M2L over V, P2L over X, and
// the parent's expansion at the box centre.  u^k and ((1+i)/2)^k come from the
// translation tables.
constexpr int kLevels = kMaxDepth + 2;
__global__ void k_pot_own(PotArgs A, FmmTables T, int64_t nact) {
  __shared__ double inv[kPotInv];
  // ln |(dx, dy)| by dx^2 + dy^2 (at most 18 in a V list), ln(2 r) by level
  __shared__ double lnd[19], lnr[kLevels];
  if (threadIdx.x >= 64 && threadIdx.x < 64 + 19) {
    const int q = threadIdx.x - 64;
    lnd[q] = q ? 0.5 * log((double)q) : 0.0;
  }
  if (threadIdx.x >= 96 && threadIdx.x < 96 + kLevels)
    lnr[threadIdx.x - 96] = log(2.0 * half_side(A, threadIdx.x - 96));
  fill_inv(inv, A.p + 2);
  const int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (a >= nact) return;
  const int B = A.active[a];
  const double r = half_side(A, A.level[B]);
  const double2 cB = centre(A, B, r);
  const int P1 = A.p + 1;
  double acc = 0.0;
  for (int64_t e = A.V_off[a] + lane; e < A.V_off[a + 1]; e += 32) {
    const int C = A.V_list[e];
    const int dx = A.ix[C] - A.ix[B], dy = A.iy[C] - A.iy[B];
    const double2* Ak = A.M + (int64_t)C * P1;
    const double2* u = T.upow + (int64_t)((dy + 3) * 7 + dx + 3) * (A.p + 2);
    // |t| = 2 r |(dx, dy)|
    acc = fma(Ak[0].x, lnr[A.level[B]] + lnd[dx * dx + dy * dy], acc);
    for (int k = 1; k <= A.p; ++k) acc -= inv[k] * (Ak[k].x * u[k].x - Ak[k].y * u[k].y);
  }
  for (int64_t e = A.X_off[a]; e < A.X_off[a + 1]; ++e) {
    const int C = A.X_list[e];
    for (int j = A.start[C] + lane; j < A.start[C] + A.count[C]; j += 32) {
      const double dx = cB.x - A.spos[j].x, dy = cB.y - A.spos[j].y;
      acc += A.smass[j] * 0.5 * log(dx * dx + dy * dy);
    }
  }
  const int Pb = A.parent[B];
  if (Pb >= 0 && A.aidx[Pb] >= 0) {
    // d^(l+1) = w^(l+1) i^(m (l+1)), w = (1+i)/2, m = 2, 3, 1, 0 for the quadrants;
    // w^(l+1) = w w^l
    const int q = B - A.child[Pb], m = q == 0 ? 2 : q == 1 ? 3 : q == 2 ? 1 : 0;
    const double2* Bl = A.L + (int64_t)Pb * P1;
    double s = 0.0;
    for (int l = lane; l <= A.p; l += 32) {
      const double2 w0 = T.wpow[l];
      const double2 w = make_double2(0.5 * (w0.x - w0.y), 0.5 * (w0.x + w0.y));
      const int ph = (m * (l + 1)) & 3;
      // Re(B_l w i^ph)
      const double2 b = Bl[l];
      const double re = b.x * w.x - b.y * w.y, im = b.x * w.y + b.y * w.x;
      s += inv[l + 1] * (ph == 0 ? re : ph == 1 ? -im : ph == 2 ? -re : im);
    }
    acc = fma(2.0 * r, s, acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) A.c0[a] = acc;
}

// Per active leaf: centre, half-side and its inverse, c_B (its increment and its
// active ancestors'), and the integrated expansion B_l / (l + 1); thread per
// (leaf, coefficient).
struct LeafPot {
  double cx, cy, r, ir, c;
  int a, pad;
};
__global__ void k_pot_leaf(PotArgs A, const int* __restrict__ leaves, int64_t nl,
                           LeafPot* __restrict__ lp, double2* __restrict__ Bi) {
  __shared__ double inv[kPotInv];
  fill_inv(inv, A.p + 2);
  const int P1 = A.p + 1;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t k = t / P1;
  if (k >= nl) return;
  const int l = (int)(t - k * P1), b = leaves[k];
  const double2 v = A.L[(int64_t)b * P1 + l];
  Bi[t] = make_double2(v.x * inv[l + 1], v.y * inv[l + 1]);
  if (l > 0) return;
  LeafPot q;
  q.r = half_side(A, A.level[b]);
  const double2 c = centre(A, b, q.r);
  q.cx = c.x; q.cy = c.y;
  q.ir = 1.0 / q.r;
  q.c = 0.0;
  q.a = A.aidx[b]; q.pad = 0;
  for (int x = b; x >= 0 && A.aidx[x] >= 0; x = A.parent[x]) q.c += A.c0[A.aidx[x]];
  lp[k] = q;
}

__device__ __forceinline__ double smooth_psi(const PotArgs& A, double x, double y) {
  return 0.5 * A.ks * (x * x + y * y) + 0.5 * A.g * (x * x - y * y);
}
// M2P of one W box: a_0 ln|t| - Re sum_{k>=1} (A_k / k) (r_C / t)^k, the
// coefficients Ak over k by Horner's rule (coef(k) = A_k / k)
template <typename F>
__device__ __forceinline__ double pot_m2p(double a0, int p, double2 t, double rC, F coef) {
  const double2 it = cinv(t);
  const double2 v = make_double2(rC * it.x, rC * it.y);
  double2 s = make_double2(0.0, 0.0);
  for (int k = p; k >= 1; --k) {
    s = s + coef(k);
    s = cmul(s, v);
  }
  return fma(a0, 0.5 * log(t.x * t.x + t.y * t.y), -s.x);
}

// Thread per ray, rays in leaf order (slot[r]: its leaf).
template <bool UM>
__global__ void __launch_bounds__(128)
k_pot_rays(PotArgs A, const double* __restrict__ rays, int64_t m, const int64_t* __restrict__ bad,
           const int* __restrict__ slot,
           const int* __restrict__ perm, const LeafPot* __restrict__ lp,
           const double2* __restrict__ Bi, int wmax, double* __restrict__ psi) {
  __shared__ double inv[kPotInv];
  fill_inv(inv, A.p + 2);
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= m || *bad) return;  // all rays lie in a leaf, or the call is refused
  const int64_t r = perm[t];
  const double x = rays[2 * r], y = rays[2 * r + 1];
  const int k0 = slot[r];
  const LeafPot q = lp[k0];
  const int a = q.a, P1 = A.p + 1;
  // L2P of the integrated local expansion
  const double2 w = make_double2((x - q.cx) * q.ir, (y - q.cy) * q.ir);
  const double2* Bl = Bi + (int64_t)k0 * P1;
  double2 acc = Bl[A.p];
  for (int l = A.p - 1; l >= 0; --l) acc = cfma(acc, w, Bl[l]);
  acc = cmul(acc, w);
  double phi = fma(q.r, acc.x, q.c);
  // P2P over U (a star exactly at the ray contributes nothing) and over W boxes
  // of at most wmax stars
  LogSum ls;
  const auto p2p = [&](int C) {
    for (int j = A.start[C]; j < A.start[C] + A.count[C]; ++j) {
      const double dx = x - A.spos[j].x, dy = y - A.spos[j].y;
      const double d2 = dx * dx + dy * dy;
      if (UM) ls.add(d2);
      else if (d2 > 0.0) phi += A.smass[j] * 0.5 * log(d2);
    }
  };
  for (int64_t e = A.U_off[a]; e < A.U_off[a + 1]; ++e) p2p(A.U_list[e]);
  for (int64_t e = A.W_off[a]; e < A.W_off[a + 1]; ++e) {
    const int C = A.W_list[e];
    if (A.count[C] <= wmax) { p2p(C); continue; }
    const double rC = half_side(A, A.level[C]);
    const double2 cC = centre(A, C, rC);
    const double2* Ak = A.M + (int64_t)C * P1;
    phi += pot_m2p(Ak[0].x, A.p, make_double2(x - cC.x, y - cC.y), rC, [&](int k) {
      return make_double2(Ak[k].x * inv[k], Ak[k].y * inv[k]);
    });
  }
  if (UM) phi += 0.5 * A.m0 * ls.value();
  psi[r] = phi + smooth_psi(A, x, y);
}

}  // namespace

void evaluate_potential(Plan& P, const double* rays, int64_t m, double* psi, cudaStream_t s) {
  if (m == 0) return;
  if (P.n_active == 0) fail(LENS_EDOMAIN, "plan has no active boxes");
  // the rays in leaf order
  const int64_t nl = P.n_active_leaves;
  RayBuckets RB;
  bucket_rays(P, rays, m, 1, RB, s);
  wait_expansions(P, s);
  Scratch c0(&P.da, sizeof(double) * (size_t)P.n_active);
  Scratch lp(&P.da, sizeof(LeafPot) * (size_t)nl);
  Scratch Bi(&P.da, sizeof(double2) * (size_t)nl * (P.p + 1));
  PotArgs A{};
  A.p = P.p;
  A.lo_x = P.root_lo[0]; A.lo_y = P.root_lo[1]; A.size = P.root_size;
  A.level = P.box_level; A.ix = P.box_ix; A.iy = P.box_iy; A.parent = P.box_parent;
  A.child = P.box_child; A.aidx = P.box_aidx; A.start = P.box_start;
  A.count = P.box_count; A.active = P.active; A.spos = P.spos; A.smass = P.smass;
  A.M = P.M; A.L = P.L;
  A.V_off = P.V_off; A.V_list = P.V_list; A.X_off = P.X_off; A.X_list = P.X_list;
  A.U_off = P.U_off; A.U_list = P.U_list; A.W_off = P.W_off; A.W_list = P.W_list;
  A.c0 = c0.as<double>();
  A.ks = P.kappa_s; A.g = P.gamma;
  A.m0 = P.mass0;
  k_pot_own<<<grid_for(P.n_active * 32, 256), 256, 0, s>>>(A, P.tab, P.n_active);
  LENS_LAUNCHED("k_pot_own");
  k_pot_leaf<<<grid_for(nl * (P.p + 1), 128), 128, 0, s>>>(A, P.active_leaves, nl, lp.as<LeafPot>(),
                                                            Bi.as<double2>());
  LENS_LAUNCHED("k_pot_leaf");
  // float64 operations of an M2P (~6 p + 45: the products with 1/k, Horner's rule, a
  // reciprocal, a logarithm) over those of a star summed directly: 5 with equal
  // masses, ~35 with a logarithm each
  const int wmax = (6 * P.p + 45) / (P.equal_mass ? 5 : 35);
  if (P.equal_mass)
    k_pot_rays<true><<<grid_for(m, 128), 128, 0, s>>>(A, rays, m, RB.bad, RB.slot.as<int>(),
                                                      RB.perm.as<int>(), lp.as<LeafPot>(),
                                                      Bi.as<double2>(), wmax, psi);
  else
    k_pot_rays<false><<<grid_for(m, 128), 128, 0, s>>>(A, rays, m, RB.bad, RB.slot.as<int>(),
                                                       RB.perm.as<int>(), lp.as<LeafPot>(),
                                                       Bi.as<double2>(), wmax, psi);
  LENS_LAUNCHED("k_pot_rays");
  check_rays(RB);
  LENS_CUDA(cudaStreamSynchronize(s));
}

}  // namespace lens
