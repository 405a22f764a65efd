// fmm.cu -- upward and downward passes of the FMM in complex form
// (Appendix A: multipole "S" and local "R" expansions, the S2S/M2M, S2R/M2L
// and R2R/L2L translation theorems; Greengard & Rokhlin 1987).
//
// The Cauchy sum f(z) = sum_j m_j / (z - z_j) gives the deflection of Eq. 1
// as alpha = conj(f).  For a box of centre c and half-side r:
//   multipole  f(z) = sum_k a_k / (z-c)^(k+1),  a_k = sum_j m_j (z_j - c)^k,
//              stored scaled: A_k = a_k / r^k;
//   local      f(z) = sum_l b_l (z-c)^l,        stored scaled: B_l = b_l r^l.
// Scaled, the child->parent M2M and parent->child L2L matrices do not depend
// on the level (child offset = (+-1 +-i) r_parent / 2), and the M2L matrix of
// two same-level boxes depends only on their integer offset:
//   M2M  A^P_l = sum_{k<=l} C(l,k) 2^-k d^(l-k) A^C_k,       d = (+-1 +-i)/2
//   L2L  B^C_j = sum_{l>=j} C(l,j) 2^-j d^(l-j) B^P_l
//   M2L  B_l  += (-1)^l u^(l+1) / r * sum_k C(k+l,k) u^k A_k,  u = r/(c_B - c_C)
// The M2L is split into a diagonal pre-scaling (u^k), one REAL binomial
// matrix applied to the complex vector, and a diagonal post-scaling, which
// halves the float64 multiply-adds of a dense complex matrix.
//   P2L  B_l  += -(m / (z-c)) (r / (z-c))^l        (X lists)
// Every step here is float64 (the precision split keeps translations in
// float64).  On GB300 the float64 pipe is ~60x slower than float32, so these
// kernels are written to issue as few DFMAs as the series allow.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "cx.cuh"
#include "lens_internal.h"

namespace lens {

namespace {

constexpr int kWarpsPerBlock = 4;

__device__ __forceinline__ double2 ld2(const double2* p) { return __ldg(p); }

// ---- P2M: one thread per leaf, accumulators in shared memory -----------------
// Leaves sorted by star count (counting sort, largest first), so that the
// lanes of a P2M warp run loops of equal length: with leaves of 1..leaf_size
// stars in tree order a warp would run its longest leaf's loop on all lanes.
// PASS 0 counts the non-empty leaves per star count and zeroes the expansions
// of empty leaves; PASS 1 places each leaf at offs[count] + rank.
template <int PASS>
__global__ void k_leaf_bins(const int* __restrict__ count, const int* __restrict__ child,
                            int64_t nb, int p, int leaf_size, int* __restrict__ bins,
                            int* __restrict__ offs, int* __restrict__ list,
                            double2* __restrict__ M) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int key = -1;
  if (b < nb && child[b] < 0) {
    const int nst = count[b];
    if (nst > 0) {
      key = min(nst, leaf_size);  // a leaf holds at most leaf_size stars
    } else if (PASS == 0) {
      double2* out = M + b * (int64_t)(p + 1);
      for (int k = 0; k <= p; ++k) out[k] = make_double2(0.0, 0.0);
    }
  }
  // one atomic per distinct count in the warp
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  const int leader = __ffs(peers) - 1;
  int base = 0;
  if (key > 0 && lane == leader) base = atomicAdd(&bins[key], __popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (PASS == 1 && key > 0) list[offs[key] + base + __popc(peers & ((1u << lane) - 1u))] = (int)b;
}

// All of it by one block, for a small tree: the two passes, the offsets and two
// memsets are five short operations (321 boxes: ~18 us with their gaps -> 3).
constexpr int kBinThreads = 1024, kBinSmallBoxes = 8192, kBinSmallLeaf = 64;

__global__ void __launch_bounds__(kBinThreads)
k_leaf_bins_small(const int* __restrict__ count, const int* __restrict__ child, int nb, int p,
                  int leaf_size, int* __restrict__ offs, int* __restrict__ list, double2* __restrict__ M) {
  __shared__ int bins[kBinSmallLeaf + 1];
  for (int k = threadIdx.x; k <= kBinSmallLeaf; k += kBinThreads) bins[k] = 0;
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += kBinThreads) {
    if (child[b] >= 0) continue;
    const int nst = count[b];
    if (nst > 0) {
      atomicAdd(&bins[min(nst, leaf_size)], 1);
    } else {
      double2* out = M + b * (int64_t)(p + 1);
      for (int k = 0; k <= p; ++k) out[k] = make_double2(0.0, 0.0);
    }
  }
  __syncthreads();
  // bins[k]: the first place of count k, largest counts first
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int k = leaf_size; k >= 1; --k) { const int c = bins[k]; bins[k] = acc; acc += c; }
    offs[0] = acc;  // leaves in the list
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += kBinThreads)
    if (child[b] < 0 && count[b] > 0) list[atomicAdd(&bins[min(count[b], leaf_size)], 1)] = b;
}

// offs[k] for counts k = leaf_size .. 1 (descending), offs[0] = total
__global__ void k_bin_offsets(const int* __restrict__ bins, int leaf_size, int* __restrict__ offs) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int acc = 0;
  for (int k = leaf_size; k >= 1; --k) { offs[k] = acc; acc += bins[k]; }
  offs[0] = acc;
}

// P2M: a_k = sum_j m_j w_j^k, w_j = (z_j - c)/r, into shared-memory
// accumulators [(p+1)][blockDim.x].  V = double2, or float2 for a float32-bulk
// plan: there the multipoles only feed far-field terms evaluated to float32
// accuracy, P2M is not one of the translations kept in float64, and the
// float64 pipe (~60x slower) would otherwise hold the upward pass on the
// build's critical path; w_j is formed in float64 and rounded once.
template <typename V>
__global__ void k_p2m(const double2* __restrict__ spos, const double* __restrict__ smass,
                      const int* __restrict__ start, const int* __restrict__ count,
                      const int* __restrict__ level, const int* __restrict__ ix,
                      const int* __restrict__ iy, const int* __restrict__ list,
                      const int* __restrict__ total, double lo_x, double lo_y, double root_size,
                      int p, double2* __restrict__ M) {
  extern __shared__ unsigned char acc_raw[];
  V* acc = reinterpret_cast<V*>(acc_raw);
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= *total) return;
  const int64_t b = list[i];
  const int nst = count[b];
  double2* out = M + b * (int64_t)(p + 1);
  const double r = root_size / (double)(2ull << level[b]);
  const double cx = lo_x + (2.0 * ix[b] + 1.0) * r, cy = lo_y + (2.0 * iy[b] + 1.0) * r;
  const double ir = 1.0 / r;
  V* a = acc + threadIdx.x;
  const int st = blockDim.x;
  V zero;
  zero.x = 0; zero.y = 0;
  for (int k = 0; k <= p; ++k) a[k * st] = zero;
  const int s0 = start[b];
  for (int j = 0; j < nst; ++j) {
    const double2 z = spos[s0 + j];
    const double m = smass[s0 + j];
    V w, pw;
    w.x = (z.x - cx) * ir; w.y = (z.y - cy) * ir;
    pw.x = m; pw.y = 0;
    for (int k = 0; k <= p; ++k) {
      a[k * st] = a[k * st] + pw;
      pw = cmul(pw, w);
    }
  }
  for (int k = 0; k <= p; ++k) out[k] = make_double2(a[k * st].x, a[k * st].y);
}

// ---- M2M: one thread per (internal box, coefficient) of a level -------------
// The four child offsets are d_q = w i^m_q with w = (1+i)/2 and m_q = 2, 3,
// 1, 0 for quadrants (-,-), (+,-), (-,+), (+,+).  Since d_q^(l-k) depends on
// q only through i^(m_q (l-k)), which repeats with period 4 in l-k,
//   A^P_l = w^l sum_{k<=l} C(l,k) conj(w)^k G_{(l-k) mod 4}[k],
//   G_r[k] = sum_m i^(m r) A^(child m)_k      (a 4-point DFT over quadrants:
//                                              additions only),
// one REAL binomial matrix on four complex vectors instead of four complex
// matrices: about a third of the float64 operations of the direct form.
// w^k and conj(w)^k are exact, so the rounding is that of the direct form: 2^-ceil(k/2)
// times one of the eight units 1, 1 +- i, ...  The powers of two go into the
// binomials (a product's rounding does not depend on them); a unit costs one addition
// a component for odd k and none for even k.  Thread (parent, k) forms the four
// H_r[k] = unit conj(w)^k G_r[k]; then the components of rows l and p - l, p + 2 terms
// together, are one thread's: lanes of a warp end at the same time, where a row a
// thread left half of the triangle idle.  An SM takes a warp's float64 instruction
// every 19 cycles, so their number is what it costs: 38 -> 24 a parent at p 16 (5.3e5
// boxes 431 -> 310 us).  A level's parents are walked through their children:
// the boxes of level l+1 are the groups of four children of the level-l splits, so
// group g (boxes c0+4g .. c0+4g+3) has one parent and no thread lands on a leaf.
constexpr int kM2MMaxThreads = 256;

__device__ __forceinline__ double flip(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}
// component c (0 real, 1 imaginary) of z times the unit of (1 + i)^k (k mod 8: 1, 1+i, i,
// -1+i, -1, -1-i, -i, 1-i), mine = z's component c, other = its other one
__device__ __forceinline__ double unit_component(int k, int c, double mine, double other) {
  // odd k: x - y and x + y up to signs; even k: x and y
  const int q = (k >> 1) & 3;  // quarter turns
  // i^q times v: component c is +-v of component c ^ (q & 1)
  double v0 = mine, v1 = other;  // components c and 1 - c of z (1 + i)^(k & 1)
  if (k & 1) {
    // (1+i)(x + iy) = (x - y) + i (x + y)
    const double sum = mine + other, dif = c ? other - mine : mine - other;  // x + y, x - y
    v0 = c ? sum : dif;
    v1 = c ? dif : sum;
  }
  // q = 1: (x, y) -> (-y, x); 2: (-x, -y); 3: (y, -x)
  const double r = (q & 1) ? v1 : v0;
  return flip(r, c ? q >= 2 : (q == 1 || q == 2));
}

// parents: per a block, their threads rounded up to whole warps
__global__ void __launch_bounds__(kM2MMaxThreads)
k_m2m(const int* __restrict__ parent, int64_t c0, int64_t ngroups, int p, int per,
      const double* __restrict__ binom, int ldb, double2* __restrict__ M) {
  extern __shared__ double2 H[];  // [parents per block][4][p+1], then the binomials
  const int P1 = p + 1, T = blockDim.x, t = threadIdx.x;
  // rows 0..p of the binomial table, triangular (row l from l (l+1) / 2), in
  // shared memory: the row sums below then wait on no global load (a small
  // level has too few blocks to keep the table in L1); times 2^-(ceil(l/2) + ceil(k/2))
  double* cb_tab = reinterpret_cast<double*>(H + (int64_t)per * 4 * P1);
  for (int i = t; i < P1 * (P1 + 1) / 2; i += T) {
    // i = l (l+1)/2 + kk, 0 <= kk <= l
    int l = (int)((sqrtf(8.f * (float)i + 1.f) - 1.f) * 0.5f);
    while (l * (l + 1) / 2 > i) --l;
    while ((l + 1) * (l + 2) / 2 <= i) ++l;
    const int kk = i - l * (l + 1) / 2;
    cb_tab[i] = mul_pow2(binom[(int64_t)l * ldb + kk], -((l + 1) / 2 + (kk + 1) / 2));
  }
  const int64_t g0 = (int64_t)blockIdx.x * per;
  const int ng = (int)min64(per, ngroups - g0);  // parents of this block
  for (int i = t; i < ng * P1; i += T) {
    const int pb = i / P1, k = i - pb * P1;
    const double2* A = M + (c0 + 4 * (g0 + pb)) * P1;  // four children, contiguous
    const double2 B0 = ld2(A + 3 * P1 + k), B1 = ld2(A + 2 * P1 + k);
    const double2 B2 = ld2(A + k), B3 = ld2(A + P1 + k);
    const double2 s02 = B0 + B2, d02 = B0 - B2, s13 = B1 + B3, d13 = B1 - B3;
    const double2 X[4] = {s02 + s13, make_double2(d02.x - d13.y, d02.y + d13.x), s02 - s13,
                          make_double2(d02.x + d13.y, d02.y - d13.x)};
    double2* h = H + (int64_t)pb * 4 * P1 + k;
    const int kc = (8 - (k & 7)) & 7;  // conj: the unit of (1 - i)^k is that of (1 + i)^(8 - k)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      // (1 - i)^k has the parity of k; one addition a component for odd k
      h[r * P1] = make_double2(unit_component(kc, 0, X[r].x, X[r].y), unit_component(kc, 1, X[r].y, X[r].x));
    }
  }
  __syncthreads();
  const int nt = 2 * ((P1 + 1) / 2);  // threads a parent: pairs of rows times two components
  for (int i0 = 0; i0 < per * nt; i0 += T) {
    const int i = i0 + t, pb = i / nt, j = i - pb * nt, c = j & 1;
    const bool on = pb < ng && i < per * nt;
    const int la = j >> 1, lb = p - la;  // la <= lb
    double va = 0.0, vb = 0.0;
    if (on) {
      const double* h = reinterpret_cast<const double*>(H + (int64_t)pb * 4 * P1) + c;
      // one loop over both rows, so that the lanes' loops are of one length
      const double* cr = cb_tab + la * (la + 1) / 2;
      const int steps = lb != la ? p + 2 : la + 1;
      int l = la, k = 0;
      double acc = 0.0;
      for (int q = 0; q < steps; ++q) {
        acc = fma(cr[k], h[2 * (((l - k) & 3) * P1 + k)], acc);
        ++k;
        if (q == la) {
          va = acc;
          acc = 0.0;
          l = lb;
          cr = cb_tab + lb * (lb + 1) / 2;
          k = 0;
        }
      }
      vb = acc;
    }
    // the other component is the neighbouring lane's (T and nt are even)
    const double oa = __shfl_xor_sync(0xffffffffu, va, 1), ob = __shfl_xor_sync(0xffffffffu, vb, 1);
    if (on) {
      const int64_t b = parent[c0 + 4 * (g0 + pb)];
      double* out = reinterpret_cast<double*>(M + b * P1) + c;
      out[2 * la] = unit_component(la, c, va, oa);
      if (lb != la) out[2 * lb] = unit_component(lb, c, vb, ob);
    }
  }
}

// ---- downward pass ---------------------------------------------------------
// The far-field part of each local expansion (M2L over the V list, P2L over
// the X list) reads only multipole expansions and stars, so one launch forms
// it for the active boxes of every level at once, one warp per box (kFarWarps warps
// for a small region): the float64 work of the coarse levels, a few boxes each,
// spreads over the whole GPU instead of a handful of SMs per level.  L2L, the
// only level-to-level dependence, then runs level by level from the top, one
// thread per component of a (box, coefficient).
//
// Bound by the float64 pipe: an SM takes a warp's float64 instruction every 19
// cycles, whatever lanes it has, and one warp issues them 64 cycles apart.  So real
// and imaginary parts sit in lanes of their own wherever a sum runs over fewer
// coefficients than lanes, and a region of few boxes gives each a whole block.
struct DownArgs {
  const int* active;
  int64_t a0, a1;
  const int* parent; const int* child; const int* level; const int* ix; const int* iy;
  const int* start; const int* count;
  const int64_t* V_off; const int* V_list;
  const int64_t* X_off; const int* X_list;
  const double2* spos; const double* smass;
  const double2* M;
  double2* L;
  FmmTables tab;
  double lo_x, lo_y, root_size, inv_size;
  int p;
  int group;         // V entries per M2L pass
  size_t smem_box;   // shared bytes per box (multiple of 16)
};

// V entries per M2L pass: 32, fewer for large p so that a warp's buffers
// (2 G (p+1) complex values) stay within 24 KB.
inline int downward_group(int p) { return std::max(1, std::min(32, 24576 / (32 * (p + 1)))); }
// Shared bytes per box: the larger of the P2L buffer ((p+1) x 33 complex +
// 64 ints; the odd row keeps the columns' sums off one bank) and the M2L buffers (2 G (p+1) complex + G ints).
constexpr int kP2lRow = 33;
inline size_t downward_smem_per_box(int p) {
  const size_t p2l = sizeof(double2) * (size_t)(p + 1) * kP2lRow + 64 * sizeof(int);
  const size_t g = (size_t)downward_group(p);
  const size_t m2l = sizeof(double2) * 2 * g * (size_t)(p + 1) + g * sizeof(int);
  return (std::max(p2l, m2l) + 15) / 16 * 16;
}

// NW warps a box: 1 (kWarpsPerBlock boxes a block) or kFarWarps (one box a block, for up
// to kFarFewBoxes active boxes, which as a warp each leave most of the pipes idle:
// 33 boxes of p 24 72 -> 17 us, 329 of p 16 42 -> 22; 4 * 152 is one warp a box on every
// sub-partition of the chip's SMs).  A box's sums are the same, term by term, for both.
constexpr int kFarWarps = 8;
constexpr int64_t kFarFewBoxes = 4 * 152;

template <int NW>
__global__ void __launch_bounds__(NW == 1 ? 32 * kWarpsPerBlock : 32 * NW) k_far_local(DownArgs A) {
  extern __shared__ double2 dsm[];
  constexpr int kT = 32 * NW;  // threads of a box
  const int t0 = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
  const int lane = threadIdx.x & 31, wib = NW == 1 ? threadIdx.x >> 5 : 0;
  const auto sync = [] { if (NW == 1) __syncwarp(); else __syncthreads(); };
  const int64_t a = A.a0 + (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kT;
  if (a >= A.a1) return;
  const int p = A.p, P1 = p + 1;
  const int B = A.active[a];
  const int lv = A.level[B];
  const double r = box_half(A.root_size, lv), ir = box_inv_half(A.inv_size, lv);
  // component c of coefficient l: item 2 l + c, thread t0 + kT s holds one
  constexpr int kItems = (2 * (kMaxOrder + 1) + kT - 1) / kT;
  double acc[kItems];
#pragma unroll
  for (int s = 0; s < kItems; ++s) acc[s] = 0.0;
  // M2L from V.  Up to G entries at a time, their (entry, coefficient) pairs
  // spread over the lanes (p + 1 = 17 coefficients would leave 15 of 32 lanes
  // idle with one entry per pass):
  //   H[e][k] = A_k u_e^k                       (pre-scale)
  //   T[e][l] = (-1)^l u_e^(l+1) / r * sum_k C(k+l, k) H[e][k]
  //   B_l    += sum_e T[e][l]
  double2* buf = dsm + (int64_t)wib * (A.smem_box / sizeof(double2));
  const int G = A.group;
  double2* H = buf;
  double2* T = buf + (int64_t)G * P1;
  int* uo = reinterpret_cast<int*>(T + (int64_t)G * P1);  // [G] offset-table rows
  const int bx = A.ix[B], by = A.iy[B];
  for (int64_t eb = A.V_off[a]; eb < A.V_off[a + 1]; eb += G) {
    const int ne = (int)min64(G, A.V_off[a + 1] - eb);
    for (int e = t0; e < ne; e += kT) {
      const int C = A.V_list[eb + e];
      uo[e] = ((A.iy[C] - by + 3) * 7 + (A.ix[C] - bx + 3)) * (p + 2);
    }
    sync();
    const int ntask = ne * P1;
    for (int t = t0; t < ntask; t += kT) {
      const int e = t / P1, k = t - e * P1;
      const int C = A.V_list[eb + e];
      H[t] = cmul(ld2(A.M + (int64_t)C * P1 + k), ld2(A.tab.upow + uo[e] + k));
    }
    sync();
    for (int t = t0; t < ntask; t += kT) {
      const int e = t / P1, l = t - e * P1;
      const double2* He = H + e * P1;
      double sx = He[0].x, sy = He[0].y;  // C(l, 0) = 1
      for (int k = 1; k <= p; ++k) {
        // C(k+l, k) = binom[(k+l)*ldb + k]
        const double c = __ldg(A.tab.binom + (int64_t)(k + l) * A.tab.ldb + k);
        const double2 v = He[k];
        sx = fma(c, v.x, sx);
        sy = fma(c, v.y, sy);
      }
      double2 post = ld2(A.tab.upow + uo[e] + l + 1);
      if (l & 1) post = make_double2(-post.x, -post.y);
      T[t] = cmul(post, make_double2(sx * ir, sy * ir));
    }
    sync();
    const double* Td = reinterpret_cast<const double*>(T);
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
      const int i = t0 + kT * s;
      if (i >= 2 * P1) break;
      double v = acc[s];
      for (int e = 0; e < ne; ++e) v = v + Td[2 * e * P1 + i];
      acc[s] = v;
    }
    sync();
  }
  // P2L from X.  The stars of the X boxes are taken 32 at a time across box
  // boundaries: lane j forms the series -m_j/(z_j-c) (r/(z_j-c))^l of its
  // star by recurrence into shared memory, then a lane sums a column's component.  (One
  // star at a time with per-lane powers would idle most of the warp when the
  // X boxes hold a few stars each.)
  const double cx = box_centre(A.lo_x, bx, r), cy = box_centre(A.lo_y, by, r);
  int* xs = reinterpret_cast<int*>(buf + (int64_t)P1 * kP2lRow);  // [32] inclusive counts, [32] starts
  for (int64_t eb = A.X_off[a]; eb < A.X_off[a + 1]; eb += 32) {
    const int ne = (int)min64(32, A.X_off[a + 1] - eb);
    int cnt = 0, st = 0;
    if (lane < ne) {
      const int C = A.X_list[eb + lane];
      cnt = A.count[C];
      st = A.start[C];
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    sync();
    if (t0 < 32) {
      xs[lane] = incl;
      xs[32 + lane] = st;
    }
    sync();
    for (int f0 = 0; f0 < total; f0 += 32) {
      const int f = f0 + lane;
      if (t0 < 32 && f < total) {
        int e = 0;
        while (xs[e] <= f) ++e;  // first box whose inclusive count exceeds f
        const int j = xs[32 + e] + f - (e ? xs[e - 1] : 0);
        const double2 z = A.spos[j];
        const double m = A.smass[j];
        const double2 inv = cinv(make_double2(z.x - cx, z.y - cy));  // 1/(z-c)
        const double2 q = make_double2(inv.x * r, inv.y * r);        // r/(z-c)
        double2 v = make_double2(-m * inv.x, -m * inv.y);            // -m/(z-c)
        for (int l = 0; l <= p; ++l) {
          buf[l * kP2lRow + lane] = v;
          v = cmul(v, q);
        }
      }
      sync();
      const int nv = min(32, total - f0);
      const double* bd = reinterpret_cast<const double*>(buf);
#pragma unroll
      for (int s = 0; s < kItems; ++s) {
        const int i = t0 + kT * s;
        if (i >= 2 * P1) break;
        const double* col = bd + 2 * (i >> 1) * kP2lRow + (i & 1);
        double v = acc[s];
        for (int jj = 0; jj < nv; ++jj) v = v + col[2 * jj];
        acc[s] = v;
      }
      sync();
    }
  }
  // by box, or by active index for the chain
  double* out = reinterpret_cast<double*>(A.L + (NW == 1 ? (int64_t)B : a) * P1);
#pragma unroll
  for (int s = 0; s < kItems; ++s) {
    const int i = t0 + kT * s;
    if (i < 2 * P1) out[i] = acc[s];
  }
}

// Component c of sum_{l >= j} S[j][l] z_l, row and z from l = j on, n terms, in order,
// each by cfma's products (-z.y or z.x with the imaginary part of S, then z.x or z.y with
// the real one).  S goes with the (l - j)-th power of (+-1 +- i) / 2: its imaginary part is
// 0 for l - j = 0 mod 4 and its real part for l - j = 2 mod 4, and a product with 0 is
// left out (1.1e5 boxes of p 12 303 -> 277 us).
__device__ __forceinline__ double l2l_component(const double2* __restrict__ S, const double2* z, int n, int c) {
  double v = 0.0;
  const auto re = [&](int t) { return c ? z[t].y : z[t].x; };
  const auto im = [&](int t) { return c ? z[t].x : flip(z[t].y, true); };
  for (int t = 0; t < n; t += 4) {
    v = fma(ld2(S + t).x, re(t), v);
    if (t + 1 < n) { const double2 s = ld2(S + t + 1); v = fma(s.x, re(t + 1), fma(s.y, im(t + 1), v)); }
    if (t + 2 < n) v = fma(ld2(S + t + 2).y, im(t + 2), v);
    if (t + 3 < n) { const double2 s = ld2(S + t + 3); v = fma(s.x, re(t + 3), fma(s.y, im(t + 3), v)); }
  }
  return v;
}

// L2L of the active boxes of one level (>= 2; above it the parent's local
// expansion is zero), one thread per component of a (box, coefficient j):
//   L_B[j] += sum_{l >= j} S_q[j][l] L_parent[l],  q = the box's quadrant.
// The parent of an active box is active and its expansion is final.  Few boxes: two
// products a term 64 cycles apart (a thread per complex coefficient, four):
// 8.5 -> 7 us a level.  Small blocks, so that the warps of a level spread over the SMs.
constexpr int kL2LThreads = 64;

__global__ void __launch_bounds__(kL2LThreads)
k_l2l(const int* __restrict__ active, int64_t a0, int64_t a1,
                      const int* __restrict__ parent, const int* __restrict__ child,
                      const double2* __restrict__ l2l, int p, double2* __restrict__ L) {
  const int P1 = p + 1;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = a0 + t / (2 * P1);
  if (a >= a1) return;
  const int i = (int)(t - (a - a0) * (2 * P1)), j = i >> 1, c = i & 1;
  const int B = active[a];
  const int par = parent[B];
  const int q = B - child[par];
  const double v = l2l_component(l2l + ((int64_t)q * P1 + j) * P1 + j, L + (int64_t)par * P1 + j, P1 - j, c);
  double* o = reinterpret_cast<double*>(L + (int64_t)B * P1 + j) + c;
  *o = *o + v;
}

// For a small region (kFarFewBoxes): a block per active box forms the local expansions of
// its ancestors from level 1 down and then its own, the same operations in the same order as
// level by level, from the far-field parts F (by active index) into L; one launch, each
// level's few boxes repeated by those below them, instead of one per level (33 boxes of p 24 on
// 4 levels 41 us with the launches' gaps -> 17, 324 boxes of p 16 on 14 levels 90 -> 35).
__global__ void k_l2l_chain(const int* __restrict__ active, const int* __restrict__ parent,
                            const int* __restrict__ aidx, const int* __restrict__ level,
                            const int* __restrict__ ix, const int* __restrict__ iy,
                            const double2* __restrict__ l2l, int p, const double2* __restrict__ F,
                            double2* __restrict__ L) {
  __shared__ int anc[kMaxDepth + 2];        // active index of the ancestor of each level
  __shared__ double2 cur[2][kMaxOrder + 1];
  const int P1 = p + 1, i = threadIdx.x, j = i >> 1, c = i & 1;
  const int B = active[blockIdx.x], lv = level[B], bx = ix[B], by = iy[B];
  if (i == 0) {
    int b = B;
    for (int l = lv; l >= 0; --l) { anc[l] = aidx[b]; if (l) b = parent[b]; }
  }
  __syncthreads();
  const bool on = i < 2 * P1;
  const auto far = [&](int l) {
    return on ? reinterpret_cast<const double*>(F + (int64_t)anc[l] * P1)[i] : 0.0;
  };
  int l = min(lv, 1);  // the expansions of levels 0 and 1 are their far parts
  double x = far(l);
  for (;;) {
    const double next = l < lv ? far(l + 1) : 0.0;
    double2* now = cur[l & 1];
    if (on) reinterpret_cast<double*>(now)[i] = x;
    if (l == lv) break;
    __syncthreads();
    ++l;
    if (on) {
      const int s = lv - l, q = ((bx >> s) & 1) | (((by >> s) & 1) << 1);
      x = next + l2l_component(l2l + ((int64_t)q * P1 + j) * P1 + j, now + j, P1 - j, c);
    }
  }
  if (on) reinterpret_cast<double*>(L + (int64_t)B * P1)[i] = x;
}

}  // namespace

// ---- host: tables ----------------------------------------------------------
void fmm_tables(Plan& P, cudaStream_t s) {
  const int p = P.p;
  const int P1 = p + 1;
  FmmTables& t = P.tab;
  t.p = p;
  t.ldb = p + 2;
  std::vector<double> t_bin((size_t)(2 * p + 2) * t.ldb, 0.0);
  const int nb = 2 * p + 2;
  const auto full = [&](int n, int k) -> double& { return t_bin[(size_t)n * t.ldb + k]; };
  std::vector<double>& bin = t_bin;
  // C(n, k), k < p + 2 (C(n, k) of row n needs only columns up to k of row n - 1)
  for (int n = 0; n < nb; ++n) {
    full(n, 0) = 1.0;
    for (int k = 1; k <= n && k < t.ldb; ++k) full(n, k) = full(n - 1, k - 1) + (k <= n - 1 ? full(n - 1, k) : 0.0);
  }
  // powers of the child offsets, by repeated products
  std::vector<std::pair<double, double>> dpow((size_t)4 * P1), wpw((size_t)P1);
  const auto powers = [&](double re, double im, std::pair<double, double>* out) {
    double pr = 1.0, pi = 0.0;
    for (int i = 0; i <= p; ++i) {
      out[i] = {pr, pi};
      const double nr = pr * re - pi * im, ni = pr * im + pi * re;
      pr = nr; pi = ni;
    }
  };
  powers(0.5, 0.5, wpw.data());
  std::vector<double2> l2l((size_t)4 * P1 * P1);
  for (int q = 0; q < 4; ++q) {
    const double dre = ((q & 1) ? 0.5 : -0.5), dim = ((q >> 1) ? 0.5 : -0.5);
    const std::pair<double, double>* dq = dpow.data() + (size_t)q * P1;
    powers(dre, dim, dpow.data() + (size_t)q * P1);
    for (int j = 0; j <= p; ++j)
      for (int l = 0; l <= p; ++l) {
        double2 v = make_double2(0.0, 0.0);
        if (l >= j) {
          const auto d = dq[l - j];
          const double c = full(l, j) * std::ldexp(1.0, -j);
          v = make_double2(c * d.first, c * d.second);
        }
        l2l[((size_t)q * P1 + j) * P1 + l] = v;
      }
  }
  std::vector<double2> up((size_t)49 * (p + 2));
  for (int dy = -3; dy <= 3; ++dy)
    for (int dx = -3; dx <= 3; ++dx) {
      const int o = (dy + 3) * 7 + (dx + 3);
      // u = r / (c_B - c_C) = -1 / (2 (dx + i dy))
      double ure = 0, uim = 0;
      if (dx != 0 || dy != 0) {
        const double den = 2.0 * (dx * (double)dx + dy * (double)dy);
        ure = -dx / den;
        uim = dy / den;
      }
      double pr = 1.0, pi = 0.0;
      for (int k = 0; k <= p + 1; ++k) {
        up[(size_t)o * (p + 2) + k] = make_double2(pr, pi);
        const double nr = pr * ure - pi * uim, ni = pr * uim + pi * ure;
        pr = nr; pi = ni;
      }
    }
  // ((1+i)/2)^k: Gaussian integers over powers of two, exact in float64
  std::vector<double2> wp((size_t)P1);
  for (int k = 0; k <= p; ++k) {
    wp[(size_t)k] = make_double2(wpw[(size_t)k].first, wpw[(size_t)k].second);
  }
  // one host block (kept in the plan until the copy has run: no wait here);
  // bin holds (2p+2)(p+2) doubles, an even count, so the complex tables
  // after it start on 16-byte boundaries
  const size_t nd = bin.size() + 2 * (l2l.size() + up.size() + wp.size());
  P.tab_host.assign(nd, 0.0);
  double* h = P.tab_host.data();
  std::memcpy(h, bin.data(), bin.size() * sizeof(double));
  size_t o = bin.size();
  for (const auto* v : {&l2l, &up, &wp}) {
    std::memcpy(h + o, v->data(), v->size() * sizeof(double2));
    o += 2 * v->size();
  }
  double* d = P.dalloc_n<double>(nd);
  LENS_CUDA(cudaMemcpyAsync(d, h, nd * sizeof(double), cudaMemcpyHostToDevice, s));
  o = bin.size();
  t.binom = d;
  t.l2l = reinterpret_cast<double2*>(d + o); o += 2 * l2l.size();
  t.upow = reinterpret_cast<double2*>(d + o); o += 2 * up.size();
  t.wpow = reinterpret_cast<double2*>(d + o);
}

void fmm_alloc(Plan& P) {
  const size_t P1 = (size_t)P.p + 1;
  if (!P.M) P.M = P.dalloc_n<double2>((size_t)P.nb * P1);
  if (!P.L) P.L = P.dalloc_n<double2>((size_t)P.nb * P1);
  if (!P.p2m_list) P.p2m_list = P.dalloc_n<int>((size_t)P.nb);
  if (!P.p2m_bins) P.p2m_bins = P.dalloc_n<int>(2 * ((size_t)P.leaf + 1));
}

void fmm_alloc_far(Plan& P) {
  if (P.n_active > 0 && P.n_active <= kFarFewBoxes)
    P.L_far = P.dalloc_n<double2>((size_t)P.n_active * (P.p + 1));
}

void fmm_p2m(Plan& P, cudaStream_t s) {
  const int p = P.p, P1 = p + 1;
  if (!P.M || !P.p2m_list || !P.p2m_bins) fail(LENS_ECUDA, "internal: expansion buffers not allocated");
  // P2M on every non-empty leaf (thread per leaf, leaves sorted by star
  // count), all levels at once
  const int L = P.leaf;
  int* cnt = P.p2m_bins;
  int* offs = cnt + (L + 1);
  int* list = P.p2m_list;
  if (P.nb <= kBinSmallBoxes && L <= kBinSmallLeaf) {
    k_leaf_bins_small<<<1, kBinThreads, 0, s>>>(P.box_count, P.box_child, (int)P.nb, p, L, offs, list, P.M);
    LENS_LAUNCHED("k_leaf_bins_small");
  } else {
    LENS_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)(L + 1), s));
    k_leaf_bins<0><<<grid_for(P.nb, 256), 256, 0, s>>>(P.box_count, P.box_child, P.nb, p, L, cnt, offs,
                                                        list, P.M);
    LENS_LAUNCHED("k_leaf_bins<count>");
    k_bin_offsets<<<1, 32, 0, s>>>(cnt, L, offs);
    LENS_LAUNCHED("k_bin_offsets");
    LENS_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)(L + 1), s));
    k_leaf_bins<1><<<grid_for(P.nb, 256), 256, 0, s>>>(P.box_count, P.box_child, P.nb, p, L, cnt, offs,
                                                        list, P.M);
    LENS_LAUNCHED("k_leaf_bins<place>");
  }
  const int tpb = 32;
  if (P.prec == LENS_FP32_BULK) {
    const size_t smem = sizeof(float2) * (size_t)P1 * tpb;
    if (smem > 48 * 1024)
      LENS_CUDA(cudaFuncSetAttribute(k_p2m<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    k_p2m<float2><<<grid_for(P.nb, tpb), tpb, smem, s>>>(
        P.spos, P.smass, P.box_start, P.box_count, P.box_level, P.box_ix, P.box_iy, list, offs,
        P.root_lo[0], P.root_lo[1], P.root_size, p, P.M);
  } else {
    const size_t smem = sizeof(double2) * (size_t)P1 * tpb;
    if (smem > 48 * 1024)
      LENS_CUDA(cudaFuncSetAttribute(k_p2m<double2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    k_p2m<double2><<<grid_for(P.nb, tpb), tpb, smem, s>>>(
        P.spos, P.smass, P.box_start, P.box_count, P.box_level, P.box_ix, P.box_iy, list, offs,
        P.root_lo[0], P.root_lo[1], P.root_size, p, P.M);
  }
  LENS_LAUNCHED("k_p2m");
}

void fmm_m2m(Plan& P, cudaStream_t s) {
  const FmmTables& t = P.tab;
  const int P1 = P.p + 1;
  // parents a block: the fewest that fill whole warps best
  const int nt = 2 * ((P1 + 1) / 2);
  int per = 1, threads = (nt + 31) / 32 * 32;
  for (int q = 2; q * nt <= kM2MMaxThreads; ++q) {
    const int th = (q * nt + 31) / 32 * 32;
    if (th <= kM2MMaxThreads && (int64_t)q * threads > (int64_t)per * th) { per = q; threads = th; }
  }
  const size_t smem = sizeof(double2) * 4 * (size_t)P1 * per + sizeof(double) * P1 * (P1 + 1) / 2;
  if (smem > 48 * 1024)
    LENS_CUDA(cudaFuncSetAttribute(k_m2m, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  for (int l = P.nlevels - 2; l >= 0; --l) {
    // level l+1 holds the children of the level-l splits, four per split
    const int64_t c0 = P.level_off[l + 1], ng = (P.level_off[l + 2] - c0) / 4;
    if (ng <= 0) continue;
    k_m2m<<<grid_for(ng, per), threads, smem, s>>>(P.box_parent, c0, ng, P.p, per, t.binom, t.ldb, P.M);
    LENS_LAUNCHED("k_m2m");
  }
}

void fmm_downward(Plan& P, cudaStream_t s) {
  const FmmTables& t = P.tab;
  if (!P.L) P.L = P.dalloc_n<double2>((size_t)P.nb * (P.p + 1));
  DownArgs A{};
  A.active = P.active;
  A.parent = P.box_parent; A.child = P.box_child; A.level = P.box_level;
  A.ix = P.box_ix; A.iy = P.box_iy; A.start = P.box_start; A.count = P.box_count;
  A.V_off = P.V_off; A.V_list = P.V_list; A.X_off = P.X_off; A.X_list = P.X_list;
  A.spos = P.spos; A.smass = P.smass; A.M = P.M; A.L = P.L; A.tab = t;
  A.lo_x = P.root_lo[0]; A.lo_y = P.root_lo[1]; A.root_size = P.root_size;
  A.inv_size = 1.0 / P.root_size; A.p = P.p;
  A.group = downward_group(P.p);
  A.smem_box = downward_smem_per_box(P.p);
  const bool few = P.L_far != nullptr;
  if (few) A.L = P.L_far;
  const size_t smem = A.smem_box * (few ? 1 : kWarpsPerBlock);
  if (smem > 48 * 1024)
    LENS_CUDA(cudaFuncSetAttribute(few ? k_far_local<kFarWarps> : k_far_local<1>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  A.a0 = 0;
  A.a1 = P.n_active;
  if (A.a1 > 0) {
    if (P.ev_far0) LENS_CUDA(cudaEventRecord(P.ev_far0, s));
    if (few) k_far_local<kFarWarps><<<(unsigned)A.a1, 32 * kFarWarps, smem, s>>>(A);
    else k_far_local<1><<<grid_for(A.a1 * 32, 32 * kWarpsPerBlock), 32 * kWarpsPerBlock, smem, s>>>(A);
    LENS_LAUNCHED("k_far_local");
    if (P.ev_far1) LENS_CUDA(cudaEventRecord(P.ev_far1, s));
  }
  const int P1 = P.p + 1;
  if (few) {
    k_l2l_chain<<<(unsigned)P.n_active, (2 * P1 + 31) / 32 * 32, 0, s>>>(
        P.active, P.box_parent, P.box_aidx, P.box_level, P.box_ix, P.box_iy, t.l2l, P.p, P.L_far, P.L);
    LENS_LAUNCHED("k_l2l_chain");
    return;
  }
  for (int l = 2; l < P.nlevels; ++l) {
    const int64_t a0 = P.active_level_off[l], a1 = P.active_level_off[l + 1];
    if (a1 <= a0) continue;
    k_l2l<<<grid_for((a1 - a0) * 2 * P1, kL2LThreads), kL2LThreads, 0, s>>>(
        P.active, a0, a1, P.box_parent, P.box_child, t.l2l, P.p, P.L);
    LENS_LAUNCHED("k_l2l");
  }
}

}  // namespace lens
