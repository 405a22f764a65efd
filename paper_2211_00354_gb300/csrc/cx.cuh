// cx.cuh -- device helpers: complex arithmetic on double2/float2, compensated
// sums, Morton interleave, binomials.  Complex numbers z = x1 + i x2 are the
// image-plane positions (Appendix A: expansions in complex form).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lens {

template <typename R> struct cx_t;
template <> struct cx_t<double> { using type = double2; };
template <> struct cx_t<float> { using type = float2; };

template <typename R> __host__ __device__ __forceinline__ typename cx_t<R>::type mk(R a, R b) {
  typename cx_t<R>::type z; z.x = a; z.y = b; return z;
}
__host__ __device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
  C z; z.x = a.x * b.x - a.y * b.y; z.y = a.x * b.y + a.y * b.x; return z;
}
// a*b + c
template <typename C> __host__ __device__ __forceinline__ C cfma(C a, C b, C c) {
  C z;
  z.x = fma(a.x, b.x, fma(-a.y, b.y, c.x));
  z.y = fma(a.x, b.y, fma(a.y, b.x, c.y));
  return z;
}
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  float2 z;
  z.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x));
  z.y = fmaf(a.x, b.y, fmaf(a.y, b.x, c.y));
  return z;
}
template <typename C, typename R> __host__ __device__ __forceinline__ C cscale(C a, R s) {
  C z; z.x = a.x * s; z.y = a.y * s; return z;
}
// 1/x for x > 0: the hardware's coarse reciprocal (the PTX ISA has rcp.approx.ftz.f64 read
// and return the upper 20 mantissa bits: a relative error of about 2^-20) and one
// third-order Newton step, y (1 + e + e^2) with e = 1 - x y: the residual e^3 is about
// 2^-60 against the last rounding's 2^-53, so the result is within an ulp.
// Three float64 operations where the compiler's division takes about ten, on a
// pipe that gives a warp one instruction per ~77 cycles and sub-partition.  Outside
// the range where the seed is normal (and for 0, infinities, NaN) it divides.
__device__ __forceinline__ bool rcp_in_range(double x) {
  return (unsigned)__double2hiint(x) - 0x00100000u < 0x7fc00000u - 0x00100000u;
}
__device__ __forceinline__ double rcp_newton(double x) {  // rcp_in_range(x)
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rcp_pos(double x) { return rcp_in_range(x) ? rcp_newton(x) : 1.0 / x; }
// 1/x for x > 0, else 0 (a star exactly on a ray)
__device__ __forceinline__ double rcp_or_zero(double x) {
  return rcp_in_range(x) ? rcp_newton(x) : x > 0.0 ? 1.0 / x : 0.0;
}

// 1/z
__device__ __forceinline__ double2 cinv(double2 z) {
  const double d = rcp_pos(z.x * z.x + z.y * z.y);
  return make_double2(z.x * d, -z.y * d);
}
__device__ __forceinline__ float frcp_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 cinv(float2 z) {
  float d = frcp_fast(z.x * z.x + z.y * z.y);
  return make_float2(z.x * d, -z.y * d);
}

// Conversions on the integer pipe.  A float64 conversion holds the float64 pipe as
// long as a float64 product does (~77 cycles a warp and sub-partition); the words
// of a value in the normal range of both types are shifted and rounded in 2-8
// integer instructions instead, with the same bits (round to nearest even), and
// everything else (zero, subnormal, huge, infinite, NaN) takes the conversion.
// A warp is sent that way by one such value, so zero, the common one, is kept out.
__device__ __forceinline__ double f2d(float x) {
  const unsigned v = __float_as_uint(x), m = v & 0x7fffffffu;
  if (m == 0u) return __hiloint2double((int)v, 0);
  if (m - 0x00800000u >= 0x7f000000u) return (double)x;
  return __hiloint2double((int)((v & 0x80000000u) | ((m >> 3) + (896u << 20))), (int)(v << 29));
}
// exponents 2^-126 .. 2^126: the result is normal after rounding, too
__device__ __forceinline__ float d2f(double x) {
  const unsigned H = (unsigned)__double2hiint(x), L = (unsigned)__double2loint(x);
  if (((H >> 20) & 0x7ffu) - 897u >= 253u) return (float)x;
  const unsigned up = ((L & 0x1fffffffu) + 0x0fffffffu + ((L >> 29) & 1u)) >> 29;
  return __uint_as_float((__funnelshift_l(L, H, 3) + up - (896u << 23)) | (H & 0x80000000u));
}

// The double of an integer > 0, and x 2^k for a normal x and result (else by a
// product): the words again.
__device__ __forceinline__ double u2d(unsigned v) {
  const int lz = __clz((int)v);
  const unsigned m = v << lz;
  return __hiloint2double((int)(((1054u - lz) << 20) | ((m & 0x7fffffffu) >> 11)), (int)(m << 21));
}
__device__ __forceinline__ double mul_pow2(double x, int k) {
  const int H = __double2hiint(x), e = ((H >> 20) & 0x7ff) + k;
  if (e <= 0 || e >= 2047 || e - k == 0 || e - k == 2047) return ldexp(x, k);
  return __hiloint2double(H + k * 0x100000, __double2loint(x));
}

// Half side and centre of the box (level, ix, iy) of a root of side `size` at lo, and
// 1 / (half side) from 1 / size: divisions by powers of two, without the float64 pipe's.
__device__ __forceinline__ double box_half(double size, int level) { return mul_pow2(size, -(level + 1)); }
__device__ __forceinline__ double box_inv_half(double isize, int level) { return mul_pow2(isize, level + 1); }
__device__ __forceinline__ double box_centre(double lo, int i, double half) {
  return fma(u2d(2u * (unsigned)i + 1u), half, lo);
}

// Error-free sum of two floats (Knuth two-sum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// Compensated accumulator (hi, lo) += x
struct fcomp {
  float hi, lo;
  __device__ __forceinline__ void add(float x) {
    float s, e;
    two_sum(hi, x, s, e);
    hi = s;
    lo += e;
  }
  __device__ __forceinline__ double value() const { return f2d(hi) + f2d(lo); }
};

// Two compensated accumulators side by side (one per ray of a pair) on
// Blackwell's two-lane float32 instructions.  The error of hi + x comes from
// Dekker's fast two-sum with the operands ordered by magnitude (the ordering
// runs on the integer/compare pipe, the three paired operations on the FMA
// pipe, instead of six for Knuth's two-sum): the exact error of a rounded sum
// is unique, so the result equals fcomp::add's.  a - b is formed as
// fma(b, -1, a), exactly a - b (the product is exact, the sum rounds once).
struct fcomp2 {
  float2 hi, lo;
  __device__ __forceinline__ void add(float2 x) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const bool kx = fabsf(hi.x) >= fabsf(x.x), ky = fabsf(hi.y) >= fabsf(x.y);
    const float2 a = make_float2(kx ? hi.x : x.x, ky ? hi.y : x.y);
    const float2 b = make_float2(kx ? x.x : hi.x, ky ? x.y : hi.y);
    const float2 s = __fadd2_rn(a, b);
    const float2 e = __ffma2_rn(__ffma2_rn(a, m1, s), m1, b);  // b - (s - a)
    hi = s;
    lo = __fadd2_rn(lo, e);
  }
  // the same sum by Knuth's two-sum: six paired operations and no compares or
  // selects, for loops whose issue slots are scarcer than the FMA pipe's cycles
  __device__ __forceinline__ void add_knuth(float2 x) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 s = __fadd2_rn(hi, x);
    const float2 b = __ffma2_rn(hi, m1, s);                      // s - hi
    const float2 a = __ffma2_rn(b, m1, s);                       // s - b
    const float2 e = __fadd2_rn(__ffma2_rn(a, m1, hi), __ffma2_rn(b, m1, x));
    hi = s;
    lo = __fadd2_rn(lo, e);
  }
};

// The lanes of the warp whose digit (8 bits) is this lane's, among the `on` ones: a
// vote a bit.  A match instruction takes longer the more values there are (radix
// scatter, 1.5e6 keys 20 -> 14 us a pass, 1e7 keys 91 -> 82).
__device__ __forceinline__ unsigned same_digit(uint32_t d, bool on) {
  unsigned peers = __ballot_sync(0xffffffffu, on);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool bit = (d >> b) & 1u;
    const unsigned m = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? m : ~m;
  }
  return peers;
}

// Spread the low 32 bits of x to the even bit positions of a 64-bit word.
__host__ __device__ __forceinline__ uint64_t spread2(uint64_t x) {
  x &= 0xffffffffull;
  x = (x | (x << 16)) & 0x0000ffff0000ffffull;
  x = (x | (x << 8)) & 0x00ff00ff00ff00ffull;
  x = (x | (x << 4)) & 0x0f0f0f0f0f0f0f0full;
  x = (x | (x << 2)) & 0x3333333333333333ull;
  x = (x | (x << 1)) & 0x5555555555555555ull;
  return x;
}
__host__ __device__ __forceinline__ uint32_t compact2(uint64_t x) {
  x &= 0x5555555555555555ull;
  x = (x | (x >> 1)) & 0x3333333333333333ull;
  x = (x | (x >> 2)) & 0x0f0f0f0f0f0f0f0full;
  x = (x | (x >> 4)) & 0x00ff00ff00ff00ffull;
  x = (x | (x >> 8)) & 0x0000ffff0000ffffull;
  x = (x | (x >> 16)) & 0x00000000ffffffffull;
  return (uint32_t)x;
}
// Morton code: x bits at even, y bits at odd positions.
__host__ __device__ __forceinline__ uint64_t morton(uint32_t ix, uint32_t iy) {
  return spread2(ix) | (spread2(iy) << 1);
}

}  // namespace lens

namespace lens {
__host__ __device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }
__host__ __device__ __forceinline__ int64_t max64(int64_t a, int64_t b) { return a > b ? a : b; }
}  // namespace lens

namespace lens {
// ---- float-float ("double-single") arithmetic on the float32 pipe --------
// A value is hi + lo with |lo| <= ulp(hi)/2 (about 48 significant bits).  On
// GB300 the float64 pipe is ~60x slower than float32, so per-ray offsets and
// the lens-equation epilogue run in this form; float64 is used once per CTA.
struct ff {
  float hi, lo;
};
// hi = x rounded to float32, lo = the (exact) rest rounded: the 29 bits below hi,
// as a signed integer, times their weight.  Exponents from 2^-74, so that the
// rest is normal.
__host__ __device__ __forceinline__ ff ff_of(double x) {
  ff r;
#ifdef __CUDA_ARCH__
  const unsigned H = (unsigned)__double2hiint(x), L = (unsigned)__double2loint(x);
  const unsigned e = (H >> 20) & 0x7ffu;
  if (e - 949u < 201u) {
    const unsigned rem = L & 0x1fffffffu;
    const unsigned up = (rem + 0x0fffffffu + ((L >> 29) & 1u)) >> 29;
    r.hi = __uint_as_float((__funnelshift_l(L, H, 3) + up - (896u << 23)) | (H & 0x80000000u));
    const int d = (int)rem - (int)(up << 29);
    r.lo = (float)((int)H < 0 ? -d : d) * __uint_as_float((e - 948u) << 23);
    return r;
  }
#endif
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}
// floor(t) for 0 <= t < 2^32 from its words; false for anything else (negative,
// infinite, NaN).  As floor and a conversion, off the float64 pipe.
__device__ __forceinline__ bool floor_u32(double t, unsigned& q) {
  const unsigned H = (unsigned)__double2hiint(t), L = (unsigned)__double2loint(t);
  const unsigned e = H >> 20;  // a set sign makes it 2048 or more
  q = 0;
  if (e < 1023u) return true;
  if (e > 1054u) return H == 0x80000000u && L == 0u;  // -0
  q = (0x80000000u | (H << 11) | (L >> 21)) >> (1054u - e);
  return true;
}
__device__ __forceinline__ ff ff_norm(float s, float e) {  // |s| >= |e|
  ff r;
  r.hi = s + e;
  r.lo = e - (r.hi - s);
  return r;
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e += a.lo + b.lo;
  return ff_norm(s, e);
}
__device__ __forceinline__ ff ff_add(ff a, float b) {
  float s, e;
  two_sum(a.hi, b, s, e);
  e += a.lo;
  return ff_norm(s, e);
}
__device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.hi, -a.lo}; }
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return ff_norm(p, e);
}
__device__ __forceinline__ ff ff_mul(ff a, float b) {
  const float p = a.hi * b;
  const float e = fmaf(a.hi, b, -p) + a.lo * b;
  return ff_norm(p, e);
}
__device__ __forceinline__ double ff_to_double(ff a) { return f2d(a.hi) + f2d(a.lo); }

// The same float-float operations on two values side by side (one per ray of
// a pair), on the two-lane float32 instructions; a - b is fma(b, -1, a), and
// -round(x*y) is round(-x*y), so every lane computes exactly what the scalar
// form computes.
struct ff2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }
__device__ __forceinline__ ff2 ff2_norm(float2 s, float2 e) {  // |s| >= |e|
  ff2 r;
  r.hi = __fadd2_rn(s, e);
  r.lo = fsub2(e, fsub2(r.hi, s));
  return r;
}
// a + b (sign = +1) or a - b (sign = -1), two-sum of the high parts
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = __fadd2_rn(a, b);
  const float2 bb = fsub2(s, a);
  e = __fadd2_rn(fsub2(a, fsub2(s, bb)), fsub2(b, bb));
}
__device__ __forceinline__ void two_diff2(float2 a, float2 b, float2& s, float2& e) {
  s = fsub2(a, b);
  const float2 bb = fsub2(s, a);
  e = fsub2(fsub2(a, fsub2(s, bb)), __fadd2_rn(b, bb));
}
__device__ __forceinline__ ff2 ff2_add(ff2 a, ff2 b) {
  float2 s, e;
  two_sum2(a.hi, b.hi, s, e);
  e = __fadd2_rn(e, __fadd2_rn(a.lo, b.lo));
  return ff2_norm(s, e);
}
__device__ __forceinline__ ff2 ff2_add(ff a, ff2 b) {  // a the same in both lanes
  return ff2_add(ff2{f2(a.hi), f2(a.lo)}, b);
}
__device__ __forceinline__ ff2 ff2_sub(ff2 a, ff2 b) {
  float2 s, e;
  two_diff2(a.hi, b.hi, s, e);
  e = __fadd2_rn(e, fsub2(a.lo, b.lo));
  return ff2_norm(s, e);
}
__device__ __forceinline__ ff2 ff2_add(ff2 a, float2 b) {
  float2 s, e;
  two_sum2(a.hi, b, s, e);
  e = __fadd2_rn(e, a.lo);
  return ff2_norm(s, e);
}
__device__ __forceinline__ ff2 ff2_sub(ff2 a, float2 b) {
  float2 s, e;
  two_diff2(a.hi, b, s, e);
  e = __fadd2_rn(e, a.lo);
  return ff2_norm(s, e);
}
__device__ __forceinline__ ff2 ff2_mul(ff a, ff2 b) {  // a the same in both lanes
  const float2 ah = f2(a.hi);
  const float2 p = __fmul2_rn(ah, b.hi);
  float2 e = __ffma2_rn(ah, b.hi, __fmul2_rn(f2(-a.hi), b.hi));  // a.hi b.hi - p, exact
  e = __ffma2_rn(ah, b.lo, __ffma2_rn(f2(a.lo), b.hi, e));
  return ff2_norm(p, e);
}
}  // namespace lens
