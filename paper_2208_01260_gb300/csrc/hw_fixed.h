// Block fixed-point arithmetic of the nonlinear reconstructions (Sec. 2.1 Step 1, Sec. 2.2) on the integer
// pipes.
//
// GB300's FP64 pipe takes 1.87 lane-operations per SM and cycle (measured), its integer pipes 38 64-bit
// additions, 25 64-bit shifts and 20 32x32->64-bit multiply-adds. A reconstruction is short chains of sums
// and products of data of one scale, so it needs no floating point between its ends: the data of a stencil
// is brought to one exponent (64-bit two's complement, 56 to 60 significant bits of the largest entry), sums
// are then exact, products keep their upper 64 bits, and only where squares are compared across scales (the
// smoothness indicators, whose small ones carry the weights) is a value normalised on its own. Every rounding
// is at most 2^-55 of the largest entry of its stencil and component, where the FP64 form rounds sums of that size
// at 2^-53, so reconstructed and limited values are nearer to the exact ones than the FP64 form's. An entry far below
// the largest (a small derivative beside its value) keeps fewer bits of its own than a double; what it loses is below
// the rounding of the sums it enters. Over whole runs the errors are level with the FP64 form's: the assembly and the
// combination of stages, which round as before, outweigh the reconstruction.
//
// Conventions: a value is x 2^u with x a 64-bit integer and u an int held beside it (per stencil, not per
// value). Operands that do not fit (subnormal, infinite or NaN data, or an exponent near the ends of the
// range) are reported by the conversions; the caller then computes on the FP64 pipe. The header compiles as
// CUDA and as plain C++ (host-side checks).
#pragma once
#include <stdint.h>

#include "hw_fp64_int.h"

namespace hw {

#define HW_FX HW_FP64_INT_FN

HW_FX int fx_max(int a, int b) { return a > b ? a : b; }
HW_FX int fx_min(int a, int b) { return a < b ? a : b; }
HW_FX int fx_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
HW_FX uint32_t fx_hi(uint64_t x) { return (uint32_t)(x >> 32); }
HW_FX uint32_t fx_lo(uint64_t x) { return (uint32_t)x; }

// ---- products -------------------------------------------------------------------------------
// a b and a b + c of 32-bit factors. Written as PTX: from C the compiler keeps product and sum apart (a signed
// 64 x 64 upper product 14 instructions instead of 5, a two-term dot product 30 instead of 12).
HW_FX uint64_t fx_mulw(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (uint64_t)a * b;
#endif
}
HW_FX uint64_t fx_madw(uint32_t a, uint32_t b, uint64_t c) {
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (uint64_t)a * b + c;
#endif
}
HW_FX int64_t fx_mulws(int32_t a, int32_t b) {
#if defined(__CUDA_ARCH__)
  int64_t r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (int64_t)a * b;
#endif
}
HW_FX int64_t fx_madws(int32_t a, int32_t b, int64_t c) {
#if defined(__CUDA_ARCH__)
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (int64_t)a * b + c;
#endif
}
HW_FX uint32_t fx_mulhi32(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// Signed limbs x = h 2^32 + l with l in [-2^31, 2^31), so that all four partial products are signed.
struct FxS {
  int32_t h, l;
};
HW_FX FxS fx_split(int64_t x) {
  FxS s;
  s.l = (int32_t)fx_lo((uint64_t)x);
  s.h = (int32_t)(fx_hi((uint64_t)x) + (fx_lo((uint64_t)x) >> 31));
  return s;
}
// a b / 2^64 + add within 2 units, for |a| < 2^61, |b| < 2^63 (the low limbs' product is left out).
HW_FX int64_t fx_mulhi(FxS a, FxS b, int64_t add) {
  const int64_t c = fx_madws(a.l, b.h, fx_mulws(a.h, b.l));
  return fx_madws(a.h, b.h, add) + (c >> 32);
}
// (a1 w1 + a2 w2) / 2^(64 - SH) within 2^SH units, for |a| <= 2^61 and |w| <= 2^62.
template <int SH>
HW_FX int64_t fx_dot2(FxS a1, FxS w1, FxS a2, FxS w2) {
  const int64_t c = fx_madws(a2.l, w2.h, fx_madws(a2.h, w2.l, fx_madws(a1.l, w1.h, fx_mulws(a1.h, w1.l))));
  const int64_t h = fx_madws(a2.h, w2.h, fx_mulws(a1.h, w1.h));
  return (int64_t)((uint64_t)h << SH) + (c >> (32 - SH));
}
// a b / 2^64 within 2 units below, for a b_hi + a_hi b < 2^64 (both below 2^63).
HW_FX uint64_t fx_mulhi_u(uint64_t a, uint64_t b) {
  const uint64_t c = fx_madw(fx_hi(a), fx_lo(b), fx_mulw(fx_lo(a), fx_hi(b)));
  return fx_madw(fx_hi(a), fx_hi(b), fx_hi(c));
}
// a^2 / 2^64 within 3 units below.
HW_FX uint64_t fx_sqhi(uint64_t a) {
  return fx_madw(fx_hi(a), fx_hi(a), (uint64_t)fx_mulhi32(fx_hi(a), fx_lo(a)) << 1);
}

// ---- conversions ----------------------------------------------------------------------------
// Biased exponent fields are kept in place (bits 20..30 of the upper word) while maxima are taken.
HW_FX uint32_t fx_absw(double x) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  return hi & 0x7fffffffu;
}
// Nonzero unless x is zero.
HW_FX uint32_t fx_any(double x) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  return lo | (hi << 1);
}
// x as a multiple of 2^(em - 1082), |result| < 2^60, for a group whose largest biased exponent is em (at
// least 64): exact down to that unit, towards zero below it; zero and subnormal x give 0.
HW_FX int64_t fx_from_double(double x, int em) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const uint64_t m = (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 39) | ((uint64_t)lo << 7)) >> fx_min(em - e, 63);
  const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);
  return (int64_t)((m ^ s) - s);
}
// A double as x 2^u with |x| in [2^61, 2^62) (0 for zero and subnormal arguments).
HW_FX int64_t fx_mantissa(double x, int& u) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  const int e = (int)((hi >> 20) & 0x7ffu);
  u = e - 1084;
  const uint64_t m = e == 0 ? 0 : ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 41) | ((uint64_t)lo << 9);
  const uint64_t s = (uint64_t)(int64_t)((int32_t)hi >> 31);
  return (int64_t)((m ^ s) - s);
}
// x 2^u rounded to nearest, for |x| < 2^63 and results in the normal range (the callers bound u).
HW_FX double fx_to_double(int64_t x, int u) {
  const uint32_t s = (uint32_t)((uint64_t)x >> 63);
  uint64_t a = ((uint64_t)x ^ (0ull - s)) + s;
  const bool small = fx_hi(a) == 0;
  const int n = fx_clz(small ? fx_lo(a) : fx_hi(a)) + (small ? 31 : -1);  // leading bit to 62
  a = (a << n) + 0x200u;
  // the leading bit adds one to the exponent field, a carry of the rounding another
  const uint64_t r = a >> 10;
  const uint32_t h = fx_hi(r) + ((uint32_t)(u + 1084 - n) << 20) + (s << 31);
  return x == 0 ? 0.0 : f64_from_words(fx_lo(r), h);
}

// A positive constant as m 2^u with m in [2^62, 2^63), for fx_to_double_scaled. bad: results could leave the normal range.
// Those are below 2^963 times the constant (units up to 2^900, integers below 2^63) and at least 2^-900 times it, so 2^-96
// to 2^60 is safe: as a grid's factors g/(2dx) and 1/(24dx), with g = 9.8, spacings from 1e-17 to 1e27. Beyond, every
// interface of the grid is formed from its nodes again (four steps of 1024 x 1024 34.2 ms against 8.1).
struct FxScale {
  uint64_t m;
  int u;
};
HW_FX FxScale fx_scale(double c, bool& bad) {
  uint32_t lo, hi;
  f64_words(c, lo, hi);
  const int e = (int)(hi >> 20);  // negative, infinite and NaN: above the range
  bad |= (unsigned)(e - 1023 + 96) > 155u;
  FxScale s;
  s.m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 42) | ((uint64_t)lo << 10);
  s.u = e - 1085;
  return s;
}
// x 2^u times the constant, rounded to nearest (the product keeps 60 bits, so within 0.52 units in the last place), for
// |x| < 2^63. The product costs 9 integer instructions where a multiplication after the conversion costs the FP64 pipe
// 17 cycles a warp, the time of 40 of them.
HW_FX double fx_to_double_scaled(int64_t x, int u, FxScale c) {
  const uint32_t s = (uint32_t)((uint64_t)x >> 63);
  uint64_t a = ((uint64_t)x ^ (0ull - s)) + s;
  const bool small = fx_hi(a) == 0;
  const int n = fx_clz(small ? fx_lo(a) : fx_hi(a)) + (small ? 31 : -1);  // leading bit to 62
  a = fx_mulhi_u(a << n, c.m);                                            // [2^60, 2^62)
  const int k = (int)((fx_hi(a) >> 29) ^ 1u);
  const uint64_t r = ((a << k) + 0x100u) >> 9;
  const uint32_t h = fx_hi(r) + ((uint32_t)(u + c.u + 1147 - n - k) << 20) + (s << 31);
  return x == 0 ? 0.0 : f64_from_words(fx_lo(r), h);
}
// x / 4, rounded to nearest even where it is subnormal: the exponent field, without the FP64 pipe.
HW_FX double fx_quarter(double x) {
  uint32_t lo, hi;
  f64_words(x, lo, hi);
  const int e = (int)((hi >> 20) & 0x7ffu);
  if (e <= 2 && (lo | (hi << 1)) != 0u) {
    const int n = 3 - fx_max(e, 1);
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
    const uint64_t r = (m + ((1ull << (n - 1)) - 1) + ((m >> n) & 1)) >> n;
    return f64_from_words(fx_lo(r), fx_hi(r) | (hi & 0x80000000u));
  }
  return e == 0 || e == 0x7ff ? x : f64_from_words(lo, hi - 0x200000u);
}

// ---- nonlinear weights ----------------------------------------------------------------------
// Positive quantities of their own scale: q 2^x (x relative to a scale common to the three).
HW_FX uint64_t fx_shr(uint64_t a, int n) { return a >> fx_min(n, 63); }

// b^2 + c a^2 for |a|, |b| < 2^62 and c (given as c 2^64) at most 1/4, both brought up by the same shift (at most
// cap), so that the larger keeps 61 bits. Returns q < 2^62 (1 + c) for q 2^x.
HW_FX uint64_t fx_group(int64_t b, int64_t a, uint64_t c, int cap, int& x) {
  const uint64_t sb = (uint64_t)(b >> 63), sa = (uint64_t)(a >> 63);
  const uint64_t ub = (uint64_t)b ^ sb, ua = (uint64_t)a ^ sa;  // |.| within one unit
  const int n = fx_max(fx_min(fx_clz(fx_hi(ub) | fx_hi(ua)) - 1, cap), 0);
  x = -2 * n;
  return fx_sqhi(ub << n) + fx_mulhi_u(fx_sqhi(ua << n), c);
}

// a 2^xa + b 2^xb at the larger exponent.
HW_FX uint64_t fx_add(uint64_t a, int xa, uint64_t b, int xb, int& x) {
  const int d = xa - xb;
  x = fx_max(xa, xb);
  return fx_shr(a, fx_max(-d, 0)) + fx_shr(b, fx_max(d, 0));
}

// About 2^125 / d for d in [2^62, 2^63), relative error below 2^-58: seed from the single-precision
// reciprocal, one third-order Newton-Raphson step on the residual e = 1 - d y (r = y (1 + e + e^2)).
HW_FX uint64_t fx_rcp(uint64_t d) {
  const float mf = f32_from_bits((fx_hi(d) >> 7) + 0x3f000000u);  // [1, 2): the leading 24 bits
  const uint32_t yb = f32_bits(f32_rcp_seed(mf));
  const uint32_t m = ((yb < 0x3f7fffffu ? yb : 0x3f7fffffu) & 0x7fffffu) | 0x800000u;  // y 2^24, y in [1/2, 1)
  const uint32_t y = m << 8;
  const uint64_t p = fx_madw(fx_hi(d), y, fx_mulhi32(fx_lo(d), y));  // d y at scale 2^62
  const int64_t e = (int64_t)((1ull << 62) - p);
  const int32_t es = (int32_t)(e >> 16);
  const int64_t t = e + (fx_mulws(es, es) >> 30);
  const int64_t t2 = t >> 2;
  const int64_t corr = (int64_t)(fx_mulw(m, fx_lo((uint64_t)t2)) + ((uint64_t)(m * fx_hi((uint64_t)t2)) << 32));
  return ((uint64_t)m << 39) + (uint64_t)(corr >> 21);
}

// The weights omega_1, omega_2 (at scale 2^61) proportional to G1 / t_1^2, G1 / t_2^2, G3 / t_3^2 with
// t_l = b_l^2 + k a_l^2 + c 2^xc, l = 3 with halves of b_3 and a_3 (xc even; squares at scale 2^-64): each t_l is
// normalised, the products of the other two squares taken (one reciprocal), brought to one exponent and
// divided by their sum.
template <int G1, int G3>
HW_FX void fx_weights(int64_t b1, int64_t a1, int64_t b2, int64_t a2, int64_t b3, int64_t a3, uint64_t k, uint64_t c,
                      int xc, int64_t& w1, int64_t& w2) {
  // squares whose unit would fall below c's stop there
  const int cap = -xc >> 1;
  int x1, x2, x3;
  uint64_t t1 = fx_group(b1, a1, k, cap, x1), t2 = fx_group(b2, a2, k, cap, x2), t3 = fx_group(b3, a3, k, cap - 1, x3);
  x3 -= 2;
  if (xc >= 0) {  // c above the squares' unit
    t1 = fx_shr(t1, xc);
    t2 = fx_shr(t2, xc);
    t3 = fx_shr(t3, xc + 2);
    x1 = x2 = x3 = xc;
  }
  t1 += fx_shr(c, x1 - xc);
  t2 += fx_shr(c, x2 - xc);
  t3 += fx_shr(c, x3 - xc);
  const int n1 = fx_clz(fx_hi(t1)) - 1, n2 = fx_clz(fx_hi(t2)) - 1, n3 = fx_clz(fx_hi(t3)) - 1;
  t1 = fx_sqhi(t1 << n1);
  t2 = fx_sqhi(t2 << n2);
  t3 = fx_sqhi(t3 << n3);
  x1 -= n1;
  x2 -= n2;
  x3 -= n3;
  // 1 / t_l^2 ~ (product of the other squares) 2^(-2 x_l), the largest at shift 1
  const int xm = fx_min(fx_min(x1, x2), x3);
  uint64_t p1 = fx_shr(fx_mulhi_u(t2, t3), 2 * (x1 - xm) + 1);
  uint64_t p2 = fx_shr(fx_mulhi_u(t1, t3), 2 * (x2 - xm) + 1);
  const uint64_t p3 = fx_shr(fx_mulhi_u(t1, t2), 2 * (x3 - xm) + 1);
  if (G1 == 3) {
    p1 = p1 + p1 + p1;
    p2 = p2 + p2 + p2;
  }
  const uint64_t den = p1 + p2 + p3 * G3;
  const int n = fx_clz(fx_hi(den)) - 1;
  const uint64_t r = fx_rcp(den << n);
  w1 = (int64_t)fx_mulhi_u(p1 << n, r);
  w2 = (int64_t)fx_mulhi_u(p2 << n, r);
}

// Weights' epsilon: (constant times) eps as m 2^u with u even and m in [2^58, 2^60).
struct FxEps {
  uint64_t m;
  int u;
};
HW_FX FxEps fx_eps(double e, bool& bad) {
  uint32_t lo, hi;
  f64_words(e, lo, hi);
  const int ex = (int)(hi >> 20);  // negative, infinite and NaN: above the range
  bad |= (unsigned)(ex - 1) >= 0x7feu;
  FxEps r;
  r.m = (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 39) | ((uint64_t)lo << 7)) >> (ex & 1);
  r.u = ex - 1082 + (ex & 1);
  return r;
}

// One characteristic field, one upwind side (the algebra of hweno_side, hw_device.cuh): f0..f2 and p0..p2 as
// multiples of 2^u, each below 2^57; eps carries 20/781. Returns 6 times the weighted value (below 2^61), and
// omega_1, omega_2 at scale 2^61 for the source.
//   t_l (20/781) = B_l^2 + (260/2343) A_l^2 + (20/781)(p1^2 + eps), l = 3 with e/2 for A, g3/2 for B;
//   sum(omega_l q_l) = q_3 + omega_1 (q_1 - q_3) + omega_2 (q_2 - q_3) with 12 (q_1 - q_3) = 2 A_1 - e,
//   12 (q_2 - q_3) = -2 A_2 - e, 12 q_3 = 12 f_1 + 6 p_1 + e.
constexpr uint64_t FX_C_A = 0x1c6874411eb3d83aull;  // 260/2343 2^64
constexpr uint64_t FX_C_P = 0x68e4236698bf6d27ull;  // 640/781 2^63
constexpr uint64_t FX_C_L = 0x3b13b13b13b13b13ull;  // 3/13 2^64
HW_FX int64_t fx_hweno_side(int64_t f0, int64_t f1, int64_t f2, int64_t p0, int64_t p1, int64_t p2, FxEps eps, int u,
                            int64_t& w1, int64_t& w2) {
  const int64_t d1 = f0 - f1, d2 = f1 - f2;
  const int64_t B1 = d1 + d1 + (p0 + p1), B2 = d2 + d2 + (p1 + p2);
  const int64_t A1 = B1 + d1 + p1, A2 = B2 + d2 + p1;
  const int64_t e = d1 - d2, g = d1 + d2 + (p1 + p1);
  // (20/781)(p1^2 + eps): exponents relative to 2 u + 64
  uint64_t c = (uint64_t)p1 ^ (uint64_t)(p1 >> 63);
  const int np = fx_clz(fx_hi(c)) - 1;
  c = fx_mulhi_u(fx_sqhi(c << np), FX_C_P);
  int xc;
  c = fx_add(c, -4 - 2 * np, eps.m, eps.u - 2 * u - 64, xc);
  fx_weights<3, 4>(B1, A1, B2, A2, g, e, FX_C_A, c, xc, w1, w2);
  const int64_t b = f1 + f1 + p1;
  return b + b + b + (e >> 1) + fx_dot2<2>(fx_split(A1 + A1 - e), fx_split(w1), fx_split(-(A2 + A2) - e), fx_split(w2));
}

// Limiter of one characteristic field (limiter_field, hw_device.cuh): dl = m1 - m0, dr = m2 - m1, nl, nr below
// 2^58 as multiples of 2^u, eps carrying 3/13. Returns twice the limited value (below 2^61).
//   t_l (3/13) = a_l^2 + (3/13) p_l^2 + (3/13) eps, l = 3 with halves of m2 - m0 and of the second difference.
HW_FX int64_t fx_limiter_field(int64_t dl, int64_t dr, int64_t nl, int64_t nr, FxEps eps, int u) {
  const int64_t pl = dl + dl - nl, pr = dr + dr - nr, pc = dl + dr;
  int64_t w1, w2;
  fx_weights<1, 2>(dl - nl, pl, dr - nr, pr, dr - dl, pc, FX_C_L, eps.m, eps.u - 2 * u - 64, w1, w2);
  return pc + fx_dot2<3>(fx_split(pl + pl - pc), fx_split(w1), fx_split(pr + pr - pc), fx_split(w2));
}

}  // namespace hw
