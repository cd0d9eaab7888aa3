// fx64.cuh -- the transcendental functions of the FP64 paths in 64-bit
// fixed point: Box-Muller's logarithm, square root, sine and cosine, the
// logistic function of the tanh volatilities, and the exponential.
//
// GB300 runs FP64 on a pipe of two lanes per SM and clock: one FP64
// instruction of a warp takes as long as 64 issue slots, an integer 32 x 32
// -> 64 multiply-add about four.  The arguments of Box-Muller are 33-bit
// integers and its results are bounded, so tables, exact residuals and short
// Taylor polynomials in 64-bit integers give them with absolute errors of
// 2^-57 and below, less than the rounding of an FP64 library sequence, in a
// few tens of integer instructions instead of a few tens of FP64 ones.
// FP64 remains for the state itself (its range is unbounded) and for the
// polynomial u^k.
//
// Method: argument reduction by a table of cell points (fx64_tables.h), then
// the Taylor polynomial of the remainder, lower-order coefficients at full
// width and higher ones in 32 bits; 1/D and sqrt by Newton steps in integers
// from an approximate FP32 seed.  Error of each step, in units of the last
// place kept, is stated where it is made.
//
// The header also compiles as plain C++ (FX_HOST), which the CPU tests use
// to compare every function with arbitrary-precision values.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef FX_HOST
#include <math.h>
#define FX_FN static inline
#define FX_TABLE static const
#ifndef FX_SEED_ERR
#define FX_SEED_ERR 0.0f  // relative error put on the seeds by the tests
#endif
#else
#define FX_FN __device__ __forceinline__
#define FX_TABLE __device__ const
#endif
#include "fx64_tables.h"

namespace fx64 {

FX_FN uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
FX_FN uint32_t hi32(uint64_t a) { return (uint32_t)(a >> 32); }
FX_FN uint32_t lo32(uint64_t a) { return (uint32_t)a; }
FX_FN uint32_t mulhi32(uint32_t a, uint32_t b) { return hi32(wide(a, b)); }
// floor(a b / 2^64) without the low partial product: too small by at most 2
FX_FN uint64_t mulhi(uint64_t a, uint64_t b) {
  return wide(hi32(a), hi32(b)) + mulhi32(hi32(a), lo32(b)) + mulhi32(lo32(a), hi32(b));
}
// floor(a b / 2^32), b < 2^32
FX_FN uint64_t mulhi_32(uint64_t a, uint32_t b) { return wide(hi32(a), b) + mulhi32(lo32(a), b); }
FX_FN int64_t swide(int32_t a, int32_t b) { return (int64_t)a * b; }

#ifdef FX_HOST
FX_FN int clz(uint64_t a) { return a ? __builtin_clzll(a) : 64; }
FX_FN float u2f(uint32_t a) { return (float)a; }
FX_FN int32_t f2i(float a) { return a >= 2147483648.0f ? 2147483647 : (int32_t)a; }
FX_FN float rsqrt_seed(float a) { return (float)(1.0 / sqrt((double)a)) * (1.0f + FX_SEED_ERR); }
FX_FN float rcp_seed(float a) { return 1.0f / a * (1.0f + FX_SEED_ERR); }
FX_FN uint64_t bits(double x) {
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
}
FX_FN double from_bits(uint64_t b) {
  double x;
  memcpy(&x, &b, 8);
  return x;
}
FX_FN double exp_lib(double x) { return ::exp(x); }
FX_FN double log_lib(double x) { return ::log(x); }
FX_FN void load2(const uint64_t* t, uint64_t& a, uint64_t& b) {
  a = t[0];
  b = t[1];
}
FX_FN uint64_t load1(const uint64_t* t) { return *t; }
#else
FX_FN int clz(uint64_t a) { return __clzll((long long)a); }
FX_FN float u2f(uint32_t a) { return __uint2float_rn(a); }
FX_FN int32_t f2i(float a) { return __float2int_rz(a); }  // saturates
FX_FN float rsqrt_seed(float a) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
FX_FN float rcp_seed(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
FX_FN uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
FX_FN double from_bits(uint64_t b) { return __longlong_as_double((long long)b); }
FX_FN double exp_lib(double x) { return ::exp(x); }
FX_FN double log_lib(double x) { return ::log(x); }
FX_FN void load2(const uint64_t* t, uint64_t& a, uint64_t& b) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(t));
  a = v.x;
  b = v.y;
}
FX_FN uint64_t load1(const uint64_t* t) {
  return __ldg(reinterpret_cast<const unsigned long long*>(t));
}
#endif

// a >> n for 0 <= n, zero from n = 64 on
FX_FN uint64_t shr(uint64_t a, int n) { return n < 64 ? a >> n : 0; }

// m 2^e (m != 0) rounded to the nearest double, in its normal range
FX_FN double pack(uint64_t m, int e, uint32_t negative) {
  const int c = clz(m);
  const uint64_t n = m << c;  // value n 2^(e - c), n in [2^63, 2^64)
  const uint64_t r = (n >> 11) + ((n >> 10) & 1);
  return from_bits(r + ((uint64_t)(uint32_t)(e - c + 63 + 1022) << 52) + ((uint64_t)negative << 63));
}

// A positive double as sm 2^(se - 64), sm in [2^63, 2^64); false when it is
// not a normal number well inside the range (zero, NaN, huge, tiny).
struct Scale {
  uint64_t sm;
  int se;
};
FX_FN bool to_scale(double x, Scale& s) {
  const uint64_t b = bits(x);
  const int e = (int)(b >> 52);  // the sign bit too: negative numbers fail the test
  s.sm = 0x8000000000000000ull | (b << 11);
  s.se = e - 1022;
  return e > 523 && e < 1523;
}

// -ln((2 w + 1) 2^-33) at 2^sc.  u = y 2^-lz with y in [1/2, 1); table
// c with y c = 1 - rho (rho exact, 0 < rho < 2^-7), then
// -ln u = lz ln 2 + ln c + rho + rho^2 P(rho): absolute error below 2^-57.
// sc = 59; in the cell next to u = 1, where ln c = 0 and the result falls to
// 2^-33, sc = 69, so that its square root keeps an absolute error of 2^-53.
FX_FN uint64_t neg_log(uint32_t w, int& sc) {
  const uint64_t M = ((uint64_t)w << 32) | 0x80000000u;
  const int lz = clz(M);
  const uint64_t Y = M << lz;
  const int j = (int)(Y >> 56) & 127;
  uint64_t c, lnc;
  load2(FX_LOG_TAB + 2 * j, c, lnc);
  const uint64_t y33 = Y >> 31;  // exact: 33 significant bits, the top one set
  const uint64_t rho = (1ull << 48) - (wide(lo32(y33), lo32(c)) + (c << 32));
  const uint64_t s = rho << 22;  // sigma = 64 rho < 1/2 at 2^64
  const uint32_t sh = hi32(s);
  // P = sum sigma^n / ((n + 2) 64^n): error below 2^-51, times rho^2 < 2^-13.9
  const uint32_t q5 = (uint32_t)FX_LOG_C5 + mulhi32(sh, (uint32_t)FX_LOG_C6);
  const uint64_t q4 = FX_LOG_C4 + mulhi32(sh, q5);
  const uint64_t q3 = FX_LOG_C3 + mulhi_32(q4, sh);
  const uint64_t q2 = FX_LOG_C2 + mulhi_32(q3, sh);
  const uint64_t P = FX_LOG_C0 + mulhi(s, FX_LOG_C1 + mulhi(s, q2));
  const uint64_t s2 = wide(sh, sh) + ((uint64_t)mulhi32(sh, lo32(s)) << 1);
  const int up = (lz == 0 && j == 127) ? 10 : 0;
  sc = 59 + up;
  const uint64_t l2 = (wide(lz, hi32(FX_LN2_64)) << 27) + (wide(lz, lo32(FX_LN2_64)) >> 5);
  return l2 + lnc + (rho << (11 + up)) + (mulhi(s2, P) >> (17 - up));
}

// sqrt of A (at 2^58), as S 2^(e - 63), S in [2^62, 2^63]: two Newton steps
// on exact residuals from an FP32 seed.  The seed may be off by 2^-22 (the
// instruction: 2^-22.9), so that the residual a - s0^2 stays below 2^-20 and its
// leading 32 bits fit the product; after the steps 2^-42 and 2^-61.  Next to
// a = 1 a seed rounded up gives s0 = 1, which has no place at 2^32: s0 is held at
// 1 - 2^-32 then.
FX_FN uint64_t sqrt58(uint64_t A, int& e) {
  const int e2 = clz(A) & ~1;
  const uint64_t a = A << e2;  // [1/4, 1) at 2^64
  const int32_t rs = f2i(rsqrt_seed(u2f(hi32(a)) * 2.3283064365386963e-10f) * 1073741824.0f);  // at 2^30
  const uint32_t s30 = mulhi32(hi32(a), (uint32_t)rs);                                         // at 2^30
  const uint32_t s0 = s30 >= (1u << 30) ? 0xffffffffu : s30 << 2;                              // at 2^32
  const int64_t e0 = (int64_t)(a - wide(s0, s0));
  const uint64_t s1 = ((uint64_t)s0 << 31) + (uint64_t)(swide((int32_t)(e0 >> 13), rs) >> 19);  // at 2^63
  const uint64_t t1 = s1 >> 16;                                                                 // at 2^47
  // the low 64 bits of a 2^94 - t1^2, a number below 2^53 in size
  const uint64_t t1sq = wide(lo32(t1), lo32(t1)) + ((uint64_t)(lo32(t1) * hi32(t1)) << 33);
  const int64_t e1 = (int64_t)((a << 30) - t1sq);
  e = 3 - (e2 >> 1);
  return (t1 << 16) + (uint64_t)(swide((int32_t)(e1 >> 22), rs) >> 40);
}

// |sin| and |cos| (at 2^63) of the phase (2 w + 1) 2^-33 revolutions within
// its quadrant: the cell point's from the table, the rest delta = f pi/128,
// |f| <= 1/2, by Taylor polynomials; absolute error below 1.3 2^-60 (1.25 2^-60 at w = 855513624, the
// largest of all words)
FX_FN void trig_quadrant(uint32_t w, uint64_t& sn, uint64_t& cs) {
  const uint32_t r = (w << 2) | 2u;  // fraction of the quadrant at 2^32, exact
  uint64_t Sj, Cj;
  load2(FX_TRIG_TAB + 2 * (r >> 26), Sj, Cj);
  const uint32_t d = r << 6;  // fraction of the cell at 2^32, exact
  const bool neg = d < 0x80000000u;
  const uint32_t F = neg ? 0x80000000u - d : d - 0x80000000u;  // |f| at 2^32
  const uint64_t g = wide(F, F);
  const uint32_t gh = hi32(g);
  // sin delta = f K(f^2) and 1 - cos delta, at 2^64
  const uint32_t k5 = (uint32_t)FX_TRIG_K5 - mulhi32(gh, (uint32_t)FX_TRIG_K7);
  const uint64_t k3 = FX_TRIG_K3 - mulhi32(gh, k5);
  const uint64_t K = FX_TRIG_K1 - mulhi(g, k3);
  const uint64_t sd = mulhi_32(K, F);
  const uint64_t k4 = FX_TRIG_K4 - mulhi32(gh, (uint32_t)FX_TRIG_K6);
  const uint64_t vc = mulhi(g, FX_TRIG_K2 - mulhi_32(k4, gh));
  const uint64_t a = mulhi(Cj, sd), b = mulhi(Sj, sd);
  sn = Sj - mulhi(Sj, vc);
  cs = Cj - mulhi(Cj, vc);
  sn = neg ? sn - a : sn + a;
  cs = neg ? cs + b : cs - b;
}

// |z0| and |z1| of a Box-Muller pair, z = sm sqrt(-2 ln u0) (cos, sin)(2 pi u1),
// u = (2 w + 1) 2^-33, as m 2^(e - 62), with their signs (0 or 1)
FX_FN void box_muller_parts(uint32_t w0, uint32_t w1, uint64_t sm, uint64_t& m0, uint64_t& m1, int& e,
                            uint32_t& n0, uint32_t& n1) {
  int at;
  const uint64_t L = neg_log(w0, at);  // -ln u0 at 2^59 is -2 ln u0 at 2^58
  const uint64_t S = mulhi(sqrt58(L, e), sm);
  e -= (at - 59) >> 1;
  uint64_t sn, cs;
  trig_quadrant(w1, sn, cs);
  const uint32_t qd = w1 >> 30;
  m0 = mulhi(S, (qd & 1) ? sn : cs);  // S and the trigonometric factor at 2^63, shifted by 64
  m1 = mulhi(S, (qd & 1) ? cs : sn);
  n0 = (qd ^ (qd >> 1)) & 1;
  n1 = qd >> 1;
}

// the pair times the scale, rounded once to double
FX_FN void box_muller(uint32_t w0, uint32_t w1, const Scale& sc, double& z0, double& z1) {
  uint64_t m0, m1;
  uint32_t n0, n1;
  int e;
  box_muller_parts(w0, w1, sc.sm, m0, m1, e, n0, n1);
  e += sc.se - 62;
  z0 = pack(m0, e, n0);
  z1 = pack(m1, e, n1);
}

// the pair (sm without the power of two of the scale) as signed numbers at 2^60;
// |z| < 6.8
FX_FN void box_muller_fixed(uint32_t w0, uint32_t w1, uint64_t sm, int64_t& z0, int64_t& z1) {
  uint64_t m0, m1;
  uint32_t n0, n1;
  int e;  // at most 3
  box_muller_parts(w0, w1, sm, m0, m1, e, n0, n1);
  const int64_t a = (int64_t)((m0 << 1) >> (3 - e)), b = (int64_t)((m1 << 1) >> (3 - e));
  z0 = n0 ? -a : a;
  z1 = n1 ? -b : b;
}

// a b / 2^64 of signed numbers, to within 2
FX_FN int64_t smulhi(int64_t a, int64_t b) {
  const uint64_t m = mulhi((uint64_t)(a < 0 ? -a : a), (uint64_t)(b < 0 ? -b : b));
  return ((a ^ b) < 0) ? -(int64_t)m : (int64_t)m;
}

// y 2^(se - 58) as a double, to within 2^-58 2^se
FX_FN double from_fixed58(int64_t y, int se) {
  return pack((uint64_t)(y < 0 ? -y : y) | 1u, se - 58, y < 0 ? 1u : 0u);
}

// x at 2^57 when |x| < 32 (exact to 2^-57); false otherwise, NaN included
FX_FN bool to_fixed57(double x, int64_t& r) {
  const uint64_t b = bits(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  const int64_t v = (int64_t)shr(0x8000000000000000ull | (b << 11), 1029 - (ex > 1027 ? 1027 : ex));
  r = (int64_t)b < 0 ? -v : v;
  return ex <= 1027;
}

// 2^(-f), f = f57 2^-57 in [0, 1), at 2^63: error below 2^-61
FX_FN uint64_t pow2_neg(uint64_t f57) {
  const uint64_t T = load1(FX_EXP_TAB + (int)(f57 >> 50));
  const uint64_t g = (f57 & ((1ull << 50) - 1)) << 14;  // fraction of the cell at 2^64
  const uint32_t gh = hi32(g);
  const uint32_t b5 = (uint32_t)FX_EXP_L5 - mulhi32(gh, (uint32_t)FX_EXP_L6);
  const uint32_t b4 = (uint32_t)FX_EXP_L4 - mulhi32(gh, b5);
  const uint64_t b3 = FX_EXP_L3 - mulhi32(gh, b4);
  const uint64_t b2 = FX_EXP_L2 - mulhi(g, b3);
  const uint64_t m = mulhi(g, FX_EXP_L1 - mulhi(g, b2));
  return T - mulhi(T, m);
}

// 1 + r in [1, 2] with r = 1 / (1 + E) (inverse false: 1 - that), E = 2^-t,
// t at 2^57, t < 128: absolute error below 2^-52.8, the result's rounding and the
// truncation of t (largest of 10^9 arguments: 2^-52.95 from a double, 2^-52.85 in fixed point)
FX_FN double logistic_of(uint64_t t, bool complement) {
  const uint64_t E = shr(pow2_neg(t & ((1ull << 57) - 1)), (int)(t >> 57));
  // q = 1 / (1 + E) in [1/2, 1]: R (1 + e + e^2), e = 1 - (1 + E) R exact to 2^-61
  const uint64_t D = (1ull << 62) + (E >> 1);
  const uint32_t R = (uint32_t)f2i(rcp_seed(u2f(hi32(D)) * 9.3132257461547852e-10f) * 1073741824.0f) << 1;  // at 2^31
  const int64_t e0 = (int64_t)((1ull << 61) - mulhi_32(D, R));
  const int32_t es = (int32_t)(e0 >> 9);
  const int64_t w = e0 + (swide(es, es) >> 43);
  const int64_t Rw = (int64_t)((uint64_t)((int64_t)(int32_t)(w >> 32) * R) + mulhi32(lo32((uint64_t)w), R));
  const uint64_t q = ((uint64_t)R << 32) + ((uint64_t)Rw << 3);  // at 2^63
  const uint64_t r = complement ? (1ull << 63) - q : q;
  return from_bits(0x3ff0000000000000ull + ((r + 0x400) >> 11));
}

// 1 + 1 / (e^{2 y} + 1) in [1, 2] (absolute: of |y|); saturates for |y| >= 32
// and for infinities
FX_FN double logistic_p1(double y, bool absolute) {
  const uint64_t b = bits(y);
  const int ex = (int)(b >> 52) & 0x7ff;
  const uint64_t m = 0x8000000000000000ull | (b << 11);
  const uint64_t v = ex > 1027 ? ~0ull : shr(m, 1027 - ex);  // |y| at 2^59
  return logistic_of(mulhi(v, FX_2LOG2E_62), !(b >> 63) || absolute);
}

// the same for y at 2^57, |y| < 64 (saturating beyond 44)
FX_FN double logistic_p1_fixed(int64_t y, bool absolute) {
  const uint64_t t = mulhi((uint64_t)(y < 0 ? -y : y), FX_2LOG2E_62);  // at 2^55
  return logistic_of(t < (1ull << 62) ? t << 2 : ~0ull, y >= 0 || absolute);
}

// e^x: relative error below 2^-52.3 (largest of 5 10^8 arguments 2^-52.39, for |x| < 8
// 2^-52.57); the library's function for |x| >= 256, NaN and infinities
FX_FN double exp(double x) {
  const uint64_t b = bits(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  if (ex > 1030) return exp_lib(x);
  const uint64_t m = 0x8000000000000000ull | (b << 11);
  const uint64_t t = shr(mulhi(m, FX_LOG2E_63), 1031 - ex);  // |x| log2(e) at 2^54
  const int64_t nt = (b >> 63) ? (int64_t)t : -(int64_t)t;   // e^x = 2^-nt
  const uint64_t E = pow2_neg(((uint64_t)nt & ((1ull << 54) - 1)) << 3);
  return pack(E, -63 - (int)(nt >> 54), 0);
}

// ln x within 0.63 ulp for 1/4 <= |ln x|: x = y 2^e, y c = 1 - rho as in neg_log, rho
// exact from the low 64 bits of the product.  The sum e ln 2 + ln y is kept at 2^59, its
// error a few 2^-59, or where it does not fit (x beyond e^+-14.5) at 2^53; next to
// x = 1 it cancels, and the library's function takes over, as it does for x <= 0,
// subnormal numbers, NaN and infinities.
FX_FN double log_abs(double x) {
  const uint64_t b = bits(x);
  const int ex = (int)(b >> 52);
  if (ex == 0 || ex >= 0x7ff) return log_lib(x);
  const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;  // y at 2^53
  uint64_t c, lnc;
  load2(FX_LOG_TAB + 2 * ((int)(m >> 45) & 127), c, lnc);
  const uint64_t rho = 0 - m * c;  // at 2^68, below 2^61
  const uint64_t s = rho << 2;     // 64 rho at 2^64
  const uint32_t sh = hi32(s);
  const uint32_t q5 = (uint32_t)FX_LOG_C5 + mulhi32(sh, (uint32_t)FX_LOG_C6);
  const uint64_t q4 = FX_LOG_C4 + mulhi32(sh, q5);
  const uint64_t q3 = FX_LOG_C3 + mulhi_32(q4, sh);
  const uint64_t q2 = FX_LOG_C2 + mulhi_32(q3, sh);
  const uint64_t P = FX_LOG_C0 + mulhi(s, FX_LOG_C1 + mulhi(s, q2));
  const uint64_t s2 = wide(sh, sh) + ((uint64_t)mulhi32(sh, lo32(s)) << 1);
  const uint64_t ny = lnc + (rho >> 9) + (mulhi(s2, P) >> 17);  // -ln y at 2^59, below 2^59
  const int e = ex - 1022;
  const uint32_t ae = (uint32_t)(e < 0 ? -e : e);
  if (ae > 21) {
    const uint64_t l2 = (wide(ae, hi32(FX_LN2_64)) << 21) + (wide(ae, lo32(FX_LN2_64)) >> 11);  // |e| ln 2 at 2^53
    const int64_t r = (e < 0 ? -(int64_t)l2 : (int64_t)l2) - (int64_t)((ny + 32) >> 6);
    return pack((uint64_t)(r < 0 ? -r : r), -53, r < 0 ? 1u : 0u);
  }
  const uint64_t l2 = (wide(ae, hi32(FX_LN2_64)) << 27) + (wide(ae, lo32(FX_LN2_64)) >> 5);  // |e| ln 2 at 2^59
  const int64_t r = (e < 0 ? -(int64_t)l2 : (int64_t)l2) - (int64_t)ny;
  const uint64_t a = (uint64_t)(r < 0 ? -r : r);
  if (a < (1ull << 57)) return log_lib(x);
  return pack(a, -59, r < 0 ? 1u : 0u);
}

}  // namespace fx64
