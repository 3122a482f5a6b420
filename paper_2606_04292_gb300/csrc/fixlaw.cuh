// The constitutive laws of Table 1 for FP64 heads in 64-bit fixed point.
//
// FP64 arithmetic issues at ~1.6 operations per clock and SM on this GPU (a
// dependent one takes 64 cycles), so a law built from FP64 exponentials and
// logarithms -- 50 to 80 FP64 operations -- costs as much issue time as 4000
// FP32 instructions.  Integer multiply-adds issue 40 times as often.  Here
// the powers of a law are taken in base 2 as integers: a logarithm or
// exponent is a signed 64-bit number with 56 fraction bits (8 integer bits),
// a function value a 64-bit significand with an exponent.  One law is a few
// 64 x 64-bit products (a product's high word: three 32-bit multiplies),
// ~300 integer instructions in all, and needs FP64 only to put the rounded
// saturation into theta = theta_r + (theta_s - theta_r) Se.
//
//   log2 x:  x = 2^e M; c_j from a 65-entry table (8 bits, the least multiple
//            of 1/256 above 64/(64 + j), j the first six bits of M) makes
//            z = c_j M - 1 in [0, 0.0192), exactly, in one 64-bit product;
//            log2 M = -log2 c_j + z Q(z), Q the Taylor series of
//            log2(1 + z)/z to z^10 (remainder < 2^-65).
//   2^-u:    u = i + k/64 + r, 0 <= r < 1/64; 2^-u = 2^-i T_k (1 - r S(r)), T_k
//            a 64-entry table, S the Taylor series of (1 - 2^-r)/r to r^7
//            (remainder < 2^-70).
// The high-order terms of both series run in 32 bits: their weight z^5 (r^4)
// is below 2^-28 (2^-24), so 34 (41) fraction bits keep 2^-62.
//
// The laws in these terms (T = (alpha h)^n, t = log2 T; Haverkamp: T =
// h^beta / alpha with m = 1):
//   Se     = 2^(-m log2(1 + T)),        log2(1 + T) = log2(1 + 2^-|t|) + max(t, 0)
//   Se'    = n m Se T / (h (1 + T))     = (n - 1) 2^(-(log2(1 + T) - t) - log2 h - m log2(1 + T))
//   K/Ks   = 2^(-l m log2(1 + T)) (1 - 2^(-m (log2(1 + T) - t)))^2
// log2(1 + 2^-|t|) and 1 - 2^-u keep their relative accuracy for small
// arguments: there the series multiplies the normalised argument itself.
//
// Errors over 4e6 random soils and heads (alpha 0.3-5, n 1.05-5.5, l -2-2.5, h
// 1e-6-150; Haverkamp beta 0.5-5) against 64-bit significands, in ulps of the
// result, largest / rms: van Genuchten Se 1.1/0.30, slope 1.8/0.53, K/Ks
// 2.1/0.35; Haverkamp Se 0.9/0.27, slope 1.7/0.48, K/Ks 0.8/0.27; Gardner
// 0.8/0.30.  (In FP64 the exponent carries the rounding of n log(alpha h): tens
// of ulps.)
// Measured against the table-driven FP64 functions (GB300): theta and K of
// 128^3 cells 840 -> 118 us; preparation of a 256^3 step 6.23 -> 1.38 ms; its
// FP64 outer defect 3.96 -> 1.66 ms (the stencil's FP64 remains); an FP64
// half-sweep of 96^3 244 -> 134 us.  Bound by the integer multiplies.
//
// Arguments outside the ranges the integers hold (a head or alpha outside
// 2^+-100, an exponent |t| above 120, n outside [1/32, 16): the 2^-57 of
// log2 is carried into t n times) take the FP64 functions of fp64math.cuh (slow_* in device.cuh).
//
// A host compiler takes this file as well (the laws' integer arithmetic is
// tested so, without a device).
#pragma once

#include <cmath>
#include <cstring>

#ifdef __CUDACC__
#include "fp64math.cuh"
#define RICH_FD __device__ __forceinline__
#else
#define __device__
#include "fp64_tables.h"
#undef __device__
#define RICH_FD inline
#endif

namespace rich {
namespace fl {

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned u32;

#ifdef __CUDACC__
RICH_FD u32 mulhi32(u32 a, u32 b) { return __umulhi(a, b); }
RICH_FD u64 mulhi_exact(u64 a, u64 b) { return __umul64hi(a, b); }
RICH_FD int clz64(u64 a) { return __clzll((long long)a); }
RICH_FD u64 dbits(double x) { return (u64)__double_as_longlong(x); }
RICH_FD double bitsd(u64 b) { return __longlong_as_double((long long)b); }
RICH_FD u32 rcp_bits(u32 b) { return __float_as_uint(__frcp_rn(__uint_as_float(b))); }
static __device__ __noinline__ double slow_div(double a, double b) { return a / b; }
#else
template <typename B, typename A>
inline B bit_copy(A a) {
  static_assert(sizeof(A) == sizeof(B), "same size");
  B b;
  std::memcpy(&b, &a, sizeof b);
  return b;
}
inline u32 mulhi32(u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); }
inline u64 mulhi_exact(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
inline int clz64(u64 a) { return a ? __builtin_clzll(a) : 64; }
inline u64 dbits(double x) { return bit_copy<u64>(x); }
inline double bitsd(u64 b) { return bit_copy<double>(b); }
inline u32 rcp_bits(u32 b) { return bit_copy<u32>(1.0f / bit_copy<float>(b)); }
inline double slow_div(double a, double b) { return a / b; }
using std::fma;
#endif

// high word of a 64 x 64-bit product, at most 3 below the exact one (the
// low x low product and the carries of the cross products are dropped)
RICH_FD u64 mh(u64 a, u64 b) {
  const u32 al = (u32)a, ah = (u32)(a >> 32), bl = (u32)b, bh = (u32)(b >> 32);
  return (u64)ah * bh + ((u64)mulhi32(ah, bl) + (u64)mulhi32(al, bh));
}

// right shift that gives 0 from 64 on
RICH_FD u64 shr(u64 a, int s) { return s > 63 ? 0ull : a >> s; }

// log2(1 + z)/z at scale 2^62, z < 0.0192 at scale 2^64
RICH_FD u64 log_series(u64 z) {
  const u32 zh = (u32)(z >> 32);
  u32 s = LQ9 - mulhi32(zh, LQ10);
  s = LQ8 - mulhi32(zh, s);
  s = LQ7 - mulhi32(zh, s);
  s = LQ6 - mulhi32(zh, s);
  s = LQ5 - mulhi32(zh, s);
  u64 S = LQ4 - mh(z, (u64)s << 28);
  S = LQ3 - mh(z, S);
  S = LQ2 - mh(z, S);
  S = LQ1 - mh(z, S);
  return LQ0 - mh(z, S);
}

// (1 - 2^-r)/r at scale 2^64, r < 1/64 at scale 2^64
RICH_FD u64 exp_series(u64 r) {
  const u32 rh = (u32)(r >> 32);
  u32 s = EG6 - mulhi32(rh, EG7);
  s = EG5 - mulhi32(rh, s);
  s = EG4 - mulhi32(rh, s);
  u64 S = EG3 - mh(r, (u64)s << 23);
  S = EG2 - mh(r, S);
  S = EG1 - mh(r, S);
  return EG0 - mh(r, S);
}

// log2 of M 2^-61 in [1, 2] at scale 2^62; *z (scale 2^64) and *j: its reduction
RICH_FD u64 log2_mant(u64 M) {
  const int j = (int)(M >> 55) - 64;
  const u64* __restrict__ T = kLog2C[j];
  const u64 z = (M * T[0]) >> 5;         // (c_j M - 1) 2^69 mod 2^64: the 1 drops out
  return T[1] + mh(z, log_series(z));
}

RICH_FD bool normal_pos(u64 b) { return b - 0x0010000000000000ull < 0x7fe0000000000000ull; }

// log2 x, scale 2^56, for a positive normal x within 2^+-100
RICH_FD i64 log2_fix(u64 b, bool& ok) {
  const int e = (int)(b >> 52) - 1023;
  ok = ok && normal_pos(b) && e >= -100 && e < 100;
  const u64 M = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 9;
  return ((i64)e << 56) + (i64)((log2_mant(M) + 32) >> 6);
}

// log2 (x y): the product of the significands is kept to 62 bits
RICH_FD i64 log2_prod(u64 a, u64 b, bool& ok) {
  int e = (int)(a >> 52) + (int)(b >> 52) - 2046;
  ok = ok && normal_pos(a) && normal_pos(b) && e >= -100 && e < 100;
  const u64 A = (a << 11) | 0x8000000000000000ull, B = (b << 11) | 0x8000000000000000ull;
  u64 M = mh(A, B);                       // scale 2^62, in [1, 4)
  const int up = (int)(M >> 63);
  M >>= 1 + up;
  return ((i64)(e + up) << 56) + (i64)((log2_mant(M) + 32) >> 6);
}

// n 2^58 for n in [1/32, 16)
RICH_FD u64 to_fix58(u64 b, bool& ok) {
  const int e = (int)(b >> 52) - 1023;
  ok = ok && e >= -5 && e < 4;             // (negative, zero, infinite and NaN bits fail)
  return ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << ((6 + e) & 15);
}

// 1/y for y in [1, 2) at scale 2^63; the result at scale 2^64 (at most
// 2^64 - 1), within 2^-61: a 24-bit seed and two Newton-Raphson steps
// r <- r + r (1 - y r)
RICH_FD u64 recip_mant(u64 y) {
  const u32 rb = rcp_bits(0x3f800000u | ((u32)(y >> 40) & 0x7fffffu));   // in (1/2, 1]
  const u32 r0 = rb >= 0x3f800000u ? 0xffffff00u : ((rb & 0x7fffffu) | 0x800000u) << 8;
  const i64 e0 = (i64)(0x8000000000000000ull - ((y >> 32) * r0 + mulhi32((u32)y, r0)));   // scale 2^63
  const u64 r1 = ((u64)r0 << 32) + (u64)(((i64)(int)(e0 >> 11) * (i64)r0) >> 20);
  const i64 e1 = (i64)(0x8000000000000000ull - mh(y, r1));
  const i64 d = ((i64)(r1 >> 32) * e1) >> 31;
  const u64 r2 = r1 + (u64)d;
  return (d > 0 && r2 < r1) ? ~0ull : r2;
}

// 1 - 1/n at scale 2^64, n > 1 with the significand and exponent of b
RICH_FD u64 one_minus_inv(u64 b) {
  const int e = (int)(b >> 52) - 1023;     // 0 .. 3
  return 0ull - (recip_mant((b << 11) | 0x8000000000000000ull) >> (e & 7));
}

// a value m 2^(e - 63)
struct Val {
  u64 m;
  int e;
};

// 2^-(i + F 2^-64)
RICH_FD Val exp2_neg(int i, u64 F) {
  const u64 T = kExp2N[F >> 58];
  const u64 r = F & 0x03ffffffffffffffull;
  Val v;
  v.m = T - mh(T, mh(r, exp_series(r)));
  v.e = -i;
  return v;
}
// 2^-u, u at scale 2^56, u >= 0
RICH_FD Val exp2_neg56(u64 u) { return exp2_neg((int)(u >> 56), u << 8); }

// m 2^(e - 63) rounded to nearest; m != 0, the result a normal double
RICH_FD double to_double(Val v) {
  const int sh = clz64(v.m);
  const u64 m = v.m << sh;
  return bitsd(((u64)(v.e - sh + 1022) << 52) + (m >> 11) + ((m >> 10) & 1));
}
// (significand in [2^62, 2^63], as exp2_neg gives it)
RICH_FD double to_double_1(Val v) {
  const int sh = 1 - (int)(v.m >> 63);
  const u64 m = v.m << sh;
  return bitsd(((u64)(v.e - sh + 1022) << 52) + (m >> 11) + ((m >> 10) & 1));
}

// The power T = 2^t of a law and log2(1 + T).
struct Pow {
  i64 t;                  // scale 2^56
  u64 L1;                 // log2(1 + T), scale 2^56
  u64 l1;                 // log2(1 + 2^-|t|) = l1 2^(-61 - s)
  int s;
};
RICH_FD Pow pow_log1p(i64 t) {
  Pow p;
  p.t = t;
  const u64 w = (u64)(t < 0 ? -t : t);
  const Val e = exp2_neg56(w);             // 2^-|t| = e.m 2^(-63 - i)
  const int i = -e.e;
  const u64 f = shr(e.m, 2 + i);           // scale 2^61, at most 2^61
  const int j = (int)(f >> 55);
  const u64* __restrict__ T = kLog2C[j];
  const u64 z = ((0x2000000000000000ull + f) * T[0]) >> 5;
  const u64 S = log_series(z);
  // (j = 0: c_j = 1 and z = 2^-|t|, whose normalised significand is e.m)
  const u64 P = mh(j ? z : e.m, S);
  p.l1 = j ? (T[1] + P) >> 1 : P;
  p.s = j ? 0 : i;
  p.L1 = shr(p.l1, 5 + p.s) + (u64)(t > 0 ? t : 0);
  return p;
}

// a + b at scale 2^56; ok: |a + b| < 120 (tested on the halves: the sum of two
// such numbers can leave the 64-bit range)
RICH_FD i64 add_log(i64 a, i64 b, bool& ok) {
  const i64 h = (a >> 1) + (b >> 1);
  ok = ok && h < (60ll << 56) && h > -(60ll << 56);
  return (i64)((u64)a + (u64)b);
}

// n x for n at scale 2^58 and x at scale 2^56; ok: |n x| < 120
RICH_FD i64 scale_log(u64 n, i64 x, bool& ok) {
  const u64 ax = (u64)(x < 0 ? -x : x);
  const u64 hi = mulhi_exact(n, ax), lo = n * ax;          // scale 2^114
  ok = ok && hi < (120ull << 50);
  const i64 t = (i64)((hi << 6) | (lo >> 58));
  return x < 0 ? -t : t;
}

// ---------------------------------------------------------------------------
// One cell's parameters of the van Genuchten power (alpha h)^n, or of
// Haverkamp's h^beta / alpha, prepared once per point solve: la = log2 alpha,
// N = n (beta), M = m = 1 - 1/n.
// ---------------------------------------------------------------------------
struct Prep {
  i64 la;                 // scale 2^56
  u64 N, M;               // scale 2^58, 2^64
  bool ok;
};
template <bool VG>
RICH_FD Prep prep(double p1, double p2) {
  Prep q;
  q.ok = true;
  q.la = log2_fix(dbits(p1), q.ok);
  const u64 b = dbits(p2);
  q.N = to_fix58(b, q.ok);
  q.M = 0;
  if (VG) {
    q.ok = q.ok && b > 0x3ff0000000000000ull;
    q.M = one_minus_inv(b);
  }
  return q;
}

// The same on the host, for parameters known before a launch (a uniform soil,
// a material): log2 in extended precision, the reciprocal by exact division.
inline Prep host_prep(bool vg, double p1, double p2) {
  Prep q{0, 0, 0, false};
  const double ap = std::fabs(p1);
  if (!(p1 > 0.0) || !(ap > 0x1p-100 && ap < 0x1p100)) return q;
  if (!(p2 >= 1.0 / 32 && p2 < 16.0) || (vg && !(p2 > 1.0))) return q;
  q.la = (i64)std::llrintl(std::log2((long double)p1) * 0x1p56L);
  q.N = (u64)(p2 * 0x1p58);            // exact: p2 has 53 bits and is at least 2^-5
  if (vg) {
    int e;
    const u64 m = (u64)(std::frexp(p2, &e) * 0x1p53);               // p2 = m 2^(e - 53)
    const unsigned __int128 inv = ((unsigned __int128)1 << 117) / m;   // 2^64 / p2 = 2^(117 - e) / m
    q.M = 0ull - (u64)(inv >> e);
  }
  q.ok = true;
  return q;
}

// theta's exponent: Se = 2^-u (scale 2^56)
template <bool VG>
RICH_FD u64 se_exponent(const Pow& p, u64 M) {
  return VG ? mh(M, p.L1) : p.L1;
}

// Se of the power T = 2^t, and s = d Se/d psi without its factor (n - 1, beta)
template <bool VG>
RICH_FD void se_slope(const Prep& q, u64 hb, bool& ok, double& Se, double& s) {
  const i64 lh = log2_fix(hb, ok);
  const i64 t = VG ? scale_log(q.N, add_log(q.la, lh, ok), ok) : add_log(scale_log(q.N, lh, ok), -q.la, ok);
  const Pow p = pow_log1p(t);
  const u64 u = se_exponent<VG>(p, q.M);
  Se = to_double_1(exp2_neg56(u));
  // log2(1 + T) - t + log2 h + u at scale 2^54 (up to 470 in magnitude)
  const u64 w = shr(p.l1, 5 + p.s) + (u64)(t < 0 ? -t : 0);
  const i64 D = (i64)(w >> 2) + (i64)(u >> 2) + (lh >> 2);
  s = to_double_1(exp2_neg((int)(D >> 54), (u64)D << 10));
}

// Se alone of a prepared law
template <bool VG>
RICH_FD u64 prepared_u(const Prep& q, u64 hb, bool& ok) {
  const i64 lh = log2_fix(hb, ok);
  const i64 t = VG ? scale_log(q.N, add_log(q.la, lh, ok), ok) : add_log(scale_log(q.N, lh, ok), -q.la, ok);
  return se_exponent<VG>(pow_log1p(t), q.M);
}
template <bool VG>
RICH_FD double se_prepared(const Prep& q, u64 hb, bool& ok) {
  return to_double_1(exp2_neg56(prepared_u<VG>(q, hb, ok)));
}

// Se alone, from alpha (p1), n (p2) and h: its exponent, Se = 2^-u (scale 2^56)
template <bool VG>
RICH_FD u64 se_u(double p1, double p2, u64 hb, bool& ok) {
  const u64 nb = dbits(p2);
  const u64 N = to_fix58(nb, ok);
  i64 t;
  u64 M = 0;
  if (VG) {
    ok = ok && nb > 0x3ff0000000000000ull;
    M = one_minus_inv(nb);
    t = scale_log(N, log2_prod(dbits(p1), hb, ok), ok);
  } else {
    t = add_log(scale_log(N, log2_fix(hb, ok), ok), -log2_fix(dbits(p1), ok), ok);
  }
  return se_exponent<VG>(pow_log1p(t), M);
}
template <bool VG>
RICH_FD double se_only(double p1, double p2, u64 hb, bool& ok) {
  return to_double_1(exp2_neg56(se_u<VG>(p1, p2, hb, ok)));
}

// K/Ks of Haverkamp: A/(A + h^gamma)
RICH_FD double kr_haverkamp(double A, double gamma, u64 hb, bool& ok) {
  return se_only<false>(A, gamma, hb, ok);
}

// K/Ks of van Genuchten-Mualem: Se^l (1 - (T/(1 + T))^m)^2
RICH_FD double kr_vangenuchten(double alpha, double n, double l, u64 hb, bool& ok) {
  const u64 nb = dbits(n);
  ok = ok && nb > 0x3ff0000000000000ull;
  const u64 M = one_minus_inv(nb);
  const i64 t = scale_log(to_fix58(nb, ok), log2_prod(dbits(alpha), hb, ok), ok);
  const Pow p = pow_log1p(t);
  // u = m (log2(1 + T) - t) as a 128-bit product, its scale 2^(64 + sc + s0)
  const bool dry = t >= 0;
  const u64 X = dry ? p.l1 : shr(p.l1, 5 + p.s) + (u64)(-t);
  const int sc = dry ? 61 : 56, s0 = dry ? p.s : 0;
  const u64 hi = mulhi_exact(M, X), lo = M * X;
  const int i = dry ? 0 : (int)(hi >> 56);
  // (s0 > 0 means 2^-|t| < 1/64, so s0 >= 6 or s0 = 5 with |t| = 6 + rounding)
  const u64 F = !dry ? (hi << 8) | (lo >> 56) : (s0 ? shr(hi, s0 - 3) : (hi << 3) | (lo >> 61));
  const u64 r = F & 0x03ffffffffffffffull;
  const u64 S = exp_series(r);
  // 1 - 2^-u: u S(u) below 1/64 (with u's own normalised significand)
  Val in;
  if (i == 0 && F == r) {
    const int c = clz64(hi) & 63;
    in.m = mh((hi << c) | ((lo >> 1) >> (63 - c)), S);
    in.e = 63 - (c + sc + s0);
  } else {
    const u64 T = kExp2N[F >> 58];
    in.m = 0x8000000000000000ull - shr(T - mh(T, mh(r, S)), i);
    in.e = 0;
  }
  const int c = clz64(in.m) & 63;
  const u64 I = in.m << c;
  Val v;
  v.m = mh(I, I);
  v.e = 2 * (in.e - c) + 1;
  // Se^l: the exponent l m log2(1 + T), l of either sign
  const u64 lb = dbits(l) & 0x7fffffffffffffffull;
  if (lb) {
    i64 q = scale_log(to_fix58(lb, ok), (i64)mh(M, p.L1), ok);
    if (l < 0.0) q = -q;
    const Val E = exp2_neg((int)(q >> 56), (u64)q << 8);
    v.m = mh(v.m, E.m);
    v.e += E.e + 1;
  }
  ok = ok && v.e > -1000;
  return to_double(v);
}

// e^-(alpha h) = 2^-u: u at scale 2^56
RICH_FD u64 gardner_exponent(double alpha, u64 hb, bool& ok) {
  const u64 ab = dbits(alpha);
  const int e = (int)(ab >> 52) + (int)(hb >> 52) - 2046;
  ok = ok && normal_pos(ab) && normal_pos(hb) && e < 6;
  const u64 P = mh((ab << 11) | 0x8000000000000000ull, (hb << 11) | 0x8000000000000000ull);   // scale 2^62
  const u64 u = mh(P, LOG2E_63);                                   // scale 2^61
  return e > 5 ? 0 : shr(u, 5 - e);
}
RICH_FD double exp_gardner(double alpha, u64 hb, bool& ok) {
  return to_double_1(exp2_neg56(gardner_exponent(alpha, hb, ok)));
}

// Any of the three laws, chosen by lane (layered soils): one instruction
// stream for Haverkamp's and van Genuchten's powers (they differ in where
// log2 alpha enters and in the factor m), and Gardner's exponent selected
// before the common 2^-u; a warp that holds several materials then takes one
// law's time instead of their sum.  q: prep of the material (Gardner: N = 1,
// la = 0).  slope: also d Se/d psi without its factor.
enum { ANY_HAVERKAMP = 0, ANY_GARDNER = 1, ANY_VANGENUCHTEN = 2 };
RICH_FD u64 any_u(int law, const Prep& q, double alpha, u64 hb, bool& ok, i64& lh, i64& t, Pow& p) {
  lh = log2_fix(hb, ok);
  const i64 x = add_log(lh, law == ANY_VANGENUCHTEN ? q.la : 0, ok);
  t = add_log(scale_log(q.N, x, ok), law == ANY_HAVERKAMP ? -q.la : 0, ok);
  p = pow_log1p(t);
  return law == ANY_GARDNER ? gardner_exponent(alpha, hb, ok) : law == ANY_VANGENUCHTEN ? mh(q.M, p.L1) : p.L1;
}
template <bool SLOPE>
RICH_FD void se_any(int law, const Prep& q, double alpha, u64 hb, bool& ok, double& Se, double& s) {
  i64 lh, t;
  Pow p;
  const u64 u = any_u(law, q, alpha, hb, ok, lh, t, p);
  Se = to_double_1(exp2_neg56(u));
  if (SLOPE) {
    const u64 w = shr(p.l1, 5 + p.s) + (u64)(t < 0 ? -t : 0);
    const i64 D = (i64)(w >> 2) + (i64)(u >> 2) + (lh >> 2);
    s = to_double_1(exp2_neg((int)(D >> 54), (u64)D << 10));
    if (law == ANY_GARDNER) s = Se;
  }
}

// ---------------------------------------------------------------------------
// FP64 comparisons and quotients off the FP64 pipe (a compare issues there as
// slowly as an add, a division as eight to ten of them).
// ---------------------------------------------------------------------------
// the order of finite and infinite doubles as signed integers (-0 = +0)
RICH_FD i64 order_key(double x) {
  const i64 b = (i64)dbits(x);
  return b < 0 ? (i64)(0x8000000000000000ull - (u64)b) : b;
}
RICH_FD bool is_nan(double x) { return (dbits(x) << 1) > 0xffe0000000000000ull; }

// A divisor b and its reciprocal, rounded to nearest from 61 bits (integer
// Newton-Raphson).  div(a) is Markstein's quotient (IBM J. Res. Dev. 34,
// 1990): q = a y, then q + (a - b q) y.  It is the correctly rounded a/b for a
// correctly rounded y; this y can be the other neighbour (about once in 1200
// times), where correctness is tested and not proven: none of 2e8 random
// quotients differed from a/b.  Exponents near the ends of the range, where
// a - b q could leave it, divide plainly.
struct Divisor {
  double b, y;
  int e;
};
RICH_FD Divisor divisor(double b) {
  Divisor d;
  const u64 k = dbits(b);
  const int e = (int)((k >> 52) & 0x7ff);
  const u64 r = recip_mant((k << 11) | 0x8000000000000000ull);
  d.b = b;
  d.e = e;
  d.y = bitsd((k & 0x8000000000000000ull) | (((u64)(2044 - e) << 52) + (r >> 11) + ((r >> 10) & 1)));
  return d;
}
// whether div applies: 2^-400 <= |a|, |b| < 2^400, or a = 0
RICH_FD bool div_ok(double a, const Divisor& d) {
  const u64 k = dbits(a) << 1;
  return (u32)(d.e - 623) < 800u && ((u32)((int)(k >> 53) - 623) < 800u || k == 0);
}
RICH_FD double div(double a, const Divisor& d) {
  if (!div_ok(a, d)) return slow_div(a, d.b);
  const double q = a * d.y;
  return fma(fma(-q, d.b, a), d.y, q);
}

}  // namespace fl
}  // namespace rich
