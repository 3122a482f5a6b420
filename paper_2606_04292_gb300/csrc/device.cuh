// Device building blocks of the NGS-FAS solver: constitutive laws, the
// conservative 7-point (2d+1) stencil, the bracketed Newton point update,
// the nonlinear defect, and the transfer operators.  Grid kernels and the
// coarse tail both call these functions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fixlaw.cuh"
#include "fp64math.cuh"

namespace rich {

// COMPOSITE: a layered soil (Section 4.1's composite law, Section 4.2's two
// layers); every cell takes the law of its own material.
enum { HAVERKAMP = 0, GARDNER = 1, VANGENUCHTEN = 2, COMPOSITE = 3 };
constexpr int MAXMAT = 8;      // materials of a layered soil

// FORM_DIRECT: the unknown is psi (eq. point-update as written).
// FORM_DELTA:  the unknown is the correction delta to a frozen psi0, and the
//              storage/sink terms are the increments theta(psi0+delta) -
//              theta(psi0), S(psi0+delta) - S(psi0) evaluated without
//              cancellation (the FP32 inner problem of the mixed mode).
enum { FORM_DIRECT = 0, FORM_DELTA = 1 };

constexpr int RMAX = 6;     // max fine cells per coarse cell along one axis

template <typename T>
struct Level {
  int dim, n0, n1, n2;
  long long ncell;
  T ih2[3];                      // 1/h^2 per axis (0 on unused axes)
  T *u, *ubar, *g, *d;           // iterate, FAS restricted iterate, right side, defect
  const T *Kc, *p1, *p2, *smax;  // lagged conductivity, soil params (nullable), sink coef (nullable)
  const T *psi0;                 // FORM_DELTA: frozen state
  const T *kb[6];                // boundary face conductances (per face cell)
  const uint8_t *mat;            // COMPOSITE: material of each cell of this level
  int cs;                        // 1: g, psi0, p1, p2, smax in the colour-split layout (pix)
  unsigned rn0, rnh, rn1;        // quick_div factors of n0, ceil(n0/2), n1 (set_divisors)
};

// t / n for the block loops of the small levels (an integer division is ~20
// dependent instructions, and a phase of the coarse tail does four of them
// per cell): the high word of t ceil(2^32/n) is exact for t n < 2^32.  Factor
// 0: n = 1, or a level too big for it (more than 2^16 cells), which divides.
__host__ __device__ __forceinline__ unsigned div_factor(unsigned n, long long ncell) {
  return n > 1 && ncell <= 65536 ? 0xffffffffu / n + 1 : 0u;
}
__device__ __forceinline__ unsigned quick_div(unsigned t, unsigned n, unsigned factor) {
  if (factor) return __umulhi(t, factor);
  return n == 1 ? t : t / n;
}
template <typename T>
__host__ __device__ __forceinline__ void set_divisors(Level<T>& L) {
  L.rn0 = div_factor((unsigned)L.n0, L.ncell);
  L.rnh = div_factor((unsigned)((L.n0 + 1) >> 1), L.ncell);
  L.rn1 = div_factor((unsigned)L.n1, L.ncell);
}

// Index of cell (i0, i1, i2) (flat index i) in the per-cell parameter arrays
// g, psi0, p1, p2, smax of a level.  Natural layout: i.  Colour-split layout
// (big FP32 levels with an even n0): the cells of each colour packed row by
// row, (i0 >> 1) + n0/2 (i1 + n1 i2), the black half after the red one, so a
// half-sweep reads only its own colour's sectors of these arrays.  u, Kc and
// d keep the natural layout (the stencil reads both colours of them).
__host__ __device__ __forceinline__ unsigned pix_of(int cs, int n0, int n1, int n2, unsigned i, int i0, int i1,
                                                    int i2) {
  if (!cs) return i;
  const unsigned nh = (unsigned)n0 >> 1;
  const unsigned q = (unsigned)(i0 >> 1) + nh * ((unsigned)i1 + (unsigned)n1 * (unsigned)i2);
  return ((i0 + i1 + i2) & 1) ? q + nh * (unsigned)n1 * (unsigned)n2 : q;
}
template <typename T>
__device__ __forceinline__ unsigned pix(const Level<T>& L, long long i, int i0, int i1, int i2) {
  return pix_of(L.cs, L.n0, L.n1, L.n2, (unsigned)i, i0, i1, i2);
}

// One material of a layered soil: its law and the parameters that are not
// per-cell arrays (p1 and p2 are: the level's p1/p2 hold each cell's
// material values on every level).
template <typename T>
struct MatLaw {
  int model;
  T ts, tr, p3, p4;
};
template <>
struct MatLaw<double> {
  int model;
  double ts, tr, p3, p4;
  fl::Prep q;                    // the law's powers, prepared (Gardner: n = 1, alpha = 1)
};

struct DDMat;                    // float-float copy of a MatLaw (ddmath.cuh)

template <typename T>
struct UniformLaw {};
template <>
struct UniformLaw<double> {
  fl::Prep q;                    // a uniform soil's powers, prepared
};

template <typename T>
struct Phys : UniformLaw<T> {
  T a, xi, kappa;
  T ts, tr;                      // theta_s, theta_r
  T p1, p2, p3, p4;              // scalar soil parameters
  T h1, h2, h3, h4;              // sink thresholds
  int newton_k;                  // > 0: fixed steps; 0: to round-off
  int sink;
  int lag;                       // BDF2: 1 lags K and the xi term at psi^n, 0 at 2 psi^n - psi^(n-1)
  T r12, r34;                    // 1/(h1 - h2), 1/(h3 - h4)
  const MatLaw<T> *mats;         // COMPOSITE: material table (device, MAXMAT entries at most)
  const DDMat *ddmats;           // COMPOSITE, float-float outer layer: the same table as pairs
};

template <int M>
using LawTag = std::integral_constant<int, M>;

// a law's powers prepared on the host (fixlaw.cuh)
inline fl::Prep law_prep(int model, double p1, double p2) {
  return model == GARDNER ? fl::host_prep(false, 1.0, 1.0) : fl::host_prep(model == VANGENUCHTEN, p1, p2);
}
// the sink's slopes
template <typename T>
__host__ __device__ __forceinline__ void set_sink_slopes(Phys<T>& P) {
  P.r12 = P.h1 != P.h2 ? T(1) / (P.h1 - P.h2) : T(0);
  P.r34 = P.h3 != P.h4 ? T(1) / (P.h3 - P.h4) : T(0);
}

// Calls fn(LawTag<law>{}, phys) with the law of a cell and the physics
// record that carries its theta_s, theta_r, p3, p4: MODEL and P themselves,
// or, for a layered soil (MODEL == COMPOSITE), the law and parameters of
// material m.  Cells of one warp with different laws take the branches in turn.
template <int MODEL, typename T, typename Fn>
__device__ __forceinline__ auto with_law(const Phys<T>& P, unsigned m, Fn&& fn) {
  if constexpr (MODEL == COMPOSITE) {
    const MatLaw<T>* __restrict__ M = P.mats + m;
    Phys<T> Q = P;
    Q.ts = M->ts;
    Q.tr = M->tr;
    Q.p3 = M->p3;
    Q.p4 = M->p4;
    const int law = M->model;
    if (law == HAVERKAMP) return fn(LawTag<HAVERKAMP>{}, (const Phys<T>&)Q);
    if (law == GARDNER) return fn(LawTag<GARDNER>{}, (const Phys<T>&)Q);
    return fn(LawTag<VANGENUCHTEN>{}, (const Phys<T>&)Q);
  } else {
    return fn(LawTag<MODEL>{}, P);
  }
}

// material index of cell i (0, and no load, when the soil is not layered)
template <int MODEL>
__device__ __forceinline__ unsigned mat_at(const uint8_t* __restrict__ mat, long long i) {
  if constexpr (MODEL == COMPOSITE) return mat[i];
  else return 0u;
}
template <int MODEL, typename T>
__device__ __forceinline__ unsigned mat_of(const Level<T>& L, long long i) {
  return mat_at<MODEL>(L.mat, i);
}

template <typename T>
struct Xfer {                    // fine level -> next coarser level
  const int *pc[3];              // fine i: number of coarse contributors (1 or 2)
  const int *pj[3];              // fine i: coarse indices [2 i + k]
  const T *pw[3];                // fine i: weights [2 i + k]
  const int *rc[3];              // coarse J: number of fine contributors
  const int *ri[3];              // coarse J: fine indices [RMAX J + k]
  const T *rw[3];                // coarse J: normalised weights
};

// ---------------------------------------------------------------------------
// Constitutive laws (Table 1 of the paper); psi >= 0 gives theta_s, Ks and a
// zero capacity for all three laws.
// ---------------------------------------------------------------------------
// FP64 heads: the powers of a law run in 64-bit fixed point (fixlaw.cuh);
// arguments outside its ranges take the FP64 functions (slow_*: not inlined,
// they are all but never reached and would double every kernel's code).
__device__ __forceinline__ double vg_m(double n) { return 1.0 - 1.0 / n; }

template <int MODEL>
__device__ __noinline__ double slow_se(double h, double p1, double p2) {
  if (MODEL == HAVERKAMP) return p1 / (p1 + fx::exp(p2 * fx::log(h)));
  if (MODEL == GARDNER) return fx::exp(-(p1 * h));
  return fx::exp(-vg_m(p2) * fx::log1p(fx::exp(p2 * fx::log(p1 * h))));
}

// Se and d Se/d psi without its factor (Haverkamp beta, Gardner alpha, van
// Genuchten n - 1)
template <int MODEL>
__device__ __noinline__ double2 slow_se_slope(double h, double p1, double p2) {
  if (MODEL == HAVERKAMP) {
    const double u = fx::exp(p2 * fx::log(h));
    const double den = p1 + u;
    return make_double2(p1 / den, p1 * (u / h) / (den * den));
  }
  if (MODEL == GARDNER) {
    const double e = fx::exp(-(p1 * h));
    return make_double2(e, e);
  }
  const double t = fx::exp(p2 * fx::log(p1 * h));
  const double Se = fx::exp(-vg_m(p2) * fx::log1p(t));
  return make_double2(Se, (t / h) * Se / (1.0 + t));
}

// K/Ks.  For van Genuchten-Mualem, Se^{1/m} = 1/(1+t), so 1 - (1 - Se^{1/m})^m
// = -expm1(m log(t/(1+t))), evaluated without cancellation in both the wet
// (t < 1) and the dry (t > 1) range.  With lt = log t and e = exp(-|lt|):
//   log(1 + t)       = log1p(e) + max(lt, 0),
//   log(t / (1 + t)) = min(lt, 0) - log1p(e).
template <int MODEL>
__device__ __noinline__ double slow_kr(double h, double p1, double p2, double p3, double p4) {
  if (MODEL == HAVERKAMP) return p3 / (p3 + fx::exp(p4 * fx::log(h)));
  if (MODEL == GARDNER) return fx::exp(-(p1 * h));
  const double m = vg_m(p2), lt = p2 * fx::log(p1 * h);
  const double l1 = fx::log1p(fx::exp(-fabs(lt)));
  const double inner = -fx::expm1(m * (fmin(lt, 0.0) - l1));
  return fx::exp(-p3 * m * (l1 + fmax(lt, 0.0))) * inner * inner;
}

// psi < 0 from its bits (false for +-0 and NaN)
__device__ __forceinline__ bool unsaturated(double psi) {
  const unsigned long long b = fl::dbits(psi);
  return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull;
}

// A cell's law with its parameters prepared once per point solve (uniform
// soils: once per launch, P.q; layered soils: once per material).
template <int MODEL>
struct LawCell {
  fl::Prep q;
  double p1, p2, ds, cs;      // cs: the factor of d theta/d psi (ds beta, ds alpha, ds (n - 1))
  // uniform: P.q is this cell's
  __device__ __forceinline__ LawCell(double a, double b, bool uniform, const Phys<double>& P)
      : p1(a), p2(b), ds(P.ts - P.tr) {
    if (MODEL != GARDNER) {
      if (uniform) q = P.q;
      else q = fl::prep<MODEL == VANGENUCHTEN>(a, b);
    }
    cs = ds * (MODEL == GARDNER ? a : (MODEL == HAVERKAMP ? b : b - 1.0));
  }
  // theta(psi) and theta'(psi)
  __device__ __forceinline__ void eval(double psi, const Phys<double>& P, double& th, double& dth) const {
    if (!unsaturated(psi)) { th = P.ts; dth = 0.0; return; }
    const unsigned long long hb = fl::dbits(psi) ^ 0x8000000000000000ull;
    double Se, s;
    bool ok = true;
    if (MODEL == GARDNER) {
      Se = s = fl::exp_gardner(p1, hb, ok);
    } else {
      ok = q.ok;
      fl::se_slope<MODEL == VANGENUCHTEN>(q, hb, ok, Se, s);
    }
    if (!ok) {
      const double2 v = slow_se_slope<MODEL>(-psi, p1, p2);
      Se = v.x;
      s = v.y;
    }
    th = P.tr + ds * Se;
    dth = cs * s;
  }
};

// (the increment form prepares nothing here)
template <>
struct LawCell<-1> {};

static __device__ __noinline__ double2 slow_se_any(int law, double h, double p1, double p2) {
  if (law == HAVERKAMP) return slow_se_slope<HAVERKAMP>(h, p1, p2);
  if (law == GARDNER) return slow_se_slope<GARDNER>(h, p1, p2);
  return slow_se_slope<VANGENUCHTEN>(h, p1, p2);
}

// Layered soils: every lane its own material's law, in one instruction stream.
template <>
struct LawCell<COMPOSITE> {
  fl::Prep q;
  int law;
  double p1, p2, ds, cs;
  __device__ __forceinline__ LawCell(double a, double b, unsigned m, const Phys<double>& P)
      : p1(a), p2(b), ds(P.ts - P.tr) {
    q = P.mats[m].q;
    law = P.mats[m].model;
    cs = ds * (law == GARDNER ? a : (law == HAVERKAMP ? b : b - 1.0));
  }
  template <bool SLOPE>
  __device__ __forceinline__ void any(double psi, const Phys<double>& P, double& th, double& dth) const {
    static_assert(HAVERKAMP == fl::ANY_HAVERKAMP && GARDNER == fl::ANY_GARDNER && VANGENUCHTEN == fl::ANY_VANGENUCHTEN,
                  "law numbers");
    if (!unsaturated(psi)) { th = P.ts; dth = 0.0; return; }
    const unsigned long long hb = fl::dbits(psi) ^ 0x8000000000000000ull;
    bool ok = q.ok;
    double Se, s = 0.0;
    fl::se_any<SLOPE>(law, q, p1, hb, ok, Se, s);
    if (!ok) {
      const double2 v = slow_se_any(law, -psi, p1, p2);
      Se = v.x;
      s = v.y;
    }
    th = P.tr + ds * Se;
    if (SLOPE) dth = cs * s;
  }
  __device__ __forceinline__ void eval(double psi, const Phys<double>& P, double& th, double& dth) const {
    any<true>(psi, P, th, dth);
  }
};

template <int MODEL>
__device__ __forceinline__ double theta_only_d(double psi, double p1, double p2, const Phys<double>& P) {
  if (!unsaturated(psi)) return P.ts;
  const unsigned long long hb = fl::dbits(psi) ^ 0x8000000000000000ull;
  bool ok = true;
  double Se = MODEL == GARDNER ? fl::exp_gardner(p1, hb, ok) : fl::se_only<MODEL == VANGENUCHTEN>(p1, p2, hb, ok);
  if (!ok) Se = slow_se<MODEL>(-psi, p1, p2);
  return P.tr + (P.ts - P.tr) * Se;
}

// theta at psi of a cell of a level (m: its material; uniform: no per-cell p1, p2)
template <int MODEL>
__device__ __forceinline__ double theta_cell(double psi, double p1, double p2, unsigned m, bool uniform,
                                             const Phys<double>& P) {
  if constexpr (MODEL == COMPOSITE) {
    double th, dth;
    Phys<double> Q = P;
    Q.ts = P.mats[m].ts;
    Q.tr = P.mats[m].tr;
    LawCell<COMPOSITE>(p1, p2, m, Q).any<false>(psi, Q, th, dth);
    return th;
  } else {
    if (MODEL == GARDNER || !uniform) return theta_only_d<MODEL>(psi, p1, p2, P);
    if (!unsaturated(psi)) return P.ts;
    const unsigned long long hb = fl::dbits(psi) ^ 0x8000000000000000ull;
    bool ok = P.q.ok;
    double Se = fl::se_prepared<MODEL == VANGENUCHTEN>(P.q, hb, ok);
    if (!ok) Se = slow_se<MODEL>(-psi, p1, p2);
    return P.tr + (P.ts - P.tr) * Se;
  }
}

// Hydraulic conductivity.
template <int MODEL>
__device__ __forceinline__ double cond_d(double psi, double p1, double p2, double Ks, const Phys<double>& P) {
  if (!unsaturated(psi)) return Ks;
  const unsigned long long hb = fl::dbits(psi) ^ 0x8000000000000000ull;
  bool ok = true;
  double Kr = MODEL == HAVERKAMP ? fl::kr_haverkamp(P.p3, P.p4, hb, ok)
              : MODEL == GARDNER ? fl::exp_gardner(p1, hb, ok)
                                 : fl::kr_vangenuchten(p1, p2, P.p3, hb, ok);
  if (!ok) Kr = slow_kr<MODEL>(-psi, p1, p2, P.p3, P.p4);
  return Ks * Kr;
}

// ---------------------------------------------------------------------------
// Increment form in FP32 for the inner correction problem: Dth =
// theta(psi0 + x) - theta(psi0) and dth = theta'(psi0 + x), the differences
// through expm1/log1p of the ratio (psi0 + x)/psi0, so that Dth is accurate
// relative to itself.  The inner FP32 solve only has to be accurate to ~1e-5
// relative (the outer defect correction removes the rest), but the increments
// must stay free of cancellation: log1p and expm1 of small arguments come
// from their Taylor series (truncation below 1e-10 relative for |x| < 1/32),
// larger arguments use the hardware approximations (relative error ~1e-6 of
// a result that is then not small).
//
// The hardware's 1/x, log2 and 2^x are taken in their flush-to-zero forms:
// the plain __fdividef, __logf, __expf wrap each in three to five
// instructions that rescale subnormal operands, and a point update takes 16 of
// them.  A power of psi0 + x below 2^-126 adds nothing to 1 + t; one of psi0
// is a factor that the increment multiplies by up to e^80, so dbase() keeps
// it: heads whose power is flushed count as saturated, where the increment
// comes from psi0 + x alone, and Gardner's e^(alpha psi0) takes the plain form.
// Reciprocals of per-cell values (1/(1 + t0)) are taken once per update.
// The point update is bound by instruction issue on big levels and by its own
// instruction chain (~6 cycles per instruction of a lone warp) on small ones.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float rcp_a(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float log_a(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r * 0.69314718f;
}
__device__ __forceinline__ float exp_a(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x * 1.44269504f));
  return r;
}

// (both forms are evaluated and one is selected: no branch, so lanes of a
// warp on either side of 1/32 do not split it into two passes)
__device__ __forceinline__ float fast_log1p(float x) {
  // x - x^2/2 + x^3/3 - x^4/4 + x^5/5 - x^6/6
  const float p = fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, -1.0f / 6.0f, 0.2f), -0.25f), 1.0f / 3.0f), -0.5f), 1.0f);
  const float big = log_a(1.0f + x);
  return fabsf(x) < 0.03125f ? x * p : big;
}

__device__ __forceinline__ float fast_expm1(float x) {
  // x + x^2/2 + x^3/6 + x^4/24 + x^5/120 + x^6/720
  const float p = fmaf(x, fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.0f / 720.0f, 1.0f / 120.0f), 1.0f / 24.0f),
                                           1.0f / 6.0f), 0.5f), 1.0f);
  const float big = exp_a(x) - 1.0f;
  return fabsf(x) < 0.03125f ? x * p : big;
}

// The increment law split into the part that depends on psi0 only (once per
// point update) and the part that depends on the correction x (once per
// Newton step).
struct DBase {
  float psi0, inv_psi0;
  bool wet0;
  float a0, b0, c0;      // VG: t0, log1p(t0), Se0; Haverkamp: u0, log(u0); Gardner: e0
  float r0;              // VG: 1/(1 + t0); Haverkamp: 1/(alpha + u0)
  float m;               // VG: 1 - 1/n
};

// Largest exponent a power t = (alpha h)^n or u = h^beta of a trial state may
// reach (e^80 ~ 5.5e34, below FLT_MAX with room for 1 + t and products).  A
// bracketed point solve on a coarse level with a tiny coupling can probe
// heads of -1e6 m and beyond, where the power would overflow and its ratios
// turn into inf/inf; there theta = theta_r and theta' = 0 to far below FP32
// resolution either way, so capping the exponent changes nothing else.
constexpr float POW_EXP_MAX = 80.0f;
constexpr float POW_EXP_MIN = -87.0f;          // (2^-126 = e^-87.34)
// 2^-126: what is below it has no reciprocal here.  Heads nearer to
// saturation count as saturated, a smaller coupling as none.
constexpr float NORMAL_MIN = 1.17549435e-38f;

template <int MODEL>
__device__ __forceinline__ DBase dbase(float psi0, float p1, float p2) {
  DBase B;
  B.psi0 = psi0;
  B.a0 = B.b0 = B.c0 = B.r0 = 0.0f;
  B.m = MODEL == VANGENUCHTEN ? 1.0f - rcp_a(p2) : 0.0f;
  float lp = 0.0f;               // log of the power of h0 (no number, or -inf, from saturation on)
  if (MODEL == GARDNER) {
    B.wet0 = !(psi0 <= -NORMAL_MIN);
  } else {
    lp = p2 * log_a(MODEL == HAVERKAMP ? -psi0 : p1 * -psi0);
    // a power that would be flushed: theta(psi0) is theta_s to below 2^-125
    B.wet0 = !(lp >= POW_EXP_MIN);
  }
  B.inv_psi0 = B.wet0 ? 0.0f : rcp_a(psi0);
  if (!B.wet0) {
    if (MODEL == GARDNER) {
      B.a0 = __expf(p1 * psi0);
    } else if (MODEL == HAVERKAMP) {
      const float lu = fminf(lp, POW_EXP_MAX);   // h0^beta
      B.a0 = exp_a(lu);
      B.b0 = lu;
      B.r0 = rcp_a(p1 + B.a0);
    } else {
      const float m = B.m;
      B.a0 = exp_a(fminf(lp, POW_EXP_MAX));   // (alpha h0)^n
      B.b0 = fast_log1p(B.a0);
      B.c0 = exp_a(-m * B.b0);
      B.r0 = rcp_a(1.0f + B.a0);
    }
  }
  return B;
}

template <int MODEL>
__device__ __forceinline__ void dincr(const DBase& B, float x, float p1, float p2, const Phys<float>& P,
                                      float& Dth, float& dth) {
  const float ds = P.ts - P.tr;
  const float psi1 = B.psi0 + x;
  const bool wet1 = !(psi1 <= -NORMAL_MIN);
  if (MODEL == GARDNER) {
    const float al = p1;
    if (!B.wet0) {
      const float e0 = B.a0;
      if (!wet1) {
        const float em = fast_expm1(al * x);
        Dth = ds * e0 * em;
        dth = al * ds * e0 * (1.0f + em);
      } else {
        Dth = -ds * fast_expm1(al * B.psi0);
        dth = 0.0f;
      }
    } else if (!wet1) {
      Dth = ds * fast_expm1(al * psi1);
      dth = al * ds * exp_a(al * psi1);
    } else {
      Dth = 0.0f; dth = 0.0f;
    }
  } else if (MODEL == HAVERKAMP) {
    const float al = p1, be = p2;
    if (!B.wet0) {
      const float u0 = B.a0;
      if (!wet1) {
        // (u1 = u0 (psi1/psi0)^beta, its exponent capped as in dbase)
        // (psi1/psi0 > 0 here; its rounded value is kept above 2^-24)
        const float q = fmaxf(x * B.inv_psi0, -0.99999994f);
        const float du = u0 * fast_expm1(fminf(be * fast_log1p(q), POW_EXP_MAX - B.b0));
        const float u1 = u0 + du;
        const float r1 = rcp_a(al + u1);
        Dth = -al * ds * (du * B.r0) * r1;
        dth = al * ds * be * (u1 * r1) * (r1 * rcp_a(-psi1));
      } else {
        Dth = ds * u0 * B.r0;
        dth = 0.0f;
      }
    } else if (!wet1) {
      const float h1 = -psi1;
      const float u1 = exp_a(fminf(be * log_a(h1), POW_EXP_MAX));
      const float r1 = rcp_a(al + u1);
      Dth = -ds * u1 * r1;
      dth = al * ds * be * (u1 * r1) * (r1 * rcp_a(h1));
    } else {
      Dth = 0.0f; dth = 0.0f;
    }
  } else {
    const float al = p1, n = p2, m = B.m;
    if (!B.wet0) {
      const float t0 = B.a0, L0 = B.b0, Se0 = B.c0;
      if (!wet1) {
        // (t1 = t0 (psi1/psi0)^n, its exponent capped as in dbase)
        const float q = fmaxf(x * B.inv_psi0, -0.99999994f);     // (as for Haverkamp)
        const float dt = t0 * fast_expm1(fminf(n * fast_log1p(q), POW_EXP_MAX - B.b0));
        const float t1 = t0 + dt;
        const float dSe = Se0 * fast_expm1(-m * fast_log1p(dt * B.r0));
        const float Se1 = Se0 + dSe;
        Dth = ds * dSe;
        dth = ds * m * n * (t1 * rcp_a(-psi1)) * (Se1 * rcp_a(1.0f + t1));
      } else {
        Dth = -ds * fast_expm1(-m * L0);
        dth = 0.0f;
      }
    } else if (!wet1) {
      const float h1 = -psi1;
      const float t1 = exp_a(fminf(n * log_a(al * h1), POW_EXP_MAX));
      const float L1 = fast_log1p(t1);
      Dth = ds * fast_expm1(-m * L1);
      dth = ds * m * n * (t1 * rcp_a(h1)) * (exp_a(-m * L1) * rcp_a(1.0f + t1));
    } else {
      Dth = 0.0f; dth = 0.0f;
    }
  }
}

template <int MODEL>
__device__ __forceinline__ void dlaw_fast(float psi0, float x, float p1, float p2, const Phys<float>& P,
                                          float& Dth, float& dth) {
  dincr<MODEL>(dbase<MODEL>(psi0, p1, p2), x, p1, p2, P, Dth, dth);
}

// ---------------------------------------------------------------------------
// Sink reading: S = smax * alpha_F(psi), alpha_F piecewise linear through
// (h4,0), (h3,1), (h2,1), (h1,0), zero outside; right derivatives at kinks.
// ---------------------------------------------------------------------------
// The ramps' quotients: x r with r the rounded reciprocal of the ramp's
// width, corrected once by its remainder (Markstein, IBM J. Res. Dev. 34,
// 1990: correctly rounded), two multiply-adds instead of a division.
template <typename T>
__device__ __forceinline__ T ramp(T x, T width, T r) {
  const T q = x * r;
  return fma(fma(-q, width, x), r, q);
}
// the piece that psi lies on (0 at the wet end to 4 at the dry one) and its slope
template <typename T>
__device__ __forceinline__ int feddes_piece(T psi, const Phys<T>& P, T& da) {
  da = T(0);
  if (psi >= P.h1) return 0;
  if (psi < P.h4) return 4;
  if (psi >= P.h2) { da = -P.r12; return 1; }
  if (psi >= P.h3) return 2;
  da = P.r34;
  return 3;
}
// alpha_F(psi1) - alpha_F(psi0), on pieces k1 and k0.  A correction seldom
// crosses a kink, so point updates make it a call (by value: a reference would
// put the physics in memory): inlined, the two ramps at every update cost the
// served mix 6% (8 requests 8.66 -> 9.16 ms) and the defect-writing half-sweep
// of 256^3 6% (125 -> 132 us).  Defects alone, which evaluate it once, take it
// inline: there the call cost the 256^3 one-colour defect 15% (97 -> 112 us).
__device__ __forceinline__ float feddes_jump(float psi0, int k0, float psi1, int k1, float h1, float h2, float h3,
                                             float h4, float r12, float r34) {
  auto value = [=](float psi, int k) {
    if (k == 1) return ramp(h1 - psi, h1 - h2, r12);
    if (k == 3) return ramp(psi - h4, h3 - h4, r34);
    return k == 2 ? 1.0f : 0.0f;
  };
  return value(psi1, k1) - value(psi0, k0);
}
static __device__ __noinline__ float feddes_jump_call(float psi0, int k0, float psi1, int k1, float h1, float h2,
                                                      float h3, float h4, float r12, float r34) {
  return feddes_jump(psi0, k0, psi1, k1, h1, h2, h3, h4, r12, r34);
}

// alpha_F in FP64 on piece k: one ramp, its operands selected (with both
// inline, their FP64 operations issued in every update, with or without a
// sink).  CALL: where the physics are known to have a sink only at run time,
// the ramp is a call: inline, the 257^2 FP64 strip's steps took 1.3% longer;
// as a call where it is known, the 777-cell layered column's did.
__device__ __forceinline__ double feddes_ramp(double psi, int k, double h1, double h2, double h3, double h4,
                                              double r12, double r34) {
  const bool wet = k == 1;
  return ramp(wet ? h1 - psi : psi - h4, wet ? h1 - h2 : h3 - h4, wet ? r12 : r34);
}
static __device__ __noinline__ double feddes_ramp_call(double psi, int k, double h1, double h2, double h3, double h4,
                                                       double r12, double r34) {
  return feddes_ramp(psi, k, h1, h2, h3, h4, r12, r34);
}
template <bool CALL>
__device__ __forceinline__ void sink_direct(double psi, double smax, const Phys<double>& P, double& S, double& dS) {
  double a = 0.0, da = 0.0;
  if (P.sink && smax > 0.0) {
    const int k = feddes_piece(psi, P, da);
    a = k == 2 ? 1.0 : 0.0;
    if (k & 1)
      a = CALL ? feddes_ramp_call(psi, k, P.h1, P.h2, P.h3, P.h4, P.r12, P.r34)
               : feddes_ramp(psi, k, P.h1, P.h2, P.h3, P.h4, P.r12, P.r34);
  }
  S = a * smax;
  dS = da * smax;
}
// S at psi, for a defect: one evaluation a cell, all of it a call (in the point
// solve that cost a 2000-cell column with root uptake 35.2 ms a step instead of
// 31.7; 32.7 with plain products inline)
static __device__ __noinline__ double feddes_alpha(double psi, double h1, double h2, double h3, double h4, double r12,
                                                   double r34) {
  Phys<double> P;
  P.h1 = h1; P.h2 = h2; P.h3 = h3; P.h4 = h4;
  P.r12 = r12; P.r34 = r34;
  double da;
  const int k = feddes_piece(psi, P, da);
  return k & 1 ? feddes_ramp(psi, k, h1, h2, h3, h4, r12, r34) : (k == 2 ? 1.0 : 0.0);
}
__device__ __forceinline__ double sink_value(double psi, double smax, const Phys<double>& P) {
  return P.sink && smax > 0.0 ? smax * feddes_alpha(psi, P.h1, P.h2, P.h3, P.h4, P.r12, P.r34) : 0.0;
}

// S(psi0 + x) - S(psi0), psi0 on piece k0: exact slope * x on a common linear
// piece.  CALL: the crossing of a kink as a call.
template <bool CALL>
__device__ __forceinline__ void sink_delta(float psi0, int k0, float x, float smax, const Phys<float>& P, float& DS,
                                           float& dS) {
  float da;
  const int k1 = feddes_piece(psi0 + x, P, da);
  DS = smax * da * x;
  if (k1 != k0) {
    const float j = CALL ? feddes_jump_call(psi0, k0, psi0 + x, k1, P.h1, P.h2, P.h3, P.h4, P.r12, P.r34)
                         : feddes_jump(psi0, k0, psi0 + x, k1, P.h1, P.h2, P.h3, P.h4, P.r12, P.r34);
    DS = smax * j;
  }
  dS = smax * da;
}

// ---------------------------------------------------------------------------
// Stencil: m_ii and sum_j m_ij u_j for cell i (interior faces K_f/h^2 with
// K_f = (Kc_i + Kc_j)/2; Dirichlet faces 2 kb/h^2 on the diagonal).
// ---------------------------------------------------------------------------
// (YZI: the caller knows that the cell of a 3-d level is interior along axes
// 1 and 2, so only axis 0 is tested for boundary faces)
template <typename T, bool YZI = false>
__device__ __forceinline__ void stencil(const Level<T>& L, long long i, int i0, int i1, int i2,
                                        const T* __restrict__ u, T& mii, T& off) {
  // neighbours through base pointers and 32-bit strides (levels hold fewer
  // than 2^31 cells)
  const T* __restrict__ Kp = L.Kc + i;
  const T* __restrict__ up = u + i;
  const T Ki = Kp[0];
  T dg = T(0), of = T(0);
  // K_f / h^2 = (Kc_i + Kc_j) * (s/2): halving s is exact, so this equals
  // ((Kc_i + Kc_j) / 2) * s bit for bit
  {
    const T s = L.ih2[0], hs = T(0.5) * s;
    if (i0 > 0) { const T m = (Ki + Kp[-1]) * hs; dg += m; of += m * up[-1]; }
    else dg += T(2) * L.kb[0][i1 + L.n1 * i2] * s;
    if (i0 < L.n0 - 1) { const T m = (Ki + Kp[1]) * hs; dg += m; of += m * up[1]; }
    else dg += T(2) * L.kb[1][i1 + L.n1 * i2] * s;
  }
  if (YZI) {
    {
      const T s = L.ih2[1], hs = T(0.5) * s;
      const int st = L.n0;
      { const T m = (Ki + Kp[-st]) * hs; dg += m; of += m * up[-st]; }
      { const T m = (Ki + Kp[st]) * hs; dg += m; of += m * up[st]; }
    }
    {
      const T s = L.ih2[2], hs = T(0.5) * s;
      const int st = L.n0 * L.n1;
      { const T m = (Ki + Kp[-st]) * hs; dg += m; of += m * up[-st]; }
      { const T m = (Ki + Kp[st]) * hs; dg += m; of += m * up[st]; }
    }
    mii = dg;
    off = of;
    return;
  }
  if (L.dim > 1) {
    const T s = L.ih2[1], hs = T(0.5) * s;
    const int st = L.n0;
    if (i1 > 0) { const T m = (Ki + Kp[-st]) * hs; dg += m; of += m * up[-st]; }
    else dg += T(2) * L.kb[2][i0 + L.n0 * i2] * s;
    if (i1 < L.n1 - 1) { const T m = (Ki + Kp[st]) * hs; dg += m; of += m * up[st]; }
    else dg += T(2) * L.kb[3][i0 + L.n0 * i2] * s;
  }
  if (L.dim > 2) {
    const T s = L.ih2[2], hs = T(0.5) * s;
    const int st = L.n0 * L.n1;
    if (i2 > 0) { const T m = (Ki + Kp[-st]) * hs; dg += m; of += m * up[-st]; }
    else dg += T(2) * L.kb[4][i0 + L.n0 * i1] * s;
    if (i2 < L.n2 - 1) { const T m = (Ki + Kp[st]) * hs; dg += m; of += m * up[st]; }
    else dg += T(2) * L.kb[5][i0 + L.n0 * i1] * s;
  }
  mii = dg;
  off = of;
}

template <typename T>
__device__ __forceinline__ T tol_of();
template <>
__device__ __forceinline__ double tol_of<double>() { return 1e-15; }
template <>
__device__ __forceinline__ float tol_of<float>() { return 1e-7f; }

// Storage + sink part at x (the defect's part of N) of cell q of a level, of
// material m.  CALL: as for sink_delta.
template <typename T, int FORM, int MODEL, bool CALL = false>
__device__ __forceinline__ T storage(const Level<T>& L, T x, T psi0, T p1, T p2, T smax, unsigned m,
                                     const Phys<T>& P) {
  if constexpr (FORM == FORM_DIRECT) {
    static_assert(sizeof(T) == 8, "direct form is FP64");
    return P.a * theta_cell<MODEL>(x, p1, p2, m, !L.p1 && !L.p2, P) + sink_value(x, smax, P);
  } else {
    static_assert(sizeof(T) == 4, "increment form is FP32");
    return with_law<MODEL>(P, m, [&](auto law, const Phys<T>& Q) {
      float Dth, dth, DS = 0.0f, dS, da0;
      dlaw_fast<decltype(law)::value>(psi0, x, p1, p2, Q, Dth, dth);
      if (Q.sink && smax > 0.0f) sink_delta<CALL>(psi0, feddes_piece(psi0, Q, da0), x, smax, Q, DS, dS);
      return Q.a * Dth + DS;
    });
  }
}

// Scalar solve of  storage(x) + cc x = f  (eq. point-update).  The left side
// increases strictly (cc > 0), the root lies in [lo, hi]; Newton from x0,
// bisection whenever a step leaves the current bracket.
// NK > 0: exactly NK steps fixed at compile time (must equal P.newton_k);
// NK = 0: P.newton_k steps (0: to round-off).
// FP32 increment form with a fixed step count: a solve does not end on a
// bisection.  Where the coupling is tiny (dry cells of a steep law on a
// coarse level) the bracket spans millions of metres and its midpoint is no
// estimate of the root; after a bisection up to BISECT_EXTRA further steps
// run until one is a Newton step inside the bracket.  Solves that never
// bisect take exactly the fixed count, as before.
constexpr int BISECT_EXTRA = 12;

// Comparisons of the point solve.  FP64: on the bits, with integers
// (fixlaw.cuh); an operand that is not a number only has to keep the result
// one (clamp_to leaves it; a bracket test that fails bisects NaN ends).
__device__ __forceinline__ bool less(float a, float b) { return a < b; }
__device__ __forceinline__ bool less(double a, double b) { return fl::order_key(a) < fl::order_key(b); }
__device__ __forceinline__ bool at_most(float a, float b) { return a <= b; }
__device__ __forceinline__ bool at_most(double a, double b) { return !less(b, a); }   // (false for a NaN |a|)
__device__ __forceinline__ bool is_zero(float a) { return a == 0.0f; }
__device__ __forceinline__ bool is_zero(double a) { return (fl::dbits(a) << 1) == 0; }
__device__ __forceinline__ bool above_zero(float a) { return a > 0.0f; }
__device__ __forceinline__ bool above_zero(double a) { return (long long)fl::dbits(a) > 0 && !fl::is_nan(a); }
// a coupling that can be divided by
__device__ __forceinline__ bool couples(float a) { return a >= NORMAL_MIN; }
__device__ __forceinline__ bool couples(double a) { return above_zero(a); }
__device__ __forceinline__ float clamp_to(float x, float lo, float hi) { return x < lo ? lo : (x > hi ? hi : x); }
__device__ __forceinline__ double clamp_to(double x, double lo, double hi) {
  if (fl::is_nan(x) || fl::is_nan(lo) || fl::is_nan(hi)) return x;
  return less(x, lo) ? lo : (less(hi, x) ? hi : x);
}

// SINK: 1 / 0 the physics have a sink / none, -1 as P.sink says.
template <typename T, int FORM, int MODEL, int NK = 0, int SINK = -1>
__device__ __forceinline__ T point_solve(T cc, T f, T x0, T psi0, T p1, T p2, T smax, const Phys<T>& P,
                                         const LawCell<FORM == FORM_DIRECT ? MODEL : -1>& law) {
  if (!couples(cc)) {
    // no coupling and no shift (c = 0): shift kappa (x - x0), kappa = 1e-6 a,
    // which keeps the root and provides the bracket
    const T k = T(1e-6) * P.a;
    f += (k - cc) * x0;
    cc = k;
  }
  const bool has_sink = SINK != 0 && (SINK == 1 || P.sink) && smax > T(0);
  const T ds = P.ts - P.tr;
  T lo, hi;
  if constexpr (FORM == FORM_DIRECT) {
    const fl::Divisor dc = fl::divisor(cc);
    lo = fl::div(f - P.a * P.ts - smax, dc);
    hi = fl::div(f - P.a * P.tr, dc);
  } else {
    // FP32: both ends through one approximate reciprocal; each end has a
    // slack of (a ds + smax)/cc beyond the root, far above its 2^-22 error
    const T rc = rcp_a(cc);
    lo = (f - P.a * ds - smax) * rc;
    hi = (f + P.a * ds + smax) * rc;
  }
  T x = clamp_to(x0, lo, hi);
  const int maxit = NK > 0 ? NK : (P.newton_k > 0 ? P.newton_k : 200);
  DBase B;
  int sk0 = 0;
  if constexpr (FORM == FORM_DELTA) {
    B = dbase<MODEL>(psi0, p1, p2);
    T da0;
    if (has_sink) sk0 = feddes_piece(psi0, P, da0);
  }
  // one safeguarded step; returns true when the solve is done.  *bis: the
  // step was a bisection
  auto step = [&](bool* bis) -> bool {
    *bis = false;
    T val, der;
    if constexpr (FORM == FORM_DELTA) {
      float Dth, dth;
      dincr<MODEL>(B, x, p1, p2, P, Dth, dth);
      T DS = T(0), dS = T(0);
      if (has_sink) sink_delta<true>(psi0, sk0, x, smax, P, DS, dS);
      val = P.a * Dth + DS;
      der = P.a * dth + dS;
    } else {
      T th, dth, S, dS;
      law.eval(x, P, th, dth);
      S = dS = T(0);
      if (SINK != 0) sink_direct<(SINK < 0)>(x, smax, P, S, dS);
      val = P.a * th + S;
      der = P.a * dth + dS;
    }
    const T F = val + cc * x - f;
    const T dF = der + cc;
    if (is_zero(F)) return true;
    if (above_zero(F)) hi = x; else lo = x;
    T xn;
    if constexpr (sizeof(T) == 4) xn = x - F * rcp_a(dF);        // dF > 0; a 2-ulp step error is harmless
    else xn = x - fl::div(F, fl::divisor(dF));
    // a step strictly inside the bracket, or below round-off, is kept;
    // anything else (outside, or onto an end) is replaced by bisection
    auto below_roundoff = [&](T s) { return at_most(T(fabs(s)), tol_of<T>() * (less(T(1), fabs(x)) ? fabs(x) : T(1))); };
    if (!(less(lo, xn) && less(xn, hi)) && !below_roundoff(xn - x)) {
      xn = T(0.5) * (lo + hi);
      *bis = true;
    }
    const T stp = xn - x;
    const bool last = NK == 0 && P.newton_k <= 0 && below_roundoff(stp);
    x = xn;
    if (last) return true;
    // FP32 increment form: a step below 2^-20 of |x| leaves nothing for the
    // next one to change at this precision (quadratic convergence)
    if constexpr (FORM == FORM_DELTA) {
      if (fabsf(stp) <= 9.5367431640625e-7f * fabsf(x)) return true;
    }
    return false;
  };
  bool bis = false;
  if constexpr (NK > 0) {
    bool done = false;
#pragma unroll(NK)
    for (int it = 0; it < NK; ++it) {
      if (step(&bis)) { done = true; break; }
    }
    if (FORM == FORM_DELTA && !done) {
#pragma unroll 1
      for (int e = 0; e < BISECT_EXTRA && bis; ++e)
        if (step(&bis)) break;
    }
  } else {
    // one copy of the step (the cycles of small levels are bound by their
    // warps' instruction streams)
    int left = maxit, extra = FORM == FORM_DELTA && P.newton_k > 0 ? BISECT_EXTRA : 0;
#pragma unroll 1
    while (!step(&bis)) {
      if (--left > 0) continue;
      if (!bis || extra-- <= 0) break;
    }
  }
  return x;
}

// the point solve of a cell of material m: FP64 layered soils run it once
// with the lane's own law (LawCell<COMPOSITE>), FP32 ones law by law
template <typename T, int FORM, int MODEL, int NK = 0, int SINK = -1>
__device__ __forceinline__ T point_solve_of(const Level<T>& L, unsigned m, T cc, T f, T x0, T psi0, T p1, T p2, T smax,
                                            const Phys<T>& P) {
  if constexpr (FORM == FORM_DELTA) {
    return with_law<MODEL>(P, m, [&](auto law, const Phys<T>& Q) {
      return point_solve<T, FORM, decltype(law)::value, NK, SINK>(cc, f, x0, psi0, p1, p2, smax, Q, LawCell<-1>{});
    });
  } else if constexpr (MODEL == COMPOSITE) {
    Phys<T> Q = P;
    Q.ts = P.mats[m].ts;
    Q.tr = P.mats[m].tr;
    return point_solve<T, FORM, MODEL, NK, SINK>(cc, f, x0, psi0, p1, p2, smax, Q, LawCell<MODEL>(p1, p2, m, Q));
  } else {
    return point_solve<T, FORM, MODEL, NK, SINK>(cc, f, x0, psi0, p1, p2, smax, P,
                                                 LawCell<MODEL>(p1, p2, !L.p1 && !L.p2, P));
  }
}

template <typename T, int FORM, int MODEL, int NK = 0, int SINK = -1>
__device__ __forceinline__ void point_update(const Level<T>& L, const Phys<T>& P, long long i,
                                             int i0, int i1, int i2) {
  T mii, off;
  stencil(L, i, i0, i1, i2, L.u, mii, off);
  const T ui = L.u[i];
  const T cc = P.xi + P.kappa + mii;
  const unsigned q = pix(L, i, i0, i1, i2);
  const T f = L.g[q] + off + P.kappa * ui;
  const T p1 = L.p1 ? L.p1[q] : P.p1;
  const T p2 = L.p2 ? L.p2[q] : P.p2;
  const T smax = SINK != 0 && L.smax ? L.smax[q] : T(0);
  const T psi0 = FORM == FORM_DELTA ? L.psi0[q] : T(0);
  L.u[i] = point_solve_of<T, FORM, MODEL, NK, SINK>(L, mat_of<MODEL>(L, i), cc, f, ui, psi0, p1, p2, smax, P);
}

// Operands of one point update, gathered before any of them is used, so that
// a thread can issue the loads of its next cell before it solves the current
// one (the sweep is bound by load latency, not by bandwidth).  Face f =
// 2 axis + side; on a boundary face Kn holds the face conductance kb; on an
// axis the grid does not have, Kn = un = 0 and 1/h^2 = 0, so m_f = 0.
template <typename T>
struct CellOps {
  unsigned i;
  bool valid;
  unsigned bmask;                // bit f: face f lies on the boundary
  unsigned mat;                  // COMPOSITE: the cell's material
  T ui, Ki, g, psi0, p1, p2, smax;
  T Kn[6], un[6];
};

// YZI: the caller knows that the cell is interior along axes 1 and 2 of a
// 3-d level (no boundary face there), so only axis 0 is tested
template <typename T, int FORM, int MODEL, bool YZI = false>
__device__ __forceinline__ void gather(const Level<T>& L, const Phys<T>& P, int i0, int i1, int i2, CellOps<T>& c) {
  const unsigned i = (unsigned)(i0 + L.n0 * (i1 + L.n1 * i2));
  c.i = i;
  c.mat = mat_of<MODEL>(L, i);
  const T* __restrict__ Kp = L.Kc + i;
  const T* __restrict__ up = L.u + i;
  c.Ki = Kp[0];
  c.ui = up[0];
  const unsigned q = pix(L, i, i0, i1, i2);
  c.g = L.g[q];
  c.psi0 = FORM == FORM_DELTA ? L.psi0[q] : T(0);
  c.p1 = L.p1 ? L.p1[q] : P.p1;
  c.p2 = L.p2 ? L.p2[q] : P.p2;
  c.smax = L.smax ? L.smax[q] : T(0);
  unsigned bm = 0;
  const int ii[3] = {i0, i1, i2};
  const int nn[3] = {L.n0, L.n1, L.n2};
  const int st[3] = {1, L.n0, L.n0 * L.n1};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (YZI && a > 0) {
      c.Kn[2 * a] = Kp[-st[a]]; c.un[2 * a] = up[-st[a]];
      c.Kn[2 * a + 1] = Kp[st[a]]; c.un[2 * a + 1] = up[st[a]];
      continue;
    }
    const int fc = a == 0 ? i1 + L.n1 * i2 : (a == 1 ? i0 + L.n0 * i2 : i0 + L.n0 * i1);
    if (a >= L.dim) {
      c.Kn[2 * a] = c.Kn[2 * a + 1] = T(0);
      c.un[2 * a] = c.un[2 * a + 1] = T(0);
      continue;
    }
    if (ii[a] > 0) { c.Kn[2 * a] = Kp[-st[a]]; c.un[2 * a] = up[-st[a]]; }
    else { c.Kn[2 * a] = L.kb[2 * a][fc]; c.un[2 * a] = T(0); bm |= 1u << (2 * a); }
    if (ii[a] < nn[a] - 1) { c.Kn[2 * a + 1] = Kp[st[a]]; c.un[2 * a + 1] = up[st[a]]; }
    else { c.Kn[2 * a + 1] = L.kb[2 * a + 1][fc]; c.un[2 * a + 1] = T(0); bm |= 1u << (2 * a + 1); }
  }
  c.bmask = bm;
}

// the point update of a gathered cell (same sums, in the same order, as
// stencil() and point_update())
// m_ii (dg) and sum_j m_ij u_j (of) of a gathered cell: the sums of
// stencil(), in its order
template <typename T, bool YZI = false>
__device__ __forceinline__ void cell_sums(const Level<T>& L, const CellOps<T>& c, T& dg, T& of) {
  dg = T(0);
  of = T(0);
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    const T s = L.ih2[f >> 1];
    if ((!YZI || f < 2) && (c.bmask & (1u << f))) {
      dg += T(2) * c.Kn[f] * s;
    } else {
      const T m = (c.Ki + c.Kn[f]) * (T(0.5) * s);
      dg += m;
      of += m * c.un[f];
    }
  }
}

// g_i - N(u)_i of a gathered cell at the value x of u_i, with its sums dg, of
// (the expression of apply_N(), so both give the same bits)
template <typename T, int FORM, int MODEL>
__device__ __forceinline__ T cell_defect(const Level<T>& L, const Phys<T>& P, const CellOps<T>& c, T dg, T of, T x) {
  const T val = storage<T, FORM, MODEL, true>(L, x, c.psi0, c.p1, c.p2, c.smax, c.mat, P);
  return c.g - (val + P.xi * x + dg * x - of);
}

template <typename T, int FORM, int MODEL, int NK = 0, bool YZI = false>
__device__ __forceinline__ T solve_cell_sums(const Level<T>& L, const Phys<T>& P, const CellOps<T>& c, T dg, T of) {
  const T cc = P.xi + P.kappa + dg;
  const T f = c.g + of + P.kappa * c.ui;
  return point_solve_of<T, FORM, MODEL, NK>(L, c.mat, cc, f, c.ui, c.psi0, c.p1, c.p2, c.smax, P);
}

template <typename T, int FORM, int MODEL, int NK = 0, bool YZI = false>
__device__ __forceinline__ T solve_cell(const Level<T>& L, const Phys<T>& P, const CellOps<T>& c) {
  T dg, of;
  cell_sums<T, YZI>(L, c, dg, of);
  return solve_cell_sums<T, FORM, MODEL, NK, YZI>(L, P, c, dg, of);
}

// N(u)_i = storage(u_i) + xi u_i + m_ii u_i - sum_j m_ij u_j   (eq. Nh-def)
template <typename T, int FORM, int MODEL, bool YZI = false>
__device__ __forceinline__ T apply_N(const Level<T>& L, const Phys<T>& P, const T* __restrict__ u,
                                     long long i, int i0, int i1, int i2) {
  T mii, off;
  stencil<T, YZI>(L, i, i0, i1, i2, u, mii, off);
  const unsigned q = pix(L, i, i0, i1, i2);
  const T p1 = L.p1 ? L.p1[q] : P.p1;
  const T p2 = L.p2 ? L.p2[q] : P.p2;
  const T smax = L.smax ? L.smax[q] : T(0);
  const T psi0 = FORM == FORM_DELTA ? L.psi0[q] : T(0);
  const T val = storage<T, FORM, MODEL>(L, u[i], psi0, p1, p2, smax, mat_of<MODEL>(L, i), P);
  return val + P.xi * u[i] + mii * u[i] - off;
}

// (levels hold fewer than 2^31 cells: 32-bit division suffices)
__device__ __forceinline__ void cell_coords(const int n0, const int n1, long long i, int& i0, int& i1,
                                            int& i2) {
  const unsigned ui = (unsigned)i;
  const unsigned r = ui / (unsigned)n0;
  i0 = (int)(ui - r * (unsigned)n0);
  i1 = (int)(r % (unsigned)n1);
  i2 = (int)(r / (unsigned)n1);
}

// the same through the level's divisor factors
template <typename T>
__device__ __forceinline__ void cell_coords(const Level<T>& L, unsigned i, int& i0, int& i1, int& i2) {
  const unsigned r = quick_div(i, (unsigned)L.n0, L.rn0);
  const unsigned z = quick_div(r, (unsigned)L.n1, L.rn1);
  i0 = (int)(i - r * (unsigned)L.n0);
  i1 = (int)(r - z * (unsigned)L.n1);
  i2 = (int)z;
}

// thread index t over one colour -> cell (x pairs, colour chosen per row)
template <typename T>
__device__ __forceinline__ bool color_cell(const Level<T>& L, unsigned t, int color, int& i0, int& i1, int& i2,
                                           unsigned& i) {
  const unsigned nh = (unsigned)((L.n0 + 1) >> 1);
  const unsigned r = quick_div(t, nh, L.rnh);
  const unsigned z = quick_div(r, (unsigned)L.n1, L.rn1);
  const int p = (int)(t - r * nh);
  i1 = (int)(r - z * (unsigned)L.n1);
  i2 = (int)z;
  i0 = 2 * p + ((color + i1 + i2) & 1);
  if (i0 >= L.n0) return false;
  i = (unsigned)i0 + (unsigned)L.n0 * r;
  return true;
}

// ---------------------------------------------------------------------------
// One row of the linear interpolation from a coarse axis (nc cells) to fine
// cell i of a fine axis (nf cells): the coarse coordinate of the fine centre
// is ((2i+1) nc - nf) / (2 nf); a ghost beyond either end folds into the end
// cell with factor slo / shi (+1 constant extrapolation, -1 zero on a
// Dirichlet face).  Entries with zero weight are dropped, equal indices merged.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void interp_row(int nf, int nc, int i, double slo, double shi, int* idx, double* w,
                                           int& cnt) {
  cnt = 0;
  auto add = [&](int j, double wt) {
    if (wt == 0.0) return;
    for (int k = 0; k < cnt; ++k)
      if (idx[k] == j) { w[k] += wt; return; }
    idx[cnt] = j;
    w[cnt] = wt;
    ++cnt;
  };
  if (nf == 1) { add(0, 1.0); return; }
  const long long num = (long long)(2 * i + 1) * nc - nf, den = 2LL * nf;
  const long long J0 = num >= 0 ? num / den : -((-num + den - 1) / den);
  const double wt = (double)(num - J0 * den) / (double)den;
  const long long J1 = J0 + 1;
  if (J0 < 0) add(0, (1.0 - wt) * slo); else add((int)J0, 1.0 - wt);
  if (J1 >= nc) add(nc - 1, wt * shi); else add((int)J1, wt);
}

// ---------------------------------------------------------------------------
// Transfers (restriction: normalised full weighting; prolongation: linear).
// ---------------------------------------------------------------------------
template <typename T>
// (cs: fine is a per-cell parameter array of a colour-split level)
__device__ __forceinline__ T restrict_at(const Level<T>& F, const Xfer<T>& X, const T* __restrict__ fine,
                                         int J0, int J1, int J2, bool cs = false) {
  T s = T(0);
  const int c0 = X.rc[0][J0], c1 = X.rc[1][J1], c2 = X.rc[2][J2];
  for (int a2 = 0; a2 < c2; ++a2) {
    const int f2 = X.ri[2][RMAX * J2 + a2];
    const T w2 = X.rw[2][RMAX * J2 + a2];
    for (int a1 = 0; a1 < c1; ++a1) {
      const int f1 = X.ri[1][RMAX * J1 + a1];
      const T w1 = X.rw[1][RMAX * J1 + a1];
      const long long row = (long long)F.n0 * (f1 + (long long)F.n1 * f2);
      for (int a0 = 0; a0 < c0; ++a0) {
        const T w0 = X.rw[0][RMAX * J0 + a0];
        const int f0 = X.ri[0][RMAX * J0 + a0];
        const long long idx = cs ? (long long)pix_of(1, F.n0, F.n1, F.n2, (unsigned)(row + f0), f0, f1, f2) : row + f0;
        s += w0 * w1 * w2 * fine[idx];
      }
    }
  }
  return s;
}

// two natural-layout arrays through one reading of the tables (the sums of
// restrict_at)
template <typename T>
__device__ __forceinline__ void restrict2_at(const Level<T>& F, const Xfer<T>& X, const T* __restrict__ fa,
                                             const T* __restrict__ fb, int J0, int J1, int J2, T& a, T& b) {
  T sa = T(0), sb = T(0);
  const int c0 = X.rc[0][J0], c1 = X.rc[1][J1], c2 = X.rc[2][J2];
  for (int a2 = 0; a2 < c2; ++a2) {
    const int f2 = X.ri[2][RMAX * J2 + a2];
    const T w2 = X.rw[2][RMAX * J2 + a2];
    for (int a1 = 0; a1 < c1; ++a1) {
      const int f1 = X.ri[1][RMAX * J1 + a1];
      const T w1 = X.rw[1][RMAX * J1 + a1];
      const long long row = (long long)F.n0 * (f1 + (long long)F.n1 * f2);
      for (int a0 = 0; a0 < c0; ++a0) {
        const T w0 = X.rw[0][RMAX * J0 + a0];
        const long long idx = row + X.ri[0][RMAX * J0 + a0];
        sa += w0 * w1 * w2 * fa[idx];
        sb += w0 * w1 * w2 * fb[idx];
      }
    }
  }
  a = sa;
  b = sb;
}

// sum_J P(i, J) (u_c - ubar_c)(J)
template <typename T>
__device__ __forceinline__ T prolong_at(const Level<T>& C, const Xfer<T>& X, int i0, int i1, int i2) {
  T s = T(0);
  const int c0 = X.pc[0][i0], c1 = X.pc[1][i1], c2 = X.pc[2][i2];
  for (int a2 = 0; a2 < c2; ++a2) {
    const int J2 = X.pj[2][2 * i2 + a2];
    const T w2 = X.pw[2][2 * i2 + a2];
    for (int a1 = 0; a1 < c1; ++a1) {
      const int J1 = X.pj[1][2 * i1 + a1];
      const T w1 = X.pw[1][2 * i1 + a1];
      const long long row = (long long)C.n0 * (J1 + (long long)C.n1 * J2);
      for (int a0 = 0; a0 < c0; ++a0) {
        const T w0 = X.pw[0][2 * i0 + a0];
        const long long J = row + X.pj[0][2 * i0 + a0];
        s += w0 * w1 * w2 * (C.u[J] - C.ubar[J]);
      }
    }
  }
  return s;
}

// ---------------------------------------------------------------------------
// max-norm reductions: |x| of finite or NaN values compares as its bit
// pattern (NaN sorts above +inf, so a NaN anywhere survives the max).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long nbits(double x) {
  return (unsigned long long)__double_as_longlong(fabs(x));
}
__device__ __forceinline__ unsigned long long nbits(float x) {
  return (unsigned long long)__float_as_uint(fabsf(x));
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// block-wide max of v; every thread gets the result (uses 33 words of smem)
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* sm) {
  v = warp_max(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sm[wid] = v;
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    unsigned long long x = lane < nw ? sm[lane] : 0ull;
    x = warp_max(x);
    if (lane == 0) sm[32] = x;
  }
  __syncthreads();
  return sm[32];
}

}  // namespace rich
