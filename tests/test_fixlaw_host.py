"""The fixed-point laws (csrc/fixlaw.cuh) compiled for the host: each law's
saturation, slope and conductivity, through prepared and per-cell parameters,
against extended precision; the integer quotients against a/b.

Bounds in ulps of the result (2^-53 to 2^-52 of it), from the arithmetic:
log2 to 0.55 of its unit 2^-56, so t = n (la + lh) to 1.1 n + 1 units (n <=
5.5: 7; Haverkamp's n lh - la, n <= 5: 4.3); the saturation's exponent adds 3
units, the slope's sum of three quarters 9 more; a unit is ln 2 / 16 of an ulp
at a significand of 1 and twice that just below 2; the result is rounded once.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_04292_gb300", "csrc")
LD = np.longdouble
if np.finfo(LD).nmant < 63:
    pytest.skip("needs an extended long double", allow_module_level=True)

HARNESS = r"""
#include "fixlaw.cuh"
using namespace rich::fl;
extern "C" {
// how: 0 prep, 1 host_prep, 2 any (all with the slope), 3 parameters of a cell
void law(int model, int how, long n, const double* p1, const double* p2, const double* h, double* Se, double* s,
         unsigned char* okv) {
  for (long i = 0; i < n; ++i) {
    bool ok = true;
    const u64 hb = dbits(h[i]);
    s[i] = 0.0;
    if (how == 3) {
      Se[i] = model == 1 ? exp_gardner(p1[i], hb, ok) : model == 2 ? se_only<true>(p1[i], p2[i], hb, ok)
                                                                   : se_only<false>(p1[i], p2[i], hb, ok);
    } else {
      const bool vg = model == 2;
      const Prep q = how == 0 ? (vg ? prep<true>(p1[i], p2[i]) : prep<false>(p1[i], p2[i]))
                              : model == 1 ? host_prep(false, 1.0, 1.0) : host_prep(vg, p1[i], p2[i]);
      ok = q.ok;
      if (how == 2) se_any<true>(model, q, p1[i], hb, ok, Se[i], s[i]);
      else if (vg) se_slope<true>(q, hb, ok, Se[i], s[i]);
      else se_slope<false>(q, hb, ok, Se[i], s[i]);
    }
    okv[i] = ok;
  }
}
void kr(int model, long n, const double* p1, const double* p2, const double* l, const double* h, double* K,
        unsigned char* okv) {
  for (long i = 0; i < n; ++i) {
    bool ok = true;
    K[i] = model == 2 ? kr_vangenuchten(p1[i], p2[i], l[i], dbits(h[i]), ok)
                      : kr_haverkamp(p1[i], p2[i], dbits(h[i]), ok);
    okv[i] = ok;
  }
}
void quotient(long n, const double* a, const double* b, double* q) {
  for (long i = 0; i < n; ++i) q[i] = div(a[i], divisor(b[i]));
}
}
"""
N = 200000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixlaw")
    src, so = d / "fixlaw.cpp", d / "fixlaw.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    return C.CDLL(str(so))


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _ulps(got, ref):
    return np.max(np.abs((got.astype(LD) - ref).astype(float)) / np.spacing(ref.astype(float)))


def _soils(model, seed):
    rng = np.random.default_rng(seed)
    h = np.exp(rng.uniform(np.log(1e-6), np.log(150.0), N))
    if model == 2:
        return rng.uniform(0.3, 5.0, N), rng.uniform(1.05, 5.5, N), h
    if model == 1:
        p1 = rng.uniform(0.3, 5.0, N)
        return p1, np.ones(N), np.minimum(h, 60.0 / p1)
    return np.exp(rng.uniform(-5, 13, N)), rng.uniform(0.5, 5.0, N), h      # (|t| up to 119 of 120)


@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("how", [0, 1, 2, 3])
def test_saturation_and_slope(lib, model, how):
    if model == 1 and how < 2:
        pytest.skip("Gardner's exponent has nothing to prepare")
    p1, p2, h = _soils(model, 10 * model + how)
    Se, s, ok = np.empty(N), np.empty(N), np.empty(N, np.uint8)
    lib.law(model, how, C.c_long(N), _p(p1), _p(p2), _p(h), _p(Se), _p(s), _p(ok))
    assert np.all(ok)
    a, n, x = p1.astype(LD), p2.astype(LD), h.astype(LD)
    if model == 1:
        ref, slope = np.exp(-a * x), np.exp(-a * x)
    else:
        T = np.exp(n * np.log(a * x)) if model == 2 else np.exp(n * np.log(x)) / a
        m = 1 - 1 / n if model == 2 else LD(1)
        ref = np.exp(-m * np.log1p(T))
        slope = ref / (1 + 1 / T) / x
    assert _ulps(Se, ref) <= {0: 1.2, 1: 0.9, 2: 1.4}[model]
    if how < 3:
        assert _ulps(s, slope) <= {0: 1.8, 1: 0.9, 2: 2.1}[model]


@pytest.mark.parametrize("l", [0.5, 0.0, -1.0, -2.0, 2.5])
def test_conductivity_of_van_genuchten(lib, l):
    p1, p2, h = _soils(2, 41)
    K, ok, lv = np.empty(N), np.empty(N, np.uint8), np.full(N, l)
    lib.kr(2, C.c_long(N), _p(p1), _p(p2), _p(lv), _p(h), _p(K), _p(ok))
    a, n, x = p1.astype(LD), p2.astype(LD), h.astype(LD)
    m, lt = 1 - 1 / n, n * np.log(a * x)
    e = np.log1p(np.exp(-np.abs(lt)))
    ref = np.exp(-LD(l) * m * (e + np.maximum(lt, 0))) * np.expm1(m * (np.minimum(lt, 0) - e)) ** 2
    assert np.all(ok)
    assert _ulps(K, ref) <= 2.2


def test_conductivity_of_haverkamp(lib):
    p1, p2, h = _soils(0, 42)
    K, ok = np.empty(N), np.empty(N, np.uint8)
    lib.kr(0, C.c_long(N), _p(p1), _p(p2), _p(p2), _p(h), _p(K), _p(ok))
    assert np.all(ok)
    assert _ulps(K, 1 / (1 + np.exp(p2.astype(LD) * np.log(h.astype(LD))) / p1.astype(LD))) <= 1.2


def test_quotients(lib):
    rng = np.random.default_rng(7)
    n = 2000000
    b = np.ldexp(rng.uniform(1, 2, n), rng.integers(-380, 380, n)) * rng.choice([-1.0, 1.0], n)
    a = np.ldexp(rng.uniform(1, 2, n), rng.integers(-380, 380, n))
    edge = np.array([1.0, np.nextafter(2.0, 0), np.nextafter(1.0, 2), 3.0, 1.5, 0.0, 5e-324, 1e308, np.inf])
    a[:81], b[:81] = np.repeat(edge, 9), np.tile(edge, 9)
    q = np.empty(n)
    lib.quotient(C.c_long(n), _p(a), _p(b), _p(q))
    with np.errstate(all="ignore"):
        ref = a / b
    assert np.array_equal(q, ref, equal_nan=True)
