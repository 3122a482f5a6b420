"""The fixed-point FP64 laws (theta, K of Table 1) at the edges of their
ranges, against extended-precision values (needs a GPU).

The heads cover the reduction's edges (alpha h at and beside powers of two and
the table's steps j/64, the switch 2^-|t| = 1/64, T = 1) and both sides of
the limits beyond which the FP64 functions take over (alpha h of 2^+-100, |t| =
120, n = 16, |l| = 1/32).  Tolerances: inside the ranges K/Ks carries at most
2.2 ulps and theta's Se 1 ulp, plus the rounding of the last product and sum;
outside, the FP64 functions' own: the roundings of alpha h (n/2 ulps of T) and
of the exponent (|t| ulps), times the powers of T in K, on top of a few ulps
of each function.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402

LD = np.longdouble
EPS = 2.0 ** -52
TS, TR = 0.368, 0.102


def _eval(model, h, p1, p2, p3=0.0, p4=0.0):
    """theta and K (Ks = 1) at -h through the library."""
    n = len(h)
    prob = W.random_problem(1, n, W.VANGENUCHTEN, 1, precision=0)
    prob["soil"] = dict(prob["soil"], model=model, Ks=1.0, theta_s=TS, theta_r=TR, p1=float(p1[0]),
                        p2=float(p2[0]) if len(p2) else 0.0, p3=p3, p4=p4, p1_field=p1,
                        p2_field=p2 if len(p2) else None)
    with R.Solver(prob) as s:
        return s.soil_eval(-h)


def _near(v):
    return np.concatenate([np.nextafter(v, 0.0), v, np.nextafter(v, np.inf)])


def _heads(rng):
    """Values of alpha h (or h): powers of two, table steps, random spreads."""
    steps = (1.0 + np.arange(64) / 64.0)
    return np.concatenate([_near(2.0 ** np.arange(-30, 31)), _near(steps), _near(0.5 * steps),
                           np.exp(rng.uniform(-40, 30, 4000)), 1.0 + rng.uniform(-0.03, 0.03, 500)])


@pytest.mark.parametrize("n", [1.0625, 1.2, 2.0, 3.5, 6.0, 15.9, 16.0, 63.9])
@pytest.mark.parametrize("l", [0.5, 0.0, -1.0, 0.03, 2.5])
def test_van_genuchten(n, l):
    rng = np.random.default_rng(3)
    ah = np.concatenate([_heads(rng), _near(2.0 ** (np.arange(-16, 17) / n)), _near(2.0 ** (np.array([-6.0, 6.0]) / n)),
                         2.0 ** np.array([-110.0, -100.0, -99.5, 99.5, 101.0]), 2.0 ** (np.array([-121, -119, 119, 121]) / n)])
    al = rng.uniform(0.5, 5.0, len(ah))
    h = ah / al
    th, K = _eval(W.VANGENUCHTEN, h, al, np.full(len(h), n), p3=l)
    N, m = LD(n), 1 - 1 / LD(n)
    lt = N * np.log(al.astype(LD) * h.astype(LD))
    e = np.exp(-np.abs(lt))
    L1, lr = np.log1p(e) + np.maximum(lt, 0), np.minimum(lt, 0) - np.log1p(e)
    Se = np.exp(-m * L1)
    Kr = np.exp(-LD(l) * m * L1) * np.expm1(m * lr) ** 2
    t = np.abs(lt.astype(float)) / np.log(2.0)
    fast = (n < 16) & (t < 119.9) & (np.abs(np.log2(ah)) < 99)
    fastK = fast & (abs(l) >= 1 / 32 or l == 0.0) & (abs(l) * (L1 * m).astype(float) / np.log(2.0) < 119.9)
    tolS = np.where(fast, 1.0, 16.0 + n + 4.0 * t) * EPS * Se.astype(float)
    assert np.all(np.abs(th - (LD(TR) + LD(TS - TR) * Se)).astype(float) <= (TS - TR) * tolS + TS * EPS)
    keep = Kr > 1e-280
    tolK = np.where(fastK, 3.0, 32.0 + (n + 8.0 * t) * (2 + abs(l))) * EPS
    assert np.all((np.abs(K - Kr) / Kr).astype(float)[keep] <= tolK[keep])


@pytest.mark.parametrize("beta", [0.04, 0.9, 3.96, 8.0])
def test_haverkamp(beta):
    rng = np.random.default_rng(4)
    h = np.concatenate([_heads(rng), 2.0 ** np.array([-110.0, 99.5, 101.0])])
    al = np.exp(rng.uniform(-8, 15, len(h)))
    th, K = _eval(W.HAVERKAMP, h, al, np.full(len(h), beta), p3=0.7, p4=beta + 0.5)
    u = h.astype(LD) ** LD(beta) / al.astype(LD)
    v = h.astype(LD) ** LD(beta + 0.5) / LD(0.7)
    t = np.maximum(np.abs(np.log2(u.astype(float))), beta * np.abs(np.log2(h)))
    fast = (t < 119.9) & (np.abs(np.log2(h)) < 99)
    tol = np.where(fast, 1.0, 16.0 + 4.0 * t) * EPS
    assert np.all(np.abs(th - (LD(TR) + LD(TS - TR) / (1 + u))).astype(float) <= (TS - TR) * tol + TS * EPS)
    t = np.maximum(np.abs(np.log2(v.astype(float))), (beta + 0.5) * np.abs(np.log2(h)))
    tol = np.where((t < 119.9) & (np.abs(np.log2(h)) < 99), 2.0, 32.0 + 8.0 * t) * EPS
    assert np.all((np.abs(K - 1 / (1 + v)) * (1 + v)).astype(float) <= tol)


def test_gardner_and_saturation():
    rng = np.random.default_rng(5)
    al = np.concatenate([rng.uniform(0.1, 5.0, 4000), np.ones(6)])
    h = np.concatenate([np.exp(rng.uniform(-60, 3, 4000)), [63.9, 64.1, 1e-300, 300.0, 0.0, -1.0]])
    th, K = _eval(W.GARDNER, h, al, np.empty(0))
    e = np.where(h > 0, np.exp(-al.astype(LD) * np.maximum(h, 0).astype(LD)), LD(1))
    tol = np.where(al * h < 63.9, 2.0, 16.0 + 4.0 * al * h) * EPS
    assert np.all((np.abs(K - e) / e).astype(float) <= tol)
    assert np.all(np.abs(th - (LD(TR) + LD(TS - TR) * e)).astype(float) <= (TS - TR) * tol + TS * EPS)
    assert th[-2] == th[-1] == TS and K[-2] == K[-1] == 1.0
