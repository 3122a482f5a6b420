"""Float-float theta (needs a GPU) against the FP64 laws: both take the
saturation from the same fixed-point law, so they differ by the pair's
rounding alone.  With u = 2^-46 (a split double, a pair product, a pair sum)
theta = theta_r + ds Se is within 4 u theta_s of the exact value of its
operands, plus FP64's own 2 ulp.

Soils: each law uniform and with per-cell fields, and a layered soil.  Heads:
the whole range, the edges of the fixed-point ranges (tiny and huge heads,
which take the general functions), zeros of both signs.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402

TOL = 4 * 2.0 ** -46 + 4 * 2.0 ** -53


def _problem(soil):
    if soil == "layers":
        p = W.random_problem(3, (16, 12, 11), W.VANGENUCHTEN, 5)
        return W.with_materials(p, W.test_materials(), W.material_pattern(p, "random", 3, 5)), 1.0
    law, fields = soil
    p = W.random_problem(3, (16, 12, 11), law, 6, hetero=fields)
    return p, p["soil"]["theta_s"]


@pytest.mark.parametrize("soil", [(m, f) for m in (W.HAVERKAMP, W.GARDNER, W.VANGENUCHTEN) for f in (False, True)]
                         + ["layers"], ids=str)
def test_pair_theta_is_the_fp64_theta(soil):
    prob, ts = _problem(soil)
    gs = R.Solver(prob)
    rng = np.random.Generator(np.random.PCG64(9))
    psi = -np.exp(rng.uniform(np.log(1e-12), np.log(1e6), gs.N))
    edges = [0.0, -0.0, 1.0, -5e-324, -1e-310, -1e-300, -2.0 ** -100, -2.0 ** -101, -1e30, -1e300, -1.0, -2.0]
    psi[:len(edges)] = edges
    th64, _ = gs.soil_eval(psi, arith=0)
    thdd, _ = gs.soil_eval(psi, arith=1)
    assert np.all(np.isfinite(thdd))
    assert np.max(np.abs(thdd - th64)) <= TOL * ts
