"""The FP32 increment law where a power of the frozen state, or the coupling
to the neighbours, leaves FP32's normal range (needs a GPU): heads close to
saturation under a steep law, and dry Gardner soils whose conductivity has all
but vanished.

One outer correction of a four-cell column, whose inner problem is solved to
its round-off.  The correction law is good to ~2e-5 of the storage change (an
exponent of up to 90 through hardware logarithms and exponentials) or, where
e^(alpha psi0) has 16 bits left, to 2e-5 as well, so the FP64 defect falls by
more than 1e3; with the storage term lost it does not fall at all.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402


def _drop(soil, bc, psi0, dt):
    """||defect|| after one outer correction over the one before it."""
    opts = W.default_opts(precision=2, tol=1e-30, max_outer=1, inner_cycles=50, inner_rtol=1e-7, newton_iters=0,
                          coarsest_max_n=4, coarse_max_sweeps=400, coarse_rtol=1e-7)
    prob = dict(dim=1, n=(4, 1, 1), L=(1.0, 1.0, 1.0), soil=soil, bc=bc, sink=W.no_sink(),
                psi0=np.full(4, psi0), psi_prev=None, dt=dt, nsteps=1, scheme=1, opts=opts)
    with R.Solver(prob) as gs:
        assert gs.nlevels == 1
        status, info = gs.step(check=False)
        assert status == R.RICH_ENOCONV and info["outer_iters"] == 1
        return info["resid"] / info["resid0"]


# (storage change and flow over the step are of one size: a ds |dSe| ~ K |dpsi| / h^2)
@pytest.mark.parametrize("law,p1,p2,psi0", [
    (W.VANGENUCHTEN, 1.0, 5.0, -2.5e-8), (W.VANGENUCHTEN, 1.0, 5.0, -1e-40), (W.VANGENUCHTEN, 1.0, 15.0, -2.9e-3),
    (W.VANGENUCHTEN, 1.0, 15.0, -1e-3), (W.VANGENUCHTEN, 2.0, 1.5, -1e-39), (W.VANGENUCHTEN, 1.0, 5.0, -3e-8),
    (W.HAVERKAMP, 1.0, 9.0, -5e-5), (W.HAVERKAMP, 1.0, 9.0, -1e-5), (W.HAVERKAMP, 1.0, 3.0, -1e-38),
    (W.GARDNER, 2.0, 0.0, -1e-39)])
def test_drainage_from_just_below_saturation(law, p1, p2, psi0):
    soil = W._soil(law, Ks=1e-5, theta_s=0.4, theta_r=0.1, p1=p1, p2=p2, p3=0.5 if law != W.HAVERKAMP else 1.0,
                   p4=p2)
    bc = W._bc([W.DIRICHLET, W.NOFLUX], [-0.5, 0.0])
    r = _drop(soil, bc, psi0, 2.5 if p2 > 4 else 250.0)
    assert r <= 1e-3, r


@pytest.mark.parametrize("psi0", [-86.0, -88.0, -90.0, -91.0])
def test_infiltration_into_a_dry_gardner_soil(psi0):
    soil = W._soil(W.GARDNER, Ks=100.0, theta_s=0.4, theta_r=0.1, p1=1.0)
    bc = W._bc([W.NOFLUX, W.FLUX], [0.0, 1e-6])
    r = _drop(soil, bc, psi0, 1.0)
    assert r <= 1e-3, r


@pytest.mark.parametrize("psi0", [-79.0, -81.0, -86.0, -90.0, -91.0])
def test_infiltration_into_a_gardner_soil_that_hardly_conducts(psi0):
    """K / h^2 below 2^-126 (1e-5 e^-79 = 5e-40) and not yet 0 in FP32."""
    soil = W._soil(W.GARDNER, Ks=1e-5, theta_s=0.4, theta_r=0.1, p1=1.0)
    bc = W._bc([W.NOFLUX, W.FLUX], [0.0, 1e-6])
    r = _drop(soil, bc, psi0, 1.0)
    assert r <= 1e-3, r
