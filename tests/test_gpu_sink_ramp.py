"""The root-uptake ramps of the FP64 sink are correctly rounded quotients
(needs a GPU): bit for bit numpy's (h1 - psi)/(h1 - h2) and (psi - h4)/(h3 -
h4).  Saturated cells of a vanishing conductivity and storage rate, so that
the defect of a zero right side is the sink alone.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402


@pytest.mark.parametrize("h", [(5.0, 1.0, 0.5, 0.1), (3.3, 3.1, 2.9, 0.7), (1e-3, 7e-4, 7e-4, 1e-5),
                               (2.0 ** 60, 3.0, 1.0, 0.9)])
def test_ramps_are_correctly_rounded(h):
    n = 3000
    h1, h2, h3, h4 = h
    rng = np.random.default_rng(11)
    psi = np.concatenate([rng.uniform(h2, h1, n // 2), rng.uniform(h4, h3, n - n // 2)])
    psi[:4] = h1, h2, h3, h4
    prob = W.random_problem(1, n, W.VANGENUCHTEN, 3, sink=True, precision=0, bc_kinds=[W.NOFLUX, W.NOFLUX])
    prob["soil"]["Ks"] = 1e-290
    prob["sink"].update(h1=h1, h2=h2, h3=h3, h4=h4, root_depth=1e3, root_decay=1e3)
    prob["psi0"] = psi
    with R.Solver(prob) as gs:
        gs.prepare(1e290, 1)
        gs.set_level(0, 1, np.zeros(n))
        gs.set_level(0, 0, psi)
        gs.residual(0)
        S = -gs.get_level(0, 7)
        smax = gs.get_level(0, 5)
    assert np.all(smax > 0)
    with np.errstate(divide="ignore", invalid="ignore"):
        a = np.where(psi >= h1, 0.0, np.where(psi < h4, 0.0, np.where(psi >= h2, (h1 - psi) / (h1 - h2), np.where(
            psi >= h3, 1.0, (psi - h4) / (h3 - h4)))))
    assert np.array_equal(S[a > 0], (a * smax)[a > 0])
    assert np.all(np.abs(S[a == 0]) < 1e-200)           # (the last trace of the flow)
