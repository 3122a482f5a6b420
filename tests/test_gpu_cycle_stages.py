"""FP64 cycles in one launch (needs a GPU) against the same cycles put together
from single stages (half-sweeps, defect, restriction, right side,
interpolation: a grid kernel each): the same bits, whatever part of the
hierarchy one block or a cluster takes.

From tail_start on the transfers go through the tables, as the stages do where
the levels do not nest; so tail_cells varies on sizes whose levels are all odd,
and the sizes that nest keep their tail to the coarsest level.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402

ODD = [(257,), (4097,), (65, 65), (129, 65), (33, 17, 17)]
CASES = [(n, t) for n in ODD for t in (1, 300, 4096)] + [(n, 1) for n in [(256,), (64, 64), (96, 64), (16, 16, 16),
                                                                          (32, 16, 32)]]


def _cycle(gs, l, o):
    if l == gs.nlevels - 1:
        gs.sweep(l)
        return
    for _ in range(o["nu1"]):
        gs.sweep(l)
    gs.restrict_tau(l)
    visits = o["cycle_gamma"] if o["gamma_levels"] <= 0 or l < o["gamma_levels"] else 1
    for _ in range(visits):
        _cycle(gs, l + 1, o)
    gs.prolong(l)
    for _ in range(o["nu2"]):
        gs.sweep(l)


@pytest.mark.parametrize("n,tail_cells", CASES, ids=str)
@pytest.mark.parametrize("gamma,sink,ordering", [(1, True, 1), (2, False, 1), (1, False, 0)])
def test_cycle_is_its_stages(n, tail_cells, gamma, sink, ordering):
    prob = W.random_problem(len(n), n, W.VANGENUCHTEN, 9, hetero=True, sink=sink, ordering=ordering,
                            coarsest_max_n=2, coarse_max_sweeps=1, cycle_gamma=gamma, gamma_levels=2,
                            tail_cells=tail_cells)
    a, b = R.Solver(prob), R.Solver(prob)
    a.prepare(prob["dt"], 1)
    b.prepare(prob["dt"], 1)
    for _ in range(2):
        a.vcycle()
        _cycle(b, 0, prob["opts"])
    assert np.array_equal(a.get_level(0, 0), b.get_level(0, 0))
