"""The coarsest level's sweeps (needs a GPU): a solve that meets a state again
ends early, with the bits that all of its sweeps would leave.

One-level grids, so a cycle is the coarsest solve alone.  coarse_rtol is far
below round-off: without the early end every solve takes all its sweeps.  The
reference takes the same sweeps one cycle (of one sweep) at a time.  Sizes: one
cell, a few, the 64 cells that are followed, one more than that.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402


@pytest.mark.parametrize("n", [(1,), (4,), (64,), (65,), (5, 4), (8, 8), (4, 4, 4), (3, 4, 2)])
@pytest.mark.parametrize("ordering", [1, 0])
@pytest.mark.parametrize("newton", [2, 0])
def test_repeated_states_end_with_the_same_bits(n, ordering, newton):
    def solver(cmax):
        prob = W.random_problem(len(n), n, W.VANGENUCHTEN, 31, sink=True, ordering=ordering, newton_iters=newton,
                                coarsest_max_n=65, coarse_rtol=1e-300, coarse_max_sweeps=cmax)
        gs = R.Solver(prob)
        assert gs.nlevels == 1
        gs.prepare(prob["dt"], 1)
        return gs

    one = solver(1)
    done = 0
    for cmax in (2, 3, 4, 5, 8, 33, 400, 401):
        while done < cmax:
            one.vcycle()
            done += 1
        many = solver(cmax)
        many.vcycle()
        assert np.array_equal(many.get_level(0, 0), one.get_level(0, 0)), cmax
