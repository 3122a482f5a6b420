"""The coarsest level's sweeps in FP32 (needs a GPU): a solve that meets a
state again ends early, with the bits that all of its sweeps would leave.

One-level grids with one outer correction, so the inner solve is the coarsest
one alone; coarse_rtol is far below round-off.  The reference takes the same
sweeps as cycles of one sweep each, which never look back: alone, in a batch and
as columns.  The sweeps that ran are counted (cell_updates).
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402


def _problem(n, seed, cmax, cycles, **kw):
    p = W.random_problem(len(n), n, W.VANGENUCHTEN, seed, precision=2, tol=1e-30, max_outer=1, inner_rtol=0.0,
                         coarsest_max_n=65, coarse_rtol=1e-30, coarse_max_sweeps=cmax, inner_cycles=cycles, **kw)
    p["psi0"] = 0.2 * p["psi0"] - 0.5
    return p


def _alone(p):
    with R.Solver(p) as gs:
        assert gs.nlevels == 1
        _, info = gs.step(check=False)
        return gs.state(), info["cell_updates"] // gs.N


def _period(n, seed, newton, upto):
    """The period that the sweeps' states have reached after `upto` sweeps."""
    last = _alone(_problem(n, seed, 1, upto, newton_iters=newton))[0]
    for p in range(1, 60):
        if np.array_equal(_alone(_problem(n, seed, 1, upto - p, newton_iters=newton))[0], last):
            return p
    return 0


@pytest.mark.parametrize("n", [(1,), (5,), (64,), (65,), (8, 8), (4, 4, 4), (3, 4, 2)], ids=str)
@pytest.mark.parametrize("newton", [2, 0])
def test_same_bits(n, newton):
    for cmax in (2, 3, 5, 8, 33, 400, 401):
        state, sweeps = _alone(_problem(n, 31, cmax, 1, newton_iters=newton))
        ref, all_sweeps = _alone(_problem(n, 31, 1, cmax, newton_iters=newton))
        assert np.array_equal(state, ref), cmax
        assert all_sweeps == cmax
        assert sweeps <= cmax if np.prod(n) <= 64 else sweeps == cmax      # (more cells are not looked at)


@pytest.mark.parametrize("n", [(1,), (5,), (4, 4)], ids=str)
def test_solves_do_end_early(n):
    """Most soils' sweeps come back to a state, some at a period above 1."""
    seeds = range(31, 37)
    early = [_alone(_problem(n, s, 400, 1))[1] < 400 for s in seeds]
    assert sum(early) >= 4
    assert any(e and _period(n, s, 2, 200) > 1 for e, s in zip(early, seeds))


def test_columns_and_batches():
    sizes, seeds = (2, 5, 17, 64, 65), (31, 32, 33)
    probs = lambda cmax, cycles: [_problem((n,), s, cmax, cycles) for n in sizes for s in seeds]
    sides = []
    for cmax, cycles in ((400, 1), (1, 400)):
        cols = R.Columns(probs(cmax, cycles))
        cols.run(60.0, 1)
        sides.append((cols.state(), cols.stats()["updates"]))
        cols.close()
    assert np.array_equal(sides[0][0], sides[1][0])
    assert np.all(sides[0][1] <= sides[1][1]) and np.sum(sides[0][1] < sides[1][1]) >= 6   # (of 9 short columns)

    s = torch.cuda.Stream().cuda_stream
    many = [R.Solver(p, stream=s) for p in probs(400, 1)]
    b = R.Batcher(len(many), stream=s)
    _, info = b.step(many, [p["dt"] for p in probs(400, 1)], [1] * len(many))
    for gs, i, p in zip(many, info, probs(400, 1)):
        state, sweeps = _alone(p)
        assert np.array_equal(gs.state(), state) and i["cell_updates"] == sweeps * gs.N
