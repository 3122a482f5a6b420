"""Batched coarse tails (needs a GPU): whatever number of requests meet in a
launch, and so whatever cluster size it takes and whichever levels go into
it, each request's step is the one it takes alone, bit for bit.

Counts sit at the sizes' limits on a device that holds 7 clusters of 16 blocks,
15 of 8, 36 of 4 and 76 of 2 at once, and past the 64 descriptors of a launch.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402

OPTS = dict(precision=2, tol=1e-9)


def _requests():
    """A request of every kind: dimensions, laws, a sink, odd and even sizes."""
    return [W.random_problem(1, 300, W.VANGENUCHTEN, 1, sink=True, **OPTS),
            W.random_problem(2, (33, 30), W.GARDNER, 2, **OPTS),
            W.random_problem(2, (67, 64), W.VANGENUCHTEN, 3, hetero=True, **OPTS),
            W.random_problem(3, (17, 16, 15), W.HAVERKAMP, 4, **OPTS),
            W.random_problem(3, (26, 25, 24), W.VANGENUCHTEN, 5, sink=True, **OPTS)]


def _check(probs, alone):
    s = torch.cuda.Stream().cuda_stream
    many = [R.Solver(p, stream=s) for p in probs]
    b = R.Batcher(len(many), stream=s)
    status, info = b.step(many, [p["dt"] for p in probs], [1] * len(many))
    for k, gs in enumerate(many):
        st, one, state = alone[k % len(alone)]
        assert status[k] == st and info[k]["cycles"] == one["cycles"] and info[k]["resid"] == one["resid"]
        assert np.array_equal(gs.state(), state), k
        gs.close()
    b.close()


def _alone(probs):
    out = []
    for p in probs:
        with R.Solver(p, stream=torch.cuda.Stream().cuda_stream) as gs:
            st, info = gs.step(check=False)
            out.append((st, info, gs.state()))
    return out


def test_any_number_of_requests():
    kinds = _requests()
    alone = _alone(kinds)
    for n in (1, 7, 8, 15, 16, 36, 37, 64, 77):
        _check([kinds[k % len(kinds)] for k in range(n)], alone)


@pytest.mark.parametrize("n", [2, 9, 18])
@pytest.mark.parametrize("sizes", [[(80, 80, 79), (82, 81, 82)], [(514, 510), (514, 514)]])
def test_levels_on_both_sides_of_the_clusters_limit(n, sizes):
    """Level 1 just below and just above the 66000 cells that clusters take."""
    probs = [W.random_problem(len(m), m, W.VANGENUCHTEN, 6, **OPTS) for m in sizes]
    for p in probs:
        p["psi0"] = 0.2 * p["psi0"] - 0.5
    alone = _alone(probs)
    _check([probs[k % 2] for k in range(n)], alone)
