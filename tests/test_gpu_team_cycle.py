"""The coarse tail and the small-grid step as thread-block clusters (needs a
GPU): FP64 cycles against the oracle, and mixed steps the same bits, whatever
part of the hierarchy a cluster, a single block or the grid kernels take.

Sizes sit at the switches: levels just below and above the cells one block
keeps (256 in FP64, 1024 in FP32), the small-step limit of 4096, the biggest
level a cluster takes (4608 cells in FP64; 32768 in 2-d and 16384 in 3-d in
FP32), odd and even.  FP64 cycle tests run Newton to round-off, as every
iterate comparison does, at the oracle's 1e-10.
"""
import numpy as np
import pytest

from oracle.oracle import ORC_OK, Oracle
from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402

FP64_CASES = [((255,), 1, 0), ((257,), 2, 2), ((4096,), 1, 3), ((4097,), 1, 0), ((64, 64), 2, 2), ((65, 65), 1, 0),
              ((136, 134), 2, 0), ((16, 16, 16), 2, 2), ((33, 17, 19), 1, 3)]


def _problem(n, cycle, gamma_levels, **kw):
    return W.random_problem(len(n), n, W.VANGENUCHTEN, 5, hetero=True, sink=True, newton_iters=0,
                            coarse_max_sweeps=3, coarse_rtol=1e-30, cycle_gamma=cycle, gamma_levels=gamma_levels, **kw)


@pytest.mark.parametrize("n,gamma,gamma_levels", FP64_CASES)
def test_fp64_steps_match_the_oracle(n, gamma, gamma_levels):
    prob = _problem(n, gamma, gamma_levels, tol=1e-12, max_cycles=40)
    orc = Oracle(prob)
    with R.Solver(prob) as gs:
        for _ in range(2):
            st, info = gs.step(check=False)
            ost, oinfo = orc.step()
            assert (st == R.RICH_OK) == (ost == ORC_OK)
            assert info["cycles"] == oinfo["cycles"]
        ref = orc.state()
        assert np.linalg.norm(gs.state() - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [(63, 33), (128, 128), (182, 181), (258, 257), (33, 32, 31), (50, 52, 54)])
@pytest.mark.parametrize("nu", [(2, 2), (0, 2)])
def test_mixed_steps_same_bits_for_any_tail(n, nu):
    """tail_cells moves the single-block levels; with it at 1 only the
    coarsest level is a tail level and the transfers above it are the grid
    kernels'."""
    states = []
    for dev in (1, 0):
        prob = W.random_problem(len(n), n, W.VANGENUCHTEN, 6, hetero=True, scheme=2, precision=2, tol=1e-10,
                                nu1=nu[0], nu2=nu[1], cycle_gamma=2, gamma_levels=2, tail_cells=1, graphs=dev)
        with R.Solver(prob, stream=torch.cuda.Stream().cuda_stream) as gs:
            if not dev:
                gs.set_coop(10 ** 6)           # grid barriers instead of cluster barriers
            # (a random field need not reach the tolerance: the outcome is compared)
            runs = [gs.step(check=False) for _ in range(2)]
            states.append((gs.state(), [(st, i["cycles"], i["resid"]) for st, i in runs]))
    assert states[0][1] == states[1][1]
    assert np.array_equal(states[0][0], states[1][0])
