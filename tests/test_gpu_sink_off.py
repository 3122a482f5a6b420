"""A sink that is switched off takes up no more water (needs a GPU): a context
that has stepped with root uptake and is then given no sink steps, bit for bit,
like one that never had a sink -- alone and in a batch, on grids whose levels
run in one block, in a cluster and in the grid kernels.
"""
import numpy as np
import pytest

from paper_2606_04292_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04292_gb300 import richards as R  # noqa: E402


def _solvers(n, precision, stream):
    """One solver whose sink was switched off after a step, one that never had one."""
    on = W.random_problem(len(n), n, W.VANGENUCHTEN, 8, sink=True, precision=precision, tol=1e-10)
    on["psi0"] = 0.1 * on["psi0"] - 0.08          # on the uptake's ramp, -0.25 to -0.1 m
    off = dict(on, sink=W.no_sink())
    a = R.Solver(on, stream=stream)
    a.step()
    a.set_sink(off["sink"])
    a.set_state(on["psi0"])
    return a, R.Solver(off, stream=stream), on["dt"]


@pytest.mark.parametrize("n", [(60,), (70, 61), (40, 36, 33)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_step_without_the_sink(n, precision):
    s = torch.cuda.Stream().cuda_stream
    a, b, _ = _solvers(n, precision, s)
    assert a.step() == b.step()
    assert np.array_equal(a.state(), b.state())


@pytest.mark.parametrize("n", [(60,), (70, 61), (40, 36, 33)])
def test_batched_step_without_the_sink(n):
    s = torch.cuda.Stream().cuda_stream
    a, b, dt = _solvers(n, 2, s)
    status, info = R.Batcher(2, stream=s).step([a, b], [dt, dt], [1, 1])
    assert status == [R.RICH_OK] * 2 and info[0] == info[1]
    assert np.array_equal(a.state(), b.state())
