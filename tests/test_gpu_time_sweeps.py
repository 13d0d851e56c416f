"""weno_time_sweeps and weno_autotune time the kernels that a step runs: the
kernels' names, which hold their template arguments, as the profiler lists
them (tile shapes pinned)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


def _sweeps(f):
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return {e.name for e in p.events() if "k_sweep<" in e.name or "k_march<" in e.name}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("n,tiles", [([9001], [0]), ([70, 45], [3, 1]), ([70, 45], [3, 7]), ([40, 20, 24], [3, 1, 2])])
def test_timed_kernels_are_those_of_a_step(n, tiles, precision):
    prob, U = P.random_state(len(n), n, 3, "smooth")
    s = weno.Solver(prob, precision)
    s.set_tiles(tiles)
    s.set_state(U)
    s.step(1.0)
    A, t = s.get_state()
    # the profiler may miss what runs while it starts for the first time
    step = _sweeps(lambda: s.step(1.0)) or _sweeps(lambda: s.step(1.0))
    if not step:
        pytest.skip("the profiler lists no kernels here")
    s.set_state(A, t)
    timed = _sweeps(lambda: s.time_sweeps(2))
    B, _ = s.get_state()
    assert timed == step
    assert np.array_equal(A, B)
    s.step(1.0)                       # and the next step is not disturbed
    C, tc = s.get_state()
    s.set_state(A, t)
    s.step(1.0)
    D, td = s.get_state()
    s.close()
    assert tc == td and np.array_equal(C, D)
