"""Time bookkeeping of the grid solver, whose last sweep takes the wave speeds
of the next step: calls split in every way, a target time changed between
calls, a new state, a measurement in between, and a state that fails.  The
same steps must give the same bits however they are called (no tolerance)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


def _problem(dim, splitting):
    n = {1: [9000], 2: [70, 45], 3: [20, 16, 14]}[dim]   # 1D: beyond the one-launch lines
    prob, U = P.random_state(dim, n, 3, "smooth" if dim == 3 else "mixed")
    prob["splitting"] = splitting
    return prob, U


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("dim,splitting", [(1, "llf"), (1, "lf"), (2, "llf"), (2, "lf"), (3, "llf"), (3, "lf")])
def test_calls_split_in_every_way(dim, splitting, precision):
    prob, U = _problem(dim, splitting)
    s = weno.Solver(prob, precision)
    s.set_state(U)
    for _ in range(7):
        s.step(1.0)
    A, ta = s.get_state()
    s.set_state(U)
    assert s.advance(1.0, 3) == 3
    s.time_sweeps(1)
    s.totals()
    s.enqueue_steps(1.0, 2)
    s.step(1.0)
    assert s.advance(1.0, 1) == 1
    B, tb = s.get_state()
    assert ta == tb and np.array_equal(A, B)
    # the end time reached exactly, then moved on
    mid = 0.6 * ta
    s.set_state(U)
    s.advance(mid)
    C, tc = s.get_state()
    assert tc == mid
    s.enqueue_steps(mid, 2)                       # nothing left to do
    D, td = s.get_state()
    assert td == mid and np.array_equal(C, D)
    s.advance(ta)
    E, te = s.get_state()
    fresh = weno.Solver(prob, precision)
    fresh.set_state(C, mid)
    fresh.advance(ta)
    F, tf = fresh.get_state()
    assert te == tf == ta and np.array_equal(E, F)
    s.close()
    fresh.close()


def test_steps_and_time_are_the_oracles():
    prob, U = _problem(2, "llf")
    s = weno.Solver(prob, "fp64")
    s.set_state(U)
    s.advance(1.0, 6)
    V, t = s.get_state()
    s.close()
    W = U.copy()
    st, to, k = orc.advance(prob, W, 0.0, 1.0, max_steps=6)
    assert st == 0 and k == 6 and abs(t - to) <= 6e-15 * to


@pytest.mark.parametrize("how", ["step", "advance", "enqueue"])
def test_an_inadmissible_state_fails_the_first_step(how):
    prob, U = P.random_state(2, [40, 30], 3, "smooth")
    U = U.copy()
    U[3, 10, 10] = -1.0
    s = weno.Solver(prob, "fp64")
    s.set_state(U)
    with pytest.raises(weno.WenoError) as e:
        if how == "step":
            s.step(1.0)
        else:
            if how == "enqueue":
                s.enqueue_steps(1.0, 2)
            s.advance(1.0, 3)
    assert e.value.status == weno.WENO_ERR_NONPHYSICAL
    V, t = s.get_state()
    assert t == 0.0 and s.time()[1] == 0 and np.array_equal(V, U)
    good = P.random_state(2, [40, 30], 3, "smooth")[1]
    s.set_state(good)                             # a new state clears the failure
    assert s.advance(1.0, 2) == 2
    s.close()
