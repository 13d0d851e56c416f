"""One-launch stepping of short 1D lines (a cluster of CTAs, each a segment)
against the batch kernel, which shares only the face routines: line lengths at
the changes of the cluster size and of the segment capacity, every boundary
condition, both splittings and precision; chunks of steps in one call and one
by one; a failing run.  The states must be the same bits (no tolerance)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


def _batch(prob, U, precision, steps):
    n = U.shape[1]
    b = weno.Batch([n], prob["lo"][0], prob["hi"][0], [prob["t_end"]], precision,
                   bc=(prob["bc_lo"][0], prob["bc_hi"][0]), max_steps=steps, splitting=weno.SPLITTINGS[prob["splitting"]],
                   hybrid=prob["hybrid"], weights=weno.WEIGHTS[prob["weights"]])
    D = b.pack([U])
    b.run(D)
    st, k, t = b.results()
    out = b.unpack(D)[0]
    b.close()
    return out, int(st[0]), int(k[0]), float(t[0])


def _line(prob, U, precision, steps, chunk=None):
    s = weno.Solver(prob, precision)
    s.set_state(U)
    done, status = 0, 0
    try:
        while done < steps:
            k = s.advance(prob["t_end"], min(chunk or steps, steps - done))
            done += k
            if k == 0:
                break
    except weno.WenoError as e:
        status = e.status
    V, t = s.get_state()
    k = s.time()[1]
    s.close()
    return V.astype(np.float64), status, k, t


LENGTHS = [3, 4, 11, 23, 24, 47, 48, 95, 96, 191, 192, 255, 1000, 4080, 4081, 8176, 8177]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("n", LENGTHS)
def test_lengths(n, precision):
    prob, U = P.random_state(1, [n], 3 + n, "mixed" if n > 20 else "smooth")
    prob["t_end"] = 0.3
    A, B = _line(prob, U, precision, 9, 4), _batch(prob, U, precision, 9)
    assert A[1:] == B[1:]
    assert np.array_equal(A[0], B[0])


@pytest.mark.parametrize("bc", [P.BC_TRANSMISSIVE, P.BC_REFLECT, P.BC_PERIODIC])
@pytest.mark.parametrize("splitting,weights,hybrid", [("llf", "reg", 1), ("rf", "reg", 1), ("llf", "wang", 2), ("rf", "is", 0)])
def test_boundaries_and_options(bc, splitting, weights, hybrid):
    prob, U = P.random_state(1, [77], 5, "mixed")
    prob.update(bc_lo=[bc], bc_hi=[bc], splitting=splitting, weights=weights, hybrid=hybrid, t_end=0.05)
    A, B = _line(prob, U, "fp64", 10 ** 6), _batch(prob, U, "fp64", 0)
    assert A[1:] == B[1:] and A[1] == 0 and A[3] == 0.05
    assert np.array_equal(A[0], B[0])


def test_inflow_and_step_by_step():
    prob, U = P.sod(130)
    prob.update(bc_lo=[P.BC_INFLOW], bc_state=[[1.0, 0.3, 2.6, 0.0, 0.0], [0.0] * 5])
    s = weno.Solver(prob, "fp64")
    s.set_state(U)
    for _ in range(12):
        s.step(prob["t_end"])
    A, ta = s.get_state()
    s.set_state(U)
    s.enqueue_steps(prob["t_end"], 5)
    s.enqueue_steps(prob["t_end"], 7)
    B, tb = s.get_state()
    assert ta == tb and np.array_equal(A, B)
    # further steps than the end time allows do nothing
    s.enqueue_steps(tb, 3)
    C, tc = s.get_state()
    s.close()
    assert tc == tb and np.array_equal(C, B)


def test_failure_keeps_the_last_good_state():
    prob, U = P.problem_123(200)
    U = U.copy()
    U[2, 90:110] *= 0.35            # almost no pressure: the run fails after some steps
    A, B = _line(prob, U, "fp64", 10 ** 6), _batch(prob, U, "fp64", 0)
    assert A[1] == weno.WENO_ERR_NONPHYSICAL
    assert A[1:] == B[1:]
    assert np.array_equal(A[0], B[0])
