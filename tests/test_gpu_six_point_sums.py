"""The FP64 six-point sums on the integer pipes (grids of 32768 cells and
more): against the oracle where alignment and rounding can go wrong, and the
batches on the same side of the size rule as the grid solver.

Tolerance of the comparison with the oracle: both sides form each face flux
(times 60) from sums of six terms with coefficients up to 37, so they differ
by at most a few hundred units of 2^-53 of the largest flux of the stencil;
1e-12 of max |F| / dx leaves a factor of about ten."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


def _state(kind, nx, ny):
    """A 2D periodic state whose stencils test the alignment of exponents."""
    prob, _ = P.random_state(2, [8, 8], 1, "smooth")
    prob["n"] = [nx, ny]
    x = P.centers(0, 1, nx)[None, :]
    y = P.centers(0, 1, ny)[:, None]
    one = np.ones((ny, nx))
    s = np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    rho, u, v, p = one, 0.3 * one, 0.1 * one, one
    if kind == "powers":            # values on both sides of powers of two, sign changes
        rho, u, v, p = 1 + 0.02 * s, 0.5 * s, np.sin(4 * np.pi * (x + y)), 1.6 + 0.3 * s
    elif kind == "zero":            # exactly zero momenta beside non-zero ones
        u = np.where(s > 0, s * s, 0.0) * one
        v = 0.0 * one
    elif kind == "range":           # factors of a million from cell to cell
        rho = np.where((x > 0.3) & (x < 0.6), 1e3, 1e-3) * one
        p = np.where((y > 0.2) & (y < 0.7), 1e4, 1e-2) * one
        u = v = 0.0 * one
    elif kind == "tiny":            # a transverse momentum far below the others
        u, v = 0.2 * s, 1e-200 * s
        rho = 1 + 0.1 * s
    return prob, P.prim_to_cons(prob["gamma"], rho * one, [u * one, v * one], p * one)


@pytest.mark.parametrize("kind", ["powers", "zero", "range", "tiny", "constant"])
@pytest.mark.parametrize("nx,ny", [(256, 128), (331, 99)])
def test_rhs_against_the_oracle(kind, nx, ny):
    prob, U = _state(kind, nx, ny)
    s = weno.Solver(prob, "fp64")
    R = s.rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    s.close()
    O = orc.rhs(prob, U)
    if kind == "constant":
        assert np.all(R == 0.0)
        return
    g = prob["gamma"]
    u, v = U[1] / U[0], U[2] / U[0]
    p = (g - 1) * (U[3] - 0.5 * U[0] * (u * u + v * v))
    c = np.sqrt(g * p / U[0])
    speed = np.abs(u) + np.abs(v) + c
    for k in range(4):
        flux = np.max(speed * np.abs(U[k])) + np.max(p * (np.abs(u) + np.abs(v) + (k in (1, 2))))
        scale = flux * max(nx, ny)
        assert np.max(np.abs(R[k] - O[k])) <= 1e-12 * scale + 1e-300, k


def test_non_finite_input_gives_non_finite_output():
    prob, U = _state("powers", 256, 128)
    for bad in (np.nan, np.inf):
        V = U.copy()
        V[0, 40, 50] = bad
        s = weno.Solver(prob, "fp64")
        R = s.rhs(torch.from_numpy(V).cuda()).cpu().numpy()
        s.close()
        assert not np.isfinite(R[:, 40, 50]).all()
        far = np.ones(U.shape[1:], bool)
        far[34:47, :] = False
        far[:, 44:57] = False
        assert np.isfinite(R[:, far]).all()


@pytest.mark.parametrize("nx,ny", [(182, 180), (182, 181)])   # 32760 and 32942 cells: both sides of the rule
def test_2d_batch_takes_the_grid_solvers_form(nx, ny):
    prob, U = P.random_state(2, [nx, ny], 7, "mixed")
    s = weno.Solver(prob, "fp64")
    s.set_state(U)
    s.advance(1.0, 3)
    A, _ = s.get_state()
    s.close()
    b = weno.Batch2D([40, nx], [30, ny], (0.0, 0.0), (1.0, 1.0), [1.0, 1.0], "fp64", bc_lo=(2, 2), bc_hi=(2, 2),
                     max_steps=3)
    other = P.random_state(2, [40, 30], 8, "mixed")[1]
    D = b.pack([other, U])
    b.run(D)
    assert np.array_equal(b.unpack(D)[1], A)
    b.close()


def test_1d_batch_takes_the_grid_solvers_form():
    n = 32768
    prob, U = P.random_state(1, [n], 5, "mixed")
    s = weno.Solver(prob, "fp64")
    s.set_state(U)
    s.advance(1.0, 2)
    A, _ = s.get_state()
    s.close()
    b = weno.Batch([100, n], 0.0, 1.0, [1.0, 1.0], "fp64", bc=(2, 2), max_steps=2)
    D = b.pack([P.random_state(1, [100], 6, "mixed")[1], U])
    b.run(D)
    assert np.array_equal(b.unpack(D)[1], A)
    b.close()
