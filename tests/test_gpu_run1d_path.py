"""Which calls step a line in one launch, and with how many CTAs: the lengths of
tests/test_gpu_run1d.py and those below lie on both sides of these changes only
while this holds.  States are the batch kernel's bits (no tolerance)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402
from tests.test_gpu_run1d import _batch, _line  # noqa: E402


def _ctas(n, precision, splitting="llf"):
    prob, _ = P.random_state(len(n), n, 1, "smooth")
    prob["splitting"] = splitting
    s = weno.Solver(prob, precision)
    c = s.run1d_ctas()
    s.close()
    return c


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
def test_ctas_by_length(precision):
    for n, c in [(3, 1), (23, 1), (24, 2), (47, 2), (48, 4), (95, 4), (96, 8), (191, 8), (192, 16), (1000, 16)]:
        assert _ctas([n], precision) == c, n
    edge = 2032 if precision == "fp64" else 8176
    assert _ctas([edge], precision) == 16 and _ctas([edge + 1], precision) == 0


def test_what_keeps_kernels_per_step():
    assert _ctas([200], "fp64", "rf") == 16
    assert _ctas([200], "fp64", "lf") == 0
    assert _ctas([40, 30], "fp64") == 0
    assert weno.load().weno_run1d_ctas(None) == 0


@pytest.mark.parametrize("n", [2031, 2032, 2033])
def test_states_at_the_capacity_edge(n):
    prob, U = P.random_state(1, [n], 3, "mixed")
    prob["t_end"] = 0.3
    A, B = _line(prob, U, "fp64", 9, 4), _batch(prob, U, "fp64", 9)
    assert A[1:] == B[1:]
    assert np.array_equal(A[0], B[0])
