"""Which calls step a line in one launch, and with how many CTAs: the lengths of
tests/test_gpu_run1d.py lie on both sides of these changes only while this
holds."""
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


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
    edge = 4080 if precision == "fp64" else 8176
    assert _ctas([edge], precision) == 16 and _ctas([edge + 1], precision) == 0


def test_what_keeps_kernels_per_step():
    assert _ctas([200], "fp64", "rf") == 16
    assert _ctas([200], "fp64", "lf") == 0
    assert _ctas([40, 30], "fp64") == 0
    assert weno.load().weno_run1d_ctas(None) == 0
