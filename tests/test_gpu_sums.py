"""The two six-point sums in their integer form against exact rational sums.

Tolerances, from the form itself: the bits dropped in the alignment sum to less
than 31 x 2^-57 of the stencil's largest value (detector) and 91 x 2^-59 of its
largest product of value and coefficient (central flux), and the result is
rounded once (2^-53 of it)."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402

DETECTOR = (1, -5, 10, -10, 5, -1)
CENTRAL = (1, -8, 37, 37, -8, 1)


def _sums(x):
    return weno.weno_sums_selftest(torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()).cpu().numpy()


def _check(x):
    d, c = _sums(x)
    for i in range(len(x)):
        f = [Fraction(float(v)) for v in x[i]]
        ed, ec = (sum(k * v for k, v in zip(co, f)) for co in (DETECTOR, CENTRAL))
        big, prod = max(abs(v) for v in f), max(abs(k * v) for k, v in zip(CENTRAL, f))
        assert abs(Fraction(d[i]) - ed) <= 31 * big / 2 ** 57 + abs(ed) / 2 ** 53, (i, x[i])
        assert abs(Fraction(c[i]) - ec) <= 91 * prod / 2 ** 59 + abs(ec) / 2 ** 53, (i, x[i])


@pytest.mark.parametrize("slot", range(6))
def test_one_large_value(slot):
    """The largest value in each slot, the others 2^-4 to 2^-12 and 2^-1 to
    2^-70 of it, of one sign and of both."""
    rng = np.random.default_rng(slot)
    for lo, hi in ((4, 12), (1, 70)):
        x = rng.uniform(1, 2, (400, 6)) * 2.0 ** -rng.uniform(lo, hi, (400, 6))
        x[:, slot] = rng.uniform(1, 2, 400)
        _check(np.concatenate([x, x * rng.choice([-1, 1], (400, 6))]) * 2.0 ** rng.integers(-900, 900, (800, 1)))


def test_smooth_and_mixed_stencils():
    rng = np.random.default_rng(7)
    t = np.arange(6) - 2.5
    smooth = rng.uniform(0.5, 4, (400, 1)) + 0.02 * rng.uniform(-1, 1, (400, 1)) * t + 1e-3 * rng.uniform(-1, 1, (400, 1)) * t * t
    _check(np.concatenate([smooth, rng.uniform(-1, 1, (400, 6)), np.where(rng.random((400, 6)) < 0.5, 0.0, smooth)]))


def test_mirrored_and_negated_stencils():
    rng = np.random.default_rng(8)
    x = rng.uniform(-1, 1, (500, 6)) * 2.0 ** -rng.uniform(0, 20, (500, 6))
    d, c = _sums(x)
    dm, cm = _sums(x[:, ::-1])
    dn, cn = _sums(-x)
    assert np.array_equal(dm, -d) and np.array_equal(cm, c) and np.array_equal(dn, -d) and np.array_equal(cn, -c)


def test_ends_of_the_range():
    big, nan, inf = 2.0 ** 1023, np.nan, np.inf
    d, c = _sums(np.array([[big, 0, 0, 0, 0, 0], [0, 2.0 ** 1020, 0, 0, 0, 0], [0, 0, 2.0 ** 1017, 0, 0, 0],
                           [0, 0, big, big, 0, 0], [0, big, 0, 0, 0, 0]]))
    assert list(d[:3]) == [big, -5 * 2.0 ** 1020, 10 * 2.0 ** 1017] and d[4] == -inf
    assert list(c[:3]) == [big, -big, 37 * 2.0 ** 1017] and not np.isfinite(c[3:]).any()
    x = np.array([[inf, 1, 1, 1, 1, 1], [1, 1, 1, nan, 1, 1], [1, -inf, 1, 1, inf, 1]])
    assert not np.isfinite(_sums(x)).any()
    d, c = _sums(np.array([[0.0] * 6, [-0.0] * 6, [3.0, 0, 0, 0, 0, 0], [0, 0, 0, 7.0, 0, 0]]))
    assert list(d) == [0.0, 0.0, 3.0, -70.0] and list(c) == [0.0, 0.0, 3.0, 259.0]
