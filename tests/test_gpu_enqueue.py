"""Steps enqueued without a synchronizing call in between, after steps that
stopped short at their end time: the state is not in the buffer that the host
counted it to.  The same steps must give the same bits however they are
enqueued (no tolerance)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


@pytest.mark.parametrize("extra", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("dim,n,splitting,precision", [(1, [77], "llf", "fp64"), (1, [9001], "lf", "fp32"),
                                                       (2, [70, 45], "llf", "fp64"), (2, [61, 33], "lf", "mixed"),
                                                       (3, [20, 16, 14], "llf", "fp32")])
def test_enqueue_past_an_end_time_and_on(dim, n, splitting, precision, extra):
    prob, U = P.random_state(dim, n, 3, "smooth")
    prob["splitting"] = splitting
    s = weno.Solver(prob, precision)
    s.set_state(U)
    for _ in range(4):
        s.step(1.0)
    mid = s.time()[0]
    s.step(1.0)
    end = s.time()[0] + 1e-3
    runs = []
    for sync in (True, False):
        s.set_state(U)
        s.enqueue_steps(mid, 4 + extra)          # four steps, then `extra` ones that do nothing
        if sync:
            assert s.time() == (mid, 4)
        s.enqueue_steps(mid, 2)                  # nothing left to do
        if sync:
            assert s.time() == (mid, 4)
        s.enqueue_steps(end, 2)
        s.enqueue_steps(1.0, 5)
        V, t = s.get_state()
        runs.append((V, t, s.time()[1]))
    s.close()
    assert runs[0][1:] == runs[1][1:] and runs[0][2] >= 10
    assert np.array_equal(runs[0][0], runs[1][0])
