"""The batch kernel's waits: launches with fewer and with more CTAs than the
GPU holds at once (the others start when some have left, as they do beside
another stream's kernels), and waits that run out.  Every instance must carry the single solver's bits
(no tolerance)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402


def _line_batch(count, precision="fp64", t_end=0.02):
    n = [40 + 17 * (i % 60) for i in range(count)]
    states = [P.riemann_1d(k, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), t_end) for k in n]
    b = weno.Batch(n, 0.0, 1.0, [t_end] * count, precision, max_steps=12)
    return b, [U for _, U in states], states


def _run(b, states):
    D = b.pack(states)
    b.run(D)
    st, steps, t = b.results()
    return D.cpu().numpy(), st, steps, t


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ctas", [1, 3, 20000])
def test_lines_with_any_number_of_ctas(ctas, precision):
    b, states, probs = _line_batch(240, precision)
    A = _run(b, states)
    b.set_launch(ctas)
    B = _run(b, states)
    b.set_launch(0)
    C = _run(b, states)
    for x, y, z in zip(A, B, C):
        assert np.array_equal(x, y) and np.array_equal(x, z)
    assert np.all(A[1] == 0) and np.all(A[2] > 0)
    prob, U = probs[137]
    s = weno.Solver(prob, precision)
    s.set_state(U)
    s.advance(0.02, 12)
    V, _ = s.get_state()
    s.close()
    o = b.offsets
    assert np.array_equal(B[0][o[137]:o[138]].reshape(3, -1), V)
    b.close()


@pytest.mark.parametrize("ctas", [1, 20000])
def test_boxes_with_any_number_of_ctas(ctas):
    nx = [10 + 7 * (i % 9) for i in range(60)]
    ny = [9 + 5 * (i % 11) for i in range(60)]
    states = [P.random_state(2, [a, b], 70 + i, "smooth")[1] for i, (a, b) in enumerate(zip(nx, ny))]
    b = weno.Batch2D(nx, ny, (0.0, 0.0), (1.0, 1.0), [0.02] * 60, "fp64", bc_lo=(2, 2), bc_hi=(2, 2), max_steps=4)
    A = _run(b, states)
    b.set_launch(ctas)
    B = _run(b, states)
    for x, y in zip(A, B):
        assert np.array_equal(x, y)
    assert np.all(A[1] == 0) and np.all(A[2] > 0)
    b.close()


def test_a_negative_number_of_ctas_is_refused():
    b, _, _ = _line_batch(2)
    with pytest.raises(weno.WenoError) as e:
        b.set_launch(-1)
    assert e.value.status == weno.WENO_ERR_INVALID_ARG
    b.close()


@pytest.mark.parametrize("dim", [1, 2])
def test_a_wait_that_runs_out_is_reported_and_the_next_run_is_good(dim):
    """One instance of many tiles: one CTA prepares it for hundreds of
    microseconds while the others give up after a few polls."""
    if dim == 1:
        prob, U = P.riemann_1d(20000, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), 0.02)
        make = lambda: weno.Batch([20000], 0.0, 1.0, [0.02], "fp64", max_steps=3)
    else:
        prob, U = P.random_state(2, [200, 190], 9, "smooth")
        make = lambda: weno.Batch2D([200], [190], (0.0, 0.0), (1.0, 1.0), [0.02], "fp64", bc_lo=(2, 2), bc_hi=(2, 2),
                                    max_steps=3)
    b, fresh = make(), make()
    good = _run(fresh, [U])
    assert good[2][0] == 3
    b.set_wait(1)
    D = b.pack([U])
    b.run(D)
    with pytest.raises(weno.WenoError) as e:
        b.results()
    assert e.value.status == weno.WENO_ERR_TIMEOUT
    b.set_wait(0)
    for x, y in zip(_run(b, [U]), good):
        assert np.array_equal(x, y)
    with pytest.raises(weno.WenoError) as e:
        b.set_wait(-1)
    assert e.value.status == weno.WENO_ERR_INVALID_ARG
    b.close()
    fresh.close()


def test_a_long_sweep_of_one_cta_is_progress():
    """400000 cells beside thousands of short lines: every CTA has work when
    the long line's first sweep begins, so one CTA takes it whole (some tens of
    milliseconds) and the others wait for much longer than their polls."""
    n = [400000] + [100] * 4000
    b = weno.Batch(n, 0.0, 1.0, [1e-9] + [0.2] * 4000, "fp64")
    long_U = P.riemann_1d(400000, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), 0.2)[1]
    U = P.riemann_1d(100, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), 0.2)[1]
    states = [long_U] + [U] * 4000
    b.set_wait(10000)
    A = _run(b, states)
    assert np.all(A[1] == 0) and A[2][0] == 1 and np.all(A[2][1:] == A[2][1])
    b.set_wait(0)
    B = _run(b, states)
    for x, y in zip(A, B):
        assert np.array_equal(x, y)
    b.close()


def test_boxes_fit_without_room_for_their_primitives():
    """200 FP64 boxes whose work arrays fit the free memory (105 of 150 MB) and
    whose cell primitives (52 MB) do not."""
    n = [64] * 200
    states = [P.random_state(2, [64, 64], 30 + i % 3, "smooth")[1] for i in range(200)]
    make = lambda: weno.Batch2D(n, n, (0.0, 0.0), (1.0, 1.0), [0.02] * 200, "fp64", bc_lo=(2, 2), bc_hi=(2, 2),
                                max_steps=3)
    b = make()
    A = _run(b, states)                            # also loads the kernel
    b.close()
    D = b.pack(states)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - (150 << 20), dtype=torch.uint8, device="cuda")
    try:
        c = make()
        c.run(D)
        st, steps, t = c.results()
        c.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    for x, y in zip(A, (D.cpu().numpy(), st, steps, t)):
        assert np.array_equal(x, y)
