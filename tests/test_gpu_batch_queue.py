"""The batch kernel's task queue at the sizes where it can go wrong: lines at
the edges of its tiles, one instance and more instances than CTAs, runs that
end after zero or one step, and instances above and below the others' size.
Every instance must carry the single solver's bits (no tolerance)."""
import numpy as np
import pytest

from paper_1908_02464_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1908_02464_gb300 import weno  # noqa: E402

EDGES = [3, 4, 5, 6, 57, 58, 59, 121, 122, 123, 124, 127, 128, 243, 244, 245, 249, 250, 251, 255, 256, 1000]


def _solve(prob, U, precision, steps):
    s = weno.Solver(prob, precision)
    s.set_state(U)
    s.advance(prob["t_end"], steps)
    V, t = s.get_state()
    k = s.time()[1]
    s.close()
    return V.astype(np.float64), t, k


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_lines_at_tile_edges(precision, variant):
    probs = [P.riemann_1d(n, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), 0.05) for n in EDGES]
    b = weno.Batch(EDGES, 0.0, 1.0, [0.05] * len(EDGES), precision, max_steps=7)
    b.set_config(variant)
    D = b.pack([U for _, U in probs])
    b.run(D)
    st, steps, t = b.results()
    out = b.unpack(D)
    for i, (prob, U) in enumerate(probs):
        V, ti, k = _solve(prob, U, precision, 7)
        assert st[i] == 0 and steps[i] == k and t[i] == ti, EDGES[i]
        assert np.array_equal(out[i], V), EDGES[i]
    b.close()


@pytest.mark.parametrize("count,n", [(1, 5), (1, 1900), (3000, 8)])
def test_few_and_many_instances(count, n):
    prob, U = P.riemann_1d(n, (1.0, 0.1, 1.0), (0.3, 0.0, 0.2), 0.05)
    t_end = np.where(np.arange(count) % 3 == 2, 0.0, 0.05)   # every third one has nothing to do
    b = weno.Batch([n] * count, 0.0, 1.0, t_end, "fp64")
    D = b.pack([U] * count)
    for _ in range(2):                                       # a second run starts from zeroed counters
        D.copy_(b.pack([U] * count))
        b.run(D)
        st, steps, t = b.results()
        V, ti, k = _solve(prob, U, "fp64", 10 ** 6)
        out = D.view(count, 3, n).cpu().numpy()
        done = t_end > 0
        assert np.all(st == 0) and np.all(steps[done] == k) and np.all(t[done] == ti)
        assert np.all(out[done] == V) and np.all(out[~done] == U) and np.all(steps[~done] == 0)
    b.close()


@pytest.mark.parametrize("variant", [0, 1, 2])
def test_boxes_at_tile_edges(variant):
    sizes = [(3, 3), (4, 31), (31, 4), (32, 15), (33, 16), (63, 7), (64, 8), (5, 65)]
    probs = [P.random_state(2, list(s), 40 + i, "smooth") for i, s in enumerate(sizes)]
    b = weno.Batch2D([s[0] for s in sizes], [s[1] for s in sizes], (0.0, 0.0), (1.0, 1.0), [0.02] * len(sizes), "fp64",
                     bc_lo=(2, 2), bc_hi=(2, 2), max_steps=3)
    b.set_config(variant)
    D = b.pack([U for _, U in probs])
    b.run(D)
    st, steps, t = b.results()
    out = b.unpack(D)
    for i, (prob, U) in enumerate(probs):
        prob["t_end"] = 0.02
        V, ti, k = _solve(prob, U, "fp64", 3)
        assert st[i] == 0 and steps[i] == k and t[i] == ti, sizes[i]
        assert np.array_equal(out[i], V), sizes[i]
    b.close()
