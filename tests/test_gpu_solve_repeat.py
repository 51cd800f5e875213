"""Solves in one launch, again and again: the sums are formed in a fixed order whatever the blocks'
timing, so every repeat has the first one's bits and iteration count (cooperative launch at 20,200
nodes, streamed at 68,820, cluster at 1,104)."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("rows,repeats", [(23, 20), (100, 30), (185, 20)])
def test_repeated_solves_have_equal_bits(rows, repeats):
    g = synth.channel_grid(2 * rows, rows + 1, seed=rows)
    c = B.Context(dict(synth.TABLE4, nu=synth.channel_nu(392.0), period_x=g.period_x, precision=0))
    c.set_grid(g)
    c.set_fields(synth.channel_fields(g, 392.0))
    rng = np.random.default_rng(rows)
    x, y = g.node_xy[:, 0], g.node_xy[:, 1]
    src = np.cos(np.pi * x) * np.cos(np.pi * y) + 0.1 * rng.normal(size=g.nn)
    rhs, L = rng.normal(size=(g.nn, 9)), rng.uniform(0.02, 0.3, size=g.nn)
    first = None
    for _ in range(repeats):
        w, iw = c.wp_solve(rhs, L, tol=1e-9)
        p, ip = c.pressure_solve(src, np.zeros(g.nn), tol=1e-9)
        if first is None:
            first = (w, iw, p, ip)
        assert iw == first[1] and ip == first[3]
        np.testing.assert_array_equal(w, first[0])
        np.testing.assert_array_equal(p, first[2])
