"""The forms of the conjugate-gradient solves' launch, each taken where the ones before it are left
out: the same bits and iteration counts, also where a solve goes on over several launches."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("rows", [23, 60, 100])   # 1,104, 7,320 and 20,200 nodes
def test_every_form_gives_the_same_bits(rows):
    g = synth.channel_grid(2 * rows, rows + 1, seed=rows)
    F = synth.channel_fields(g, 392.0)
    rng = np.random.default_rng(rows)
    src = np.cos(np.pi * g.node_xy[:, 0]) * np.cos(np.pi * g.node_xy[:, 1]) + 0.1 * rng.normal(size=g.nn)
    first = None
    for form in range(4):
        c = B.Context(dict(synth.TABLE4, nu=synth.channel_nu(392.0), period_x=g.period_x, precision=0))
        c.set_grid(g)
        c.set_fields(F)
        c.set_solve_form(form)
        rhs, L = c.wp_rhs()
        w, iw = c.wp_solve(rhs, L, tol=1e-10)
        p, ip = c.pressure_solve(src, np.zeros(g.nn), tol=1e-13)
        with pytest.raises(B.PdfxError):
            c.pressure_solve(src, np.zeros(g.nn), tol=1e-13, max_iter=3)
        if first is None:
            first = (w, iw, p, ip)
        assert iw == first[1] and ip == first[3]
        np.testing.assert_array_equal(w, first[0])
        np.testing.assert_array_equal(p, first[2])
    if rows == 100:
        assert first[3] > 512   # more than one launch in every form
    for bad in (-1, 4):
        with pytest.raises(B.PdfxError):
            c.set_solve_form(bad)
