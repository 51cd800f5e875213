"""Kernels set up while their predecessor runs: the steps give the same bits as with an event
between the stages, which keeps every stage's first kernel behind all of the stage before."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("redist,ne_rows,ppe", [(False, 5, 40), (False, 24, 130), (True, 0, 0)])
def test_chained_steps_equal_separated_stages(precision, redist, ne_rows, ppe):
    if redist:
        w = synth.redistribution_workload("redist_tiny", ratio=4)
        g, fields, params, ppe, dt = w["grid"], w["fields"], w["params"], w["ppe"], w["dt"]
    else:
        g = synth.channel_grid(2 * ne_rows, ne_rows, seed=3)
        fields, dt = synth.channel_fields(g, 392.0), 1e-3
        params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(4, 4, 4), min_per_bin=2, minnpel=ppe // 4,
                      period_x=g.period_x, seed=1, src_x=0.5, src_y=0.5, src_r=0.1, Cs=0.02, Ct=0.7)
    outs = []
    for separated in (False, True):
        c = B.Context(dict(params, precision=precision, sort_every=4))
        c.set_grid(g)
        c.set_fields(fields)
        c.set_profiling(separated)
        c.init_particles(ppe)
        for _ in range(24):
            c.step(dt)
        st = c.get_particles()
        outs.append([st[k] for k in sorted(st)] + [*c.bins(), *c.element_stats(), c.nodal_stats()])
        assert c.check() == 0
        c.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
