"""Steps recorded into a caller's graph, run as they are and replayed in turn: the states and the
statistics of the same steps run one by one."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("rows", [9, 24])      # 144 elements and 1,104
def test_captured_and_eager_steps_in_turn(rows):
    g = synth.channel_grid(rows, rows, seed=2)
    params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(2, 2, 2), min_per_bin=2, minnpel=0, seed=3,
                  period_x=g.period_x, precision=0, sort_every=0)
    outs = []
    for captured in (False, True):
        c = B.Context(params)
        c.set_grid(g)
        c.set_fields(synth.channel_fields(g, 392.0))
        c.init_particles(30)
        if captured:
            graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                c.step(1e-3, stream=stream)
            graph.replay()
            torch.cuda.synchronize()
            c.step(1e-3)
            torch.cuda.synchronize()
            graph.replay()
            graph.replay()
            torch.cuda.synchronize()
        else:
            for _ in range(4):
                c.step(1e-3)
        s = c.get_particles()
        outs.append([s[k] for k in sorted(s)] + [*c.element_stats(), c.nodal_stats()])
        assert c.check() == 0
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
