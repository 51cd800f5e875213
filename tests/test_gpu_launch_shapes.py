"""The advance's block size: what is reported is what is taken, a choice holds at every size, and no
result depends on it."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
def test_block_size_reported_is_taken(precision):
    g = synth.channel_grid(10, 9, seed=1)
    params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(2, 2, 2), min_per_bin=2, minnpel=0, seed=1,
                  period_x=g.period_x, precision=precision)
    states = []
    for block in (None, 128, 256):
        c = B.Context(params)
        assert c.launch_shapes()["adv_block"] == 256   # no particles yet
        c.set_grid(g)
        c.set_fields(synth.channel_fields(g, 392.0))
        c.init_particles(40)
        if block is not None:
            c.set_launch_shapes(adv_block=block)
        assert c.launch_shapes()["adv_block"] == (block or 128)   # 6,400 particles: far from eight waves
        for _ in range(5):
            c.step(1e-3)
        states.append(c.get_particles())
    for s in states[1:]:
        for k in s:
            np.testing.assert_array_equal(s[k], states[0][k])
