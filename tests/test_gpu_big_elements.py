"""Elements above the tiles' 1,024 particles: the block sort's passes at and around powers of two,
with either number of threads (the mean count chooses)."""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("sizes", [[1025, 40, 2047, 0, 2048, 2049, 3001, 4096], [1025, 0, 0, 0, 0, 0, 0, 3, 0, 1500]])
def test_order_bins_and_moments(precision, sizes):
    """Pointers exactly the oracle's, conditional means and moments to the forms' tolerances, with
    runs of equal velocities ordered by particle id."""
    g = synth.channel_grid(20, 5, seed=9)
    params = dict(synth.workload("channel_tiny")["params"], bins=(4, 4, 4), min_per_bin=2, minnpel=0)
    fields = synth.channel_fields(g, 392.0)
    rng = np.random.default_rng(3)
    elem = np.repeat(np.arange(g.ne, dtype=np.int32), np.resize(np.array(sizes), g.ne))
    n = elem.size
    vel = rng.normal(size=(3, n))
    vel[:, ::5] = np.round(vel[:, ::5])
    t = g.tri[elem]
    perm = rng.permutation(n)
    st = dict(x=g.node_xy[t[:, 0], 0], y=g.node_xy[t].mean(axis=1)[:, 1], u=vel[0], v=vel[1], w=vel[2],
              om=rng.random(n), psi=rng.random(n) * (rng.random(n) < 0.5))
    st = {k: np.ascontiguousarray(v.astype(np.float32).astype(np.float64)[perm]) for k, v in st.items()}
    st["elem"] = np.ascontiguousarray(elem[perm])
    c = B.Context(dict(params, precision=precision))
    c.set_grid(g)
    c.set_fields(fields)
    c.set_particles(st, 0)
    assert c.check() == 0
    o = oracle.Oracle(g, params, fields)
    o.set_particles(st, 0)
    np.testing.assert_array_equal(c.get_particles()["cp"], o.get_particles()["cp"])
    vg, gg = c.bins()
    vo, go = o.bins()
    np.testing.assert_array_equal(gg, go)
    tol = 1e-10 if precision == 0 else 1e-6
    assert np.max(np.abs(vg - vo)) <= tol
    eg, eo = c.element_stats()[0], o.element_stats()[0]
    scale = np.maximum(np.abs(eo), np.sqrt(np.mean(eo * eo, axis=0, keepdims=True)) + 1e-300)
    assert np.max(np.abs(eg - eo) / scale) <= tol
