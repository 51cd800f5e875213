"""Fox's projection at the sizes where its one-group sort changes its way (one chunk, counts in
other chunks, merged runs with and without a partner) and its classes meet."""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402

SIZES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 95, 128, 160, 255, 256, 257, 288, 289, 320, 384, 511, 512, 513, 640, 767, 768,
         769]


@pytest.mark.parametrize("precision,acc64", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("fox_bins,mpb", [(16, 1), (5, 3)])
def test_order_bins_and_moments(precision, acc64, fox_bins, mpb):
    """FP64: pointers exactly the oracle's (a projected velocity's neighbours lie far more than
    its rounding apart), moments and conditional means to the form's 1e-10.  FP32: moments to
    1e-6, every bin of the size the oracle's has, and its scalar mean within the bins' exchange of
    nearly equal neighbours (one particle in a thousand)."""
    g = synth.channel_grid(20, 6, seed=9)
    params = dict(synth.workload("channel_tiny")["params"], bins=(4, 4, 4), min_per_bin=mpb, minnpel=0, cond_mode=1,
                  fox_bins=fox_bins)
    fields = synth.channel_fields(g, 392.0)
    rng = np.random.default_rng(5)
    elem = np.repeat(np.arange(g.ne, dtype=np.int32), np.resize(np.array(SIZES), g.ne))
    n = elem.size
    t = g.tri[elem]
    vel = rng.normal(size=(3, n))
    psi = rng.random(n) * (rng.random(n) < 0.5) + 0.2 * vel[0]
    psi[elem % 7 == 3] = 0.25                       # no scalar variance: all factors zero
    perm = rng.permutation(n)                       # ids in no order of the elements
    st = dict(x=g.node_xy[t[:, 0], 0], y=g.node_xy[t].mean(axis=1)[:, 1], u=vel[0], v=vel[1], w=vel[2],
              om=rng.random(n), psi=psi)
    st = {k: np.ascontiguousarray(v.astype(np.float32).astype(np.float64)[perm]) for k, v in st.items()}
    st["elem"] = np.ascontiguousarray(elem[perm])
    c = B.Context(dict(params, precision=precision, acc64=acc64))
    c.set_grid(g)
    c.set_fields(fields)
    c.set_particles(st, 0)
    assert c.check() == 0
    o = oracle.Oracle(g, params, fields)
    o.set_particles(st, 0)
    cg, co = c.get_particles()["cp"], o.get_particles()["cp"]
    vg, gg = c.bins()
    vo, go = o.bins()
    np.testing.assert_array_equal(gg, go)
    eg, eo = c.element_stats()[0], o.element_stats()[0]
    scale = np.maximum(np.abs(eo), np.sqrt(np.mean(eo * eo, axis=0, keepdims=True)) + 1e-300)
    assert np.max(np.abs(eg - eo) / scale) <= (1e-10 if precision == 0 else 1e-6)
    if precision == 0:
        np.testing.assert_array_equal(cg, co)
        assert np.max(np.abs(vg - vo)) <= 1e-10
    else:
        key = st["elem"].astype(np.int64) * 256
        np.testing.assert_array_equal(np.bincount(key + cg), np.bincount(key + co))
        same = cg == co
        assert same.mean() > 0.999
        ok = np.setdiff1d(np.arange(g.ne), st["elem"][~same])
        assert np.max(np.abs(vg[ok] - vo[ok])) <= 1e-6
