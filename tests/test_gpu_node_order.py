"""The FP32 form keeps an element's nodes in the order of their ids: every one of the six orders
a triangle's nodes can have, with the periodic seam and walks across elements."""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth
from helpers import STATE_KEYS, period_diff

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("seed", [1, 2])
def test_all_orders_of_an_elements_nodes(seed):
    """One step against the FP64 oracle with the FP32 form's state tolerance (1e-5); another
    element only where the position lies within that of the edge."""
    g = synth.channel_grid(20, 9, seed=seed)
    perm = np.random.default_rng(seed).permutation(g.nn)       # old id -> new id
    xy = np.empty_like(g.node_xy)
    xy[perm] = g.node_xy
    g = synth.Grid(node_xy=xy, tri=perm[g.tri].astype(np.int32), edge_tag=g.edge_tag, period_x=g.period_x)
    assert len({tuple(r) for r in np.argsort(g.tri, axis=1)}) == 6
    fields = synth.channel_fields(g, 392.0).astype(np.float32).astype(np.float64)
    params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(4, 4, 4), min_per_bin=2, minnpel=0, seed=seed,
                  period_x=g.period_x, src_x=0.5, src_y=0.5, src_r=0.1, Cs=0.02, Ct=0.7)
    o = oracle.Oracle(g, params, fields)
    o.init_particles(60)
    st = o.get_particles()
    for k in STATE_KEYS:
        st[k] = st[k].astype(np.float32).astype(np.float64)
    o.set_particles(st, 0)
    c = B.Context(dict(params, precision=1))
    c.set_grid(g)
    c.set_fields(fields)
    c.set_particles(st, 0)
    dt = 5e-4
    o.step(dt)
    c.step(dt)
    so, sg = o.get_particles(), c.get_particles()
    assert c.diag()["hops_total"] > 100 and c.diag()["walk_fallback"] == o.diag()["walk_fallback"]
    diff = sg["elem"] != so["elem"]
    for p in np.where(diff)[0]:
        assert o.lam(sg["elem"][p], so["x"][p], so["y"][p]).min() > -1e-5
    assert diff.sum() <= 20
    for k in STATE_KEYS:
        d = np.abs(period_diff(sg[k], so[k], g.period_x)) if k == "x" else np.abs(sg[k] - so[k])
        scale = np.maximum(np.abs(so[k]), np.sqrt(np.mean(so[k] ** 2)))
        assert (d / scale)[~diff].max() <= 1e-5, k
    assert c.check() == 0
