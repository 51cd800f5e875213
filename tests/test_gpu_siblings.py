"""The statistics' size classes as siblings on one stream and as branches: on either side of the
element count that chooses, every class filled, the steps give the statistics of the particles
they leave (recomputed from the states handed in afresh)."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("rows", [28, 56])      # 1,512 elements and 6,160
@pytest.mark.parametrize("precision,cond_mode", [(0, 0), (1, 0), (1, 1)])
def test_every_class_in_one_step(rows, precision, cond_mode):
    g = synth.channel_grid(28 if rows == 28 else 56, rows, seed=4)
    params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(4, 4, 4), min_per_bin=2, minnpel=0, seed=1,
                  period_x=g.period_x, precision=precision, cond_mode=cond_mode, fox_bins=16, sort_every=3)
    fields = synth.channel_fields(g, 392.0)

    def ctx():
        c = B.Context(params)
        c.set_grid(g)
        c.set_fields(fields)
        return c

    rng = np.random.default_rng(rows)
    counts = rng.choice([0, 3, 60, 255, 256, 257, 512, 513, 768, 769, 1024, 1100], size=g.ne,
                        p=[.1, .2, .3, .05, .05, .05, .05, .05, .05, .04, .03, .03])
    elem = np.repeat(np.arange(g.ne, dtype=np.int32), counts)
    n = elem.size
    cen = g.node_xy[g.tri[elem]]
    st = dict(x=cen[:, 0, 0], y=cen.mean(axis=1)[:, 1], u=rng.normal(size=n), v=rng.normal(size=n),
              w=rng.normal(size=n), om=rng.random(n) + 0.5, psi=rng.random(n) * (rng.random(n) < 0.5), elem=elem)
    st = {k: np.ascontiguousarray(v) if k == "elem" else np.ascontiguousarray(v.astype(np.float32).astype(np.float64))
          for k, v in st.items()}
    c = ctx()
    c.set_particles(st, 0)
    for _ in range(4):
        c.step(1e-6)
    s1 = c.get_particles()
    em, cnt = c.element_stats()
    v, gb = c.bins()
    nm = c.nodal_stats()
    assert c.check() == 0
    d = ctx()
    d.set_particles({k: s1[k] for k in st}, 4)
    em2, cnt2 = d.element_stats()
    v2, gb2 = d.bins()
    np.testing.assert_array_equal(cnt, cnt2)
    np.testing.assert_array_equal(cnt, np.bincount(s1["elem"], minlength=g.ne))
    np.testing.assert_array_equal(gb, gb2)
    # Fox's projection orders the particles by values that carry the moments' rounding: nearly
    # equal ones may change places, and with them their bins' means
    same = s1["cp"] == d.get_particles()["cp"]
    assert same.all() if cond_mode == 0 else same.mean() > 0.999
    ok = np.setdiff1d(np.arange(g.ne), s1["elem"][~same])
    # the same sums from the same values; the shift of the moments' sums differs (the previous
    # statistics, or none), so the forms' statistics tolerances
    tol = 1e-10 if precision == 0 else 1e-6
    for a, b in ((em, em2), (v[ok], v2[ok]), (nm, d.nodal_stats())):
        scale = np.maximum(np.abs(b), np.sqrt(np.mean(b * b, axis=0, keepdims=True)) + 1e-300)
        assert np.max(np.abs(a - b) / scale) <= tol
