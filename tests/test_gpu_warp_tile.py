"""The binning's warp tiles, and the one launch of a small grid, at the sizes, bin shapes and values where their sort could go wrong:
empty elements, one word more or less than a register column, mapped values that collide, runs
of equal velocities ordered by particle id, signed zeros and a wide range of magnitudes."""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402

SIZES = [0, 1, 2, 3, 7, 31, 32, 33, 63, 64, 65, 100, 127, 128, 129, 191, 192, 255, 256, 257, 300, 383, 511, 512, 513, 600,
         767, 768, 769]


def _state(g, values, seed):
    rng = np.random.default_rng(seed)
    counts = np.resize(np.array(SIZES), g.ne)
    elem = np.repeat(np.arange(g.ne, dtype=np.int32), counts)
    n = elem.size
    t = g.tri[elem]
    x = g.node_xy[t[:, 0], 0]
    y = g.node_xy[t].mean(axis=1)[:, 1]
    if values == "spread":
        vel = rng.normal(size=(3, n))
    elif values == "few":          # a handful of values: long runs of equals
        vel = rng.integers(-2, 3, size=(3, n)) * 0.25
        vel[rng.random((3, n)) < 0.1] = -0.0
    elif values == "equal":
        vel = np.full((3, n), 0.5)
    else:                          # one outlier sets the scale, the others nearly coincide
        vel = 1.0 + 1e-6 * rng.normal(size=(3, n))
        vel[:, ::97] = 1e6 * rng.normal(size=(3, vel[:, ::97].shape[1]))
    vel = vel.astype(np.float32).astype(np.float64)
    psi = (rng.random(n) * (rng.random(n) < 0.5)).astype(np.float32).astype(np.float64)
    perm = rng.permutation(n)      # ids in no order of the elements
    st = dict(x=x, y=y, u=vel[0], v=vel[1], w=vel[2], om=rng.random(n), psi=psi)
    return {k: np.ascontiguousarray(v[perm]) for k, v in st.items()} | {"elem": np.ascontiguousarray(elem[perm])}


@pytest.mark.parametrize("rows", [5, 18])    # 64 elements (one launch) and 680 (size classes)
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("values", ["spread", "few", "equal", "wide"])
@pytest.mark.parametrize("bins,mpb", [((4, 4, 4), 2), ((1, 1, 1), 1), ((16, 1, 1), 1), ((1, 4, 1), 3), ((2, 3, 5), 1),
                                      ((16, 16, 1), 1), ((1, 1, 7), 2)])
def test_order_bins_and_pointers_are_the_oracles(rows, precision, values, bins, mpb):
    """Pointers and effective bins exactly, conditional means and moments within the form's
    tolerance, for both size-class splits (which agree bit for bit)."""
    w = synth.workload("channel_tiny")
    g = w["grid"] if rows == 5 else synth.channel_grid(20, rows, seed=9)
    w["fields"] = synth.channel_fields(g, 392.0)
    params = dict(w["params"], bins=bins, min_per_bin=mpb, minnpel=0)
    st = _state(g, values, 5)
    outs = []
    for split in (256, 0):
        c = B.Context(dict(params, precision=precision))
        c.set_grid(g)
        c.set_fields(w["fields"])
        c.set_launch_shapes(tile_split=split)
        c.set_particles(st, 0)
        outs.append((c.get_particles()["cp"], *c.bins(), c.element_stats()[0]))
        assert c.check() == 0
        c.close()
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
    o = oracle.Oracle(g, params, w["fields"])
    o.set_particles(st, 0)
    cp, vcce, gbin, em = outs[0]
    np.testing.assert_array_equal(cp, o.get_particles()["cp"])
    vo, go = o.bins()
    np.testing.assert_array_equal(gbin, go)
    tol = 1e-10 if precision == 0 else 1e-6   # the forms' statistics tolerances
    assert np.max(np.abs(vcce - vo)) <= tol
    eo = o.element_stats()[0]
    for k in (0, 1, 2, 3, 10, 11):
        scale = max(float(np.abs(st["uvw"[k - 1]]).max()) if 1 <= k <= 3 else 1.0, 1.0)
        assert np.max(np.abs(em[:, k] - eo[:, k])) <= tol * scale, k
