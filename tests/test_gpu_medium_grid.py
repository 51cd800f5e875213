"""The statistics of a medium grid in one launch: the same elements' bits as on a grid of a few hundred
elements, which takes another launch, in every size class and at the classes' edges."""
import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402

SIZES = [0, 1, 3, 60, 255, 256, 257, 512, 513, 768, 769, 1024, 1100]
SHARE = [.09, .01, .2, .35, .07, .07, .05, .04, .03, .03, .02, .02, .02]


def grid_of(rows, minimum):
    g = synth.channel_grid(rows, rows, seed=6)
    assert g.ne >= minimum
    return g


@pytest.mark.parametrize("split", [256, 0, 100])
@pytest.mark.parametrize("rows", [19, 29, 51])      # 684 elements, 1,624 and 5,100
def test_medium_grid_equals_small_grid(rows, split):
    few = grid_of(16, 480)
    many = grid_of(rows, 609)
    rng = np.random.default_rng(rows + split)
    counts = rng.choice(SIZES, size=many.ne, p=SHARE)
    assert counts.mean() < 208
    for size in SIZES:
        counts[size % few.ne] = size                # every class on the elements that both grids have
    outs = []
    for g in (few, many):
        elem = np.repeat(np.arange(g.ne, dtype=np.int32), counts[:g.ne])
        total = int(counts.sum())
        draw = np.random.default_rng(split)
        cols = {k: draw.normal(size=total).astype(np.float32).astype(np.float64) for k in ("u", "v", "w")}
        cols["u"][::3] = 0.5                         # equal values: the order goes through the ids
        cols["om"] = (draw.random(total) + 0.5).astype(np.float32).astype(np.float64)
        cols["psi"] = (draw.random(total) * (draw.random(total) < 0.5)).astype(np.float32).astype(np.float64)
        n = elem.size
        cen = g.node_xy[g.tri[elem]].mean(axis=1)
        st = dict(x=np.ascontiguousarray(cen[:, 0]), y=np.ascontiguousarray(cen[:, 1]), elem=elem,
                  **{k: np.ascontiguousarray(v[:n]) for k, v in cols.items()})
        c = B.Context(dict(synth.TABLE4, nu=synth.channel_nu(392.0), bins=(4, 4, 4), min_per_bin=2, minnpel=0, seed=1,
                           period_x=g.period_x, precision=1))
        c.set_grid(g)
        c.set_fields(synth.channel_fields(g, 392.0))
        c.set_launch_shapes(tile_split=split)
        c.set_particles(st, 0)
        assert c.check() == 0
        em, cnt = c.element_stats()
        v, gb = c.bins()
        m = few.ne
        outs.append((em[:m], cnt[:m], v[:m], gb[:m], c.get_particles()["cp"][:int(counts[:m].sum())]))
    np.testing.assert_array_equal(outs[0][1], counts[:few.ne])
    for a, b in zip(*outs):
        np.testing.assert_array_equal(a, b)
