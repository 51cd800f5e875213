"""Scalar statistics of probe elements at the edges of the finishing kernel's rounds of bins:
one bin, one below, at and above a round, and the most a call may ask for."""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("nb", [1, 127, 128, 129, 300, 4096])
def test_bins_at_the_edges_of_a_round(nb):
    """Equal, bit for bit, to the same sums taken here: the library adds in fixed point
    (2^-46), so no order of additions enters, and the quotients are single roundings."""
    w = synth.workload("channel_tiny", ppe=120)
    g = w["grid"]
    o = oracle.Oracle(g, w["params"], w["fields"])
    c = B.Context(dict(w["params"], precision=0))
    c.set_grid(g)
    c.set_fields(w["fields"])
    o.init_particles(w["ppe"])
    st = o.get_particles()
    st["psi"] = np.random.default_rng(nb).beta(0.7, 1.3, st["psi"].size)
    st["psi"][st["elem"] == 5] = 0.25          # one element in a single bin
    st["elem"][st["elem"] == 7] = 8            # one element empty
    c.set_particles(st, 0)
    elems = np.random.default_rng(1).permutation(g.ne).astype(np.int32)
    got = c.scalar_stats(elems, nb)
    s, (vcce, _) = c.get_particles(), c.bins()
    for j, e in enumerate(elems):
        at = s["elem"] == e
        psi, phi = s["psi"][at], vcce[e, s["cp"][at]]
        b = np.clip(np.floor(psi * nb).astype(int), 0, nb - 1)
        count = np.bincount(b, minlength=nb)
        sc, sd = np.zeros(nb, np.int64), np.zeros(nb, np.int64)
        np.add.at(sc, b, np.rint(phi * 2.0 ** 46).astype(np.int64))
        np.add.at(sd, b, np.rint((psi - phi) * 2.0 ** 46).astype(np.int64))
        cum = (np.cumsum(sd) - sd) / 2.0 ** 46
        with np.errstate(divide="ignore", invalid="ignore"):
            want = dict(count=count, phit=(sc / 2.0 ** 46) / count, cdiff=-(sd / 2.0 ** 46) / count,
                        cdiss=-2.0 * (1.0 / nb) * (cum + 0.5 * (sd / 2.0 ** 46)) / count)
        for k, v in want.items():
            np.testing.assert_array_equal(got[k][j], np.where(count > 0, v, 0), err_msg=k)
        if at.any():
            assert got["mom"][j, 4] == psi.min() and got["mom"][j, 5] == psi.max()
        else:
            assert not got["mom"][j].any()
