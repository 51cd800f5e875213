"""The conjugate-gradient solves at the sizes where their launch changes (csrc/k_eulerian.cu):
a cluster per component with half slices, one slice and two slices per block, the cooperative
launch with rows in shared memory, the streamed one, and rows longer than the kept entries.

A component's iteration stops at tol times its load, so two implementations' solutions differ
by at most about tol times the condition number of the Jacobi-scaled matrix, of order nn for
these two-dimensional operators: the tolerance is 4 nn tol.  Their counts differ by rounding:
two iterations, or one in a hundred.
"""
import numpy as np
import pytest

import oracle
from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402

TOL = 1e-12


def fan(k):
    """A disc of 2k triangles around one node of k neighbours and an outer ring of them."""
    a = 2 * np.pi * np.arange(k) / k
    ring = np.stack([np.cos(a), np.sin(a)], 1)
    xy = np.concatenate([[[0.0, 0.0]], ring, 2.0 * ring])
    i, j = np.arange(k), (np.arange(k) + 1) % k
    inner = np.stack([0 * i, 1 + i, 1 + j], 1)
    out1 = np.stack([1 + i, 1 + k + i, 1 + k + j], 1)
    out2 = np.stack([1 + i, 1 + k + j, 1 + j], 1)
    tri = np.concatenate([inner, out1, out2]).astype(np.int32)
    tag = np.zeros((3 * k, 3), np.int8)
    tag[k:2 * k, 0] = 2      # the edge opposite the inner vertex lies on the boundary
    return synth.Grid(xy, tri, tag, 0.0)


def grids():
    yield "fan", fan(14)
    for rows in (40, 60, 100, 185):   # 3,280, 7,320, 20,200 and 68,820 nodes
        yield "rows%d" % rows, synth.channel_grid(2 * rows, rows + 1, seed=rows)


@pytest.mark.parametrize("name,grid", list(grids()), ids=lambda v: v if isinstance(v, str) else "")
def test_solves_match_oracle_at_every_launch_shape(name, grid):
    rng = np.random.default_rng(3)
    if name == "fan":
        F = synth.uniform_fields(grid.nn, grad=rng.normal(size=6), uu=(0.5, 0.7, 0.6, 0.1, 0.05, -0.1))
        params = dict(synth.TABLE4, nu=0.01, period_x=0.0)
    else:
        F = synth.channel_fields(grid, 392.0)
        params = dict(synth.TABLE4, nu=synth.channel_nu(392.0), period_x=grid.period_x)
    F[:, 29] *= rng.uniform(0.8, 1.2, grid.nn)
    o = oracle.Oracle(grid, params, F)
    c = B.Context(dict(params, precision=0))
    c.set_grid(grid)
    c.set_fields(F)

    def close(a, b, ia, ib):
        assert abs(ia - ib) <= max(2, 0.01 * ib)
        assert np.abs(a - b).max() <= 4 * grid.nn * TOL * np.abs(b).max()

    rhs, L = o.wp_rhs()
    wo, io = o.wp_solve(rhs, L, tol=TOL)
    wg, ig = c.wp_solve(rhs, L, tol=TOL)
    close(wg, wo, ig, io)
    x, y = grid.node_xy[:, 0], grid.node_xy[:, 1]
    src = np.cos(np.pi * x) * np.cos(np.pi * y) + 0.1 * rng.normal(size=grid.nn)
    po, io = o.pressure_solve(src, np.zeros(grid.nn), tol=TOL)
    pg, ig = c.pressure_solve(src, np.zeros(grid.nn), tol=TOL)
    close(pg, po, ig, io)
    # an iteration limit that is not met is an error, and the context solves on after it
    with pytest.raises(B.PdfxError):
        c.pressure_solve(src, np.zeros(grid.nn), tol=TOL, max_iter=1)
    p2, i2 = c.pressure_solve(src, np.zeros(grid.nn), tol=TOL)
    assert i2 == ig and np.array_equal(p2, pg)
