"""Host threads solving on contexts of different sizes: a solve kernel's shared-memory limit belongs
to the function and the device, so one thread's launch must not lower what another's needs.  Each
pair runs one kernel with two sizes of shared memory: cooperative launches of one slice per block
(one system) and of several (nine systems), clusters of one slice per block and of two."""
import threading

import numpy as np
import pytest

from paper_1006_0532_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1006_0532_gb300 import _binding as B  # noqa: E402


@pytest.mark.parametrize("pair", [((70, 1), (111, 9)), ((40, 1), (60, 1))], ids=["cooperative", "cluster"])
def test_threads_solve_side_by_side(pair):
    """10,100 and 25,000 nodes; 3,300 and 7,300."""
    errors, results = [], {}
    jobs = [job for job in pair for _ in range(4)]
    start = threading.Barrier(len(jobs))

    def work(job):
        try:
            rows, systems = job
            g = synth.channel_grid(2 * rows, rows + 1, seed=rows)
            c = B.Context(dict(synth.TABLE4, nu=synth.channel_nu(392.0), period_x=g.period_x, precision=0))
            c.set_grid(g)
            c.set_fields(synth.channel_fields(g, 392.0))
            src = np.cos(np.pi * g.node_xy[:, 0]) * np.cos(np.pi * g.node_xy[:, 1])
            rhs, L = np.repeat(src[:, None], 9, axis=1), np.full(g.nn, 0.1)
            zero, stream = np.zeros(g.nn), torch.cuda.Stream()
            start.wait()
            for _ in range(300):
                p, it = (c.pressure_solve(src, zero, tol=0.5, stream=stream) if systems == 1
                         else c.wp_solve(rhs, L, tol=0.5, stream=stream))
                first = results.setdefault(job, (p, it))
                assert it == first[1] and np.array_equal(p, first[0])
        except BaseException as e:   # reported by the main thread
            errors.append((job, e))

    threads = [threading.Thread(target=work, args=(job,)) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
