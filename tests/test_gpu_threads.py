"""Two host threads with contexts of different grids: planes of 84 and of 42 KB of
nodes, whose lists one kernel builds with more shared memory than the default
limit.  Every quadrature builds them again, both threads at the same time."""

import threading

import numpy as np
import pytest

from paper_1107_5719_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1107_5719_gb300 import build as B
    B.build()
    from paper_1107_5719_gb300 import rt3d
    rt3d.load()
    return rt3d


def test_node_lists_of_two_grids_at_once(R):
    probs = [W.random_slab(nx, ny, 2, n_theta=2, n_phi=3, seed=1) for nx, ny in ((150, 140), (105, 100))]
    together = threading.Barrier(2)
    errors = []

    def work(p):
        with R.Solver(p) as s:
            first = s.formal_solution(p.B, want_lstar=False)[0]
            for _ in range(300):
                R.rt_set_quadrature(s.ctx, p.mu, p.phi, p.w)
                together.wait()
                try:
                    if not np.array_equal(s.formal_solution(p.B, want_lstar=False)[0], first):
                        errors.append("another J")
                except R.RtError as e:
                    errors.append(str(e))

    threads = [threading.Thread(target=work, args=(p,)) for p in probs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, (len(errors), errors[0])
