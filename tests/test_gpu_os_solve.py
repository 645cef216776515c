"""The operator-splitting solve as one kernel against the host-driven sweeps:
same sweep counts and bit-identical J on both sides of the sizes at which it
changes its form (coefficients in shared memory up to 256 voxels per SM, one or
two voxels per thread, Gauss-Seidel up to 600 voxels per SM), on ragged grids
and grids with fewer voxels than a warp."""

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


@pytest.mark.parametrize("method", [0, 1], ids=["jacobi", "gauss_seidel"])
@pytest.mark.parametrize("nx,ny,nz", [(3, 3, 2), (3, 4, 5), (5, 7, 139), (32, 32, 38), (33, 32, 37), (31, 45, 28),
                                      (61, 45, 34), (53, 54, 55)])
@pytest.mark.parametrize("tol,max_sweeps", [(0.0, 1), (1e-12, 300), (3e-40, 6), (1e40, 6)])
def test_one_kernel_equals_host_loop(R, method, nx, ny, nz, tol, max_sweeps):
    p = W.random_slab(nx, ny, nz, n_theta=2, n_phi=4, seed=nx + ny + nz, eps_range=(1e-3, 1.0))
    out = {}
    for graphs in (True, False):
        with R.Solver(p, os_method=method) as s:
            R.rt_set_graphs(s.ctx, graphs)
            Jfs, _ = s.formal_solution(p.B)
            out[graphs] = s.os_step(Jfs, p.B, tol_inner=tol, max_sweeps=max_sweeps)
    assert out[True][1] == out[False][1]
    assert np.array_equal(out[True][0], out[False][0])


@pytest.mark.parametrize("method", [0, 1], ids=["jacobi", "gauss_seidel"])
def test_solves_of_different_lengths_in_turn(R, method):
    """The barrier words of a solve are those that the one before it zeroed:
    fewer and more sweeps in turn, and more than the words held at first."""
    p = W.random_slab(7, 6, 8, n_theta=2, n_phi=4, seed=3, eps_range=(1e-3, 1.0))
    runs = [(0.0, 3), (0.0, 40), (1e-12, 300), (0.0, 1), (0.0, 2600), (0.0, 5), (1e-6, 50), (0.0, 1100)]
    out = {}
    for graphs in (True, False):
        with R.Solver(p, os_method=method) as s:
            R.rt_set_graphs(s.ctx, graphs)
            Jfs, _ = s.formal_solution(p.B)
            out[graphs] = [s.os_step(Jfs, p.B, tol_inner=t, max_sweeps=m) for t, m in runs]
    for (Jg, ng), (Jh, nh) in zip(out[True], out[False]):
        assert ng == nh
        assert np.array_equal(Jg, Jh)
