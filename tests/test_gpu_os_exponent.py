"""The convergence test of the sweeps where a value crosses a power of two.

Voxels whose neighbours all have eps = 1 couple to nothing (the coefficients
carry 1 - eps), so what they start from changes neither the other voxels nor
the sweep count.  They start one ulp below 1 and end at 1: a change of 1e-16
across an exponent, in every block of the sweep kernels, beside voxels that
change by some 1e-3.  Sweeps and J are those of a start from 1."""

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


# one kernel with graphs; a graph of sweeps (above 2048 voxels per SM, 600 for
# Gauss-Seidel)
@pytest.mark.parametrize("method", [0, 1], ids=["jacobi", "gauss_seidel"])
@pytest.mark.parametrize("nx,ny,nz", [(24, 18, 7), (72, 72, 66)])
@pytest.mark.parametrize("graphs", [True, False], ids=["graphs", "host"])
def test_flip_beside_a_change(R, method, nx, ny, nz, graphs):
    p = W.random_slab(nx, ny, nz, n_theta=2, n_phi=4, seed=nx)
    rng = np.random.default_rng(nz)
    coupled = ((np.arange(nx) % 6 < 2)[None, None, :] & (np.arange(ny) % 6 < 2)[None, :, None]
               & np.ones((nz, 1, 1), bool))
    p.eps = np.where(coupled, 0.05, 1.0)
    near = np.zeros_like(coupled)
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            near |= np.roll(coupled, (dy, dx), (1, 2))
    flip = ~near
    assert flip.any(axis=2).any(axis=1).all()
    # all others stay between 1/2 and 1: at most 0.002 / eps off where they start
    J_one = np.where(flip, 1.0, 0.65 + 0.15 * rng.random(p.B.shape))
    J_fs = np.where(flip, 1.0, J_one * (1.0 + 0.002 * rng.random(p.B.shape)))
    J_ulp = np.where(flip, 1.0 - 2.0 ** -53, J_one)
    with R.Solver(p, os_method=method) as s:
        R.rt_set_graphs(s.ctx, graphs)
        s.formal_solution(p.B)              # Lambda*
        J1, n1 = s.os_step(J_fs, J_one, tol_inner=1e-12, max_sweeps=300)
        J2, n2 = s.os_step(J_fs, J_ulp, tol_inner=1e-12, max_sweeps=300)
    assert np.all(J1[flip] == 1.0) and n1 > 3
    assert np.all((J1[~flip] > 0.5) & (J1[~flip] < 1.0))
    assert n2 == n1
    assert np.array_equal(J1, J2)
