"""The planes' dispatch order on both sides of the number of planes that one block
ranks (64), of a block of the kernels above it (32 planes) and on a tall grid: the
ranks of the estimate by decreasing work, ties by index, restated on the host."""

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


def _work(mean, dz):
    nz = len(mean)
    work = np.zeros(nz, int)
    for amu in (1.0, 0.5, 0.2):
        hs = dz / (2.0 * amu)
        for s in (1, -1):
            for k0 in range(nz):
                tau, n, k = 0.0, 1, k0
                while 0 <= k - s < nz and tau <= 40.0:
                    tau += hs * (mean[k] + mean[k - s])
                    k -= s
                    n += 1
                work[k0] += n
    return work


@pytest.mark.parametrize("nz", [2, 63, 64, 65, 96, 97, 129, 700])
def test_order_is_the_rank_of_the_estimate(R, nz):
    p = W.random_slab(3, 4, nz, n_theta=2, n_phi=2, seed=nz)
    # one value per plane, powers of two: means and depths are exact
    p.chi = np.broadcast_to(2.0 ** np.random.default_rng(nz).integers(-6, 7, nz)[:, None, None],
                            p.chi.shape).copy()
    ctx = R.rt_create(0, R.RT_FP64)
    try:
        R.rt_set_grid(ctx, p.nx, p.ny, p.nz, 1.0, 1.0, 1.0)
        R.rt_set_opacity(ctx, p.chi)
        order = R.rt_get_plane_order(ctx, nz)
    finally:
        R.rt_destroy(ctx)
    work = _work(p.chi[:, 0, 0], 1.0)
    assert order.tolist() == sorted(range(nz), key=lambda k: (-work[k], k))
