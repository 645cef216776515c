"""Recorded short characteristics on both sides of the plane sizes at which the
blocks change (128 and 256 nodes) and of where their planes need more shared memory
than the default limit (2560 nodes), against the oracle: 1e-12, the bar of both forms."""

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


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("nx,ny", [(16, 8), (43, 3), (16, 16), (37, 7), (64, 40), (51, 51), (64, 49)])
def test_blocks_by_plane_size(R, oracle_mod, nx, ny, prec):
    p = W.random_slab(nx, ny, 5, n_theta=6, n_phi=5, seed=nx, top_bc=W.BC_PLANCK)
    S = 0.5 + np.random.default_rng(7).random(p.B.shape)
    with R.Solver(p, precision=R.RT_DF64 if prec == "df64" else R.RT_FP64, fs_method=R.RT_FS_SHORT) as s:
        J, _ = s.formal_solution(S, want_lstar=False)
        assert R.rt_fs_record_info(s.ctx)[1]
    assert np.allclose(J, oracle_mod.formal_solution(p, S, method=oracle_mod.SHORT, lstar=False)[0], rtol=1e-12,
                       atol=0)
