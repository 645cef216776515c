"""Short characteristics with recorded weights against the oracle: the first
formal solution of an opacity (records), a later source and a later opacity,
Lambda* read with the recorded weights, and the unrecorded kernels
(rt_set_fs_record 0); planes of fewer than 32 and more than 256 nodes, nz = 2,
more directions than one launch takes, planes too large for shared memory, and
the boundary modes.  J and Lambda* to 1e-12, the bar of both forms (J: sums of
positive terms; double-float: 2^-48 of S per direction)."""

import numpy as np
import pytest

from paper_1107_5719_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RTOL = 1e-12


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


CASES = [
    dict(nx=5, ny=4, nz=2, seed=1, bottom_bc=W.BC_DIFFUSION, dz=0.6),
    dict(nx=3, ny=3, nz=7, seed=2, top_bc=W.BC_PLANCK),
    dict(nx=23, ny=17, nz=6, seed=3, dx=0.7, dy=1.3),
    dict(nx=6, ny=5, nz=4, seed=4, n_theta=36, n_phi=30),       # 1080 directions
    dict(nx=120, ny=110, nz=3, seed=5),                         # planes in global scratch
]


@pytest.mark.parametrize("prec", ["fp64", "df64"])
@pytest.mark.parametrize("record", [-1, 0], ids=["recorded", "plain"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "{nx}x{ny}x{nz}".format(**c))
def test_recorded_short_characteristics_match_oracle(R, oracle_mod, case, record, prec):
    kw = dict(dict(n_theta=6, n_phi=5), **case)
    p = W.random_slab(kw.pop("nx"), kw.pop("ny"), kw.pop("nz"), **kw)
    rng = np.random.default_rng(7)
    S1, S2 = 0.5 + rng.random(p.B.shape), 0.1 + 3.0 * rng.random(p.B.shape)
    chi2 = p.chi * (0.5 + rng.random(p.B.shape))
    q = W.Problem(p.nx, p.ny, p.nz, chi2, p.eps, p.B, p.mu, p.phi, p.w, dx=p.dx, dy=p.dy, dz=p.dz,
                  top_bc=p.top_bc, bottom_bc=p.bottom_bc)
    with R.Solver(p, precision=R.RT_DF64 if prec == "df64" else R.RT_FP64,
                  fs_method=R.RT_FS_SHORT, record=record) as s:
        J1, L1 = s.formal_solution(S1)
        assert R.rt_fs_record_info(s.ctx)[1] == (record != 0)
        J2, _ = s.formal_solution(S2, want_lstar=False)
        R.rt_set_opacity(s.ctx, chi2)
        J3, L3 = s.formal_solution(S2)
    for J, L, pr, S in ((J1, L1, p, S1), (J2, None, p, S2), (J3, L3, q, S2)):
        Jo, Lo = oracle_mod.formal_solution(pr, S, method=oracle_mod.SHORT, lstar=L is not None)
        assert np.allclose(J, Jo, rtol=RTOL, atol=0)
        if L is not None:
            scale = np.abs(Lo).reshape(27, -1).max(axis=0)
            assert np.all(np.abs(L - Lo).reshape(27, -1).max(axis=0) <= RTOL * scale)
