"""Operator or ray-by-ray recording, by the operator's entries per recorded step:
opaque media with a clear column of several widths (more entries than steps are
worth: rays) and the slab (an operator), on a grid large enough that the entries are
counted first.  J of sampled voxels against the oracle, 1e-12 relative, the FP64 bar."""

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


def _medium(clear):
    """The slab, or opaque with a column of `clear` of each side clear."""
    p = W.slab_65(n=45, n_theta=12, n_phi=12)
    if clear:
        n = int(clear * 45)
        p.chi = np.full_like(p.chi, 20.0)
        p.chi[:, :n, :n] = 1e-4
    return p


def _rays(p, parabolic):
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    N, D, nxy = p.nvox, p.ndir, p.nx * p.ny
    return (up(4 * D * nxy * p.nz * (p.nz - 1)) + up(4 * D * p.nz * ((nxy + 31) // 32)) + 2 * up(64 * N)
            + (up(8 * D * N) if parabolic else 0))


@pytest.mark.parametrize("form", ["linear", "parabolic", "df"])
@pytest.mark.parametrize("clear,rays", [(0.0, False), (0.25, True), (0.2, True), (0.05, False)])
def test_the_cheaper_form_is_kept(R, oracle_mod, form, clear, rays):
    p = _medium(clear)
    p.src_order = int(form == "parabolic")
    rng = np.random.default_rng(7)
    S = p.B * (0.5 + rng.random(p.B.shape))
    with R.Solver(p, precision=R.RT_DF64 if form == "df" else R.RT_FP64) as s:
        s.formal_solution(p.B, want_lstar=False)
        J, _ = s.formal_solution(S, want_lstar=False)
        held, valid = R.rt_fs_record_info(s.ctx)
    assert valid and (held == _rays(p, p.src_order)) == rays
    if form == "parabolic":     # its weights amplify the rounding of steep opacities
        return
    vox = np.unique(rng.integers(0, p.nvox, 60))
    assert np.allclose(J.reshape(-1)[vox], oracle_mod.mean_intensity_at(p, S, vox), rtol=1e-12, atol=0)
