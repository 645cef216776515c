"""The recorded formal solution as an assembled operator, against the oracle
at the sizes where its tables can go wrong: planes of fewer and of just over
32 voxels, one and several tiles, nx = 3 (neighbours alias across the seam),
nz = 2, all directions of one sign, one direction, and grids large enough
that the operator's size is read back and its planes recorded in chunks;
Lambda* read off it against the Lambda* kernel; and the ray-by-ray recording
where the budget holds no operator.  J to 1e-12 relative, the FP64 bar: the
sums have a few thousand positive terms of relative error ~1e-16."""

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


def _one_sided(nx, ny, nz, sign, n):
    """n directions of one sign (weights sum to 1)."""
    p = W.random_slab(nx, ny, nz, seed=41)
    rng = np.random.default_rng(n)
    p.mu = sign * (0.1 + 0.9 * rng.random(n))
    p.phi = 6.28 * rng.random(n)
    p.w = np.full(n, 1.0 / n)
    return p


PROBLEMS = {
    "3x3x5": lambda: W.random_slab(3, 3, 5, n_theta=4, n_phi=5, seed=1),
    "3x11x4-33": lambda: W.random_slab(3, 11, 4, n_theta=4, n_phi=5, seed=2, bottom_bc=W.BC_DIFFUSION),
    "8x4x7-32": lambda: W.random_slab(8, 4, 7, n_theta=6, n_phi=7, seed=3),
    "19x13x2": lambda: W.random_slab(19, 13, 2, n_theta=6, n_phi=5, seed=4, top_bc=W.BC_PLANCK),
    "up-only": lambda: _one_sided(7, 6, 9, -1.0, 5),
    "down-only": lambda: _one_sided(5, 7, 6, 1.0, 1),
    "opaque": lambda: W.random_slab(9, 8, 12, n_theta=8, n_phi=9, seed=6, chi_decades=6.0),
}


FORMS = ["linear", "parabolic", "df"]


def _form(R, form):
    return (1 if form == "parabolic" else 0, R.RT_DF64 if form == "df" else R.RT_FP64)


@pytest.mark.parametrize("form", ["linear", "df"])
@pytest.mark.parametrize("nz", [127, 128, 129, 257])
def test_tall_grids_match_oracle(R, oracle_mod, nz, form):
    """The kernels that share planes, distances and directions among lanes:
    planes on both sides of one round of the plane order (128), more slots
    than a block has warps, 35 directions of a sign (more than 32 lanes)."""
    p = W.random_slab(3, 4, nz, n_theta=10, n_phi=7, seed=nz)
    _, prec = _form(R, form)
    S = 0.5 + np.random.default_rng(6).random(p.B.shape)
    J0 = oracle_mod.formal_solution(p, S)[0]
    for record in (-1, 0):
        with R.Solver(p, precision=prec, record=record) as s:
            J, _ = s.formal_solution(S, want_lstar=False)
            assert R.rt_fs_record_info(s.ctx)[1] == (record != 0)
        assert np.allclose(J, J0, rtol=RTOL, atol=0)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("name", PROBLEMS)
def test_operator_matches_oracle(R, oracle_mod, name, form):
    p = PROBLEMS[name]()
    p.src_order, prec = _form(R, form)
    if form == "parabolic" and name == "opaque":
        pytest.skip("the parabolic weights amplify rounding over six decades per voxel")
    rng = np.random.default_rng(5)
    S1, S2 = 0.5 + rng.random(p.B.shape), 0.1 + 4.0 * rng.random(p.B.shape)
    with R.Solver(p, precision=prec) as s:
        J1, L = s.formal_solution(S1)
        J2, _ = s.formal_solution(S2, want_lstar=False)
        assert R.rt_fs_record_info(s.ctx)[1]
    with R.Solver(p, precision=prec, record=0) as s:
        _, Lk = s.formal_solution(S1)
    assert np.allclose(J1, oracle_mod.formal_solution(p, S1)[0], rtol=RTOL, atol=0)
    assert np.allclose(J2, oracle_mod.formal_solution(p, S2)[0], rtol=RTOL, atol=0)
    # double-float entries: 2^-48 per coefficient and per sum
    assert np.max(np.abs(L - Lk)) <= (1e-13 if form == "df" else 1e-14) * np.abs(Lk).max()


@pytest.mark.parametrize("form", ["linear", "df"])
def test_source_of_zeros_records_whole_rays(R, oracle_mod, form):
    """A recording made from S = 0 with zero boundaries (no intensity to
    measure the cutoff by) serves later sources."""
    p = W.random_slab(9, 7, 8, n_theta=4, n_phi=6, seed=8, bottom_bc=W.BC_ZERO)
    with R.Solver(p, precision=_form(R, form)[1]) as s:
        J0, _ = s.formal_solution(np.zeros(p.B.shape), want_lstar=False)
        J, _ = s.formal_solution(p.B, want_lstar=False)
    assert np.all(J0 == 0.0)
    assert np.allclose(J, oracle_mod.formal_solution(p, p.B)[0], rtol=RTOL, atol=0)


@pytest.mark.parametrize("form", FORMS)
def test_ray_by_ray_where_the_operator_does_not_fit(R, oracle_mod, form):
    """A budget of exactly the ray-by-ray recording, on a transparent slab
    whose operator is larger: the recording is kept ray by ray."""
    p = W.random_slab(16, 16, 6, n_theta=4, n_phi=4, seed=9, chi_decades=1.0)
    p.chi *= 1e-3
    p.src_order, prec = _form(R, form)
    N, D, nxy = p.nvox, p.ndir, p.nx * p.ny
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    need = (up(8 * D * nxy * p.nz * (p.nz - 1) // 2) + up(4 * D * p.nz * ((nxy + 31) // 32))
            + 2 * up(64 * N) + (up(8 * D * N) if p.src_order else 0))
    S1, S2 = p.B, p.B * np.random.default_rng(2).random(p.B.shape)
    with R.Solver(p, precision=prec, record=need) as s:
        J1, _ = s.formal_solution(S1, want_lstar=False)
        assert R.rt_fs_record_info(s.ctx) == (need, True)
        J2, _ = s.formal_solution(S2, want_lstar=False)
    with R.Solver(p, precision=prec, record=need - 1) as s:
        s.formal_solution(S1, want_lstar=False)
        assert R.rt_fs_record_info(s.ctx) == (0, False)
    assert np.allclose(J1, oracle_mod.formal_solution(p, S1)[0], rtol=RTOL, atol=0)
    assert np.allclose(J2, oracle_mod.formal_solution(p, S2)[0], rtol=RTOL, atol=0)


@pytest.mark.parametrize("form", ["linear", "df"])
def test_large_operator_in_chunks(R, oracle_mod, form):
    """Too large for the bound on its size: counts read back, planes in
    several chunks; sampled voxels against the oracle, and a second opacity
    in the same block."""
    p = W.slab_65(n=49, n_theta=24, n_phi=24)
    rng = np.random.default_rng(3)
    vox = np.unique(np.concatenate([np.arange(0, p.nvox, p.nvox // 40), [p.nvox - 1]]))
    with R.Solver(p, precision=_form(R, form)[1]) as s:
        for scale in (1.0, 0.3):
            q = W.Problem(p.nx, p.ny, p.nz, p.chi * scale, p.eps, p.B, p.mu, p.phi, p.w)
            S = p.B * (0.5 + rng.random(p.B.shape))
            R.rt_set_opacity(s.ctx, q.chi)
            s.formal_solution(p.B, want_lstar=False)
            J, _ = s.formal_solution(S, want_lstar=False)
            Jo = oracle_mod.mean_intensity_at(q, S, vox)
            assert np.allclose(J.reshape(-1)[vox], Jo, rtol=RTOL, atol=0)


@pytest.mark.parametrize("form", ["linear", "df"])
@pytest.mark.parametrize("nx,ny,nz", [(3, 11, 127), (3, 11, 128), (64, 32, 63), (64, 32, 64), (63, 33, 65)])
def test_apply_forms_match_march(R, form, nx, ny, nz):
    """Both sides of the numbers of tiles (254, 256; 4032, 4096, 4225) at which
    the warps of a tile change, against the march without recording."""
    p = W.random_slab(nx, ny, nz, n_theta=2, n_phi=3, seed=nz)
    p.src_order, prec = _form(R, form)
    S = 0.5 + np.random.default_rng(6).random(p.B.shape)
    J = {}
    for record in (-1, 0):
        with R.Solver(p, precision=prec, record=record) as s:
            J[record] = s.formal_solution(S, want_lstar=False)[0]
            assert R.rt_fs_record_info(s.ctx)[1] == (record != 0)
    assert np.allclose(J[-1], J[0], rtol=RTOL, atol=0)


@pytest.mark.parametrize("form", FORMS)
def test_steps_are_counted_per_formal_solution(R, form):
    """Every formal solution adds the steps of its recording, also after new
    opacities and after formal solutions that are marched."""
    p = W.random_slab(9, 8, 12, n_theta=4, n_phi=6, seed=8)
    q = W.random_slab(9, 8, 12, n_theta=4, n_phi=6, seed=9, chi_decades=5.0)
    p.src_order, prec = _form(R, form)
    q.src_order = p.src_order

    def steps(s, n):
        R.rt_reset_stats(s.ctx)
        for _ in range(n):
            s.formal_solution(p.B, want_lstar=False)
        return R.rt_get_stats(s.ctx)["steps"]

    with R.Solver(q, precision=prec) as s:
        one_q = steps(s, 1)
    with R.Solver(p, precision=prec) as s:
        one_p = steps(s, 1)
        assert one_p != one_q and steps(s, 3) == 3 * one_p
        R.rt_set_opacity(s.ctx, q.chi)
        assert steps(s, 1) == one_q and steps(s, 2) == 2 * one_q
        R.rt_set_fs_record(s.ctx, 0)
        marched = steps(s, 1)
        R.rt_set_fs_record(s.ctx, -1)
        assert steps(s, 2) == 2 * one_q
    assert 0 < marched <= one_q
