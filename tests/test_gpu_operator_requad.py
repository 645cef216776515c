"""Changes of the quadrature of a context (more and fewer directions, all of one
sign) give the J and Lambda* of a new context, bit for bit, also where opacities
change in between."""

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


@pytest.mark.parametrize("form", ["linear", "parabolic", "df"])
@pytest.mark.parametrize("shape", [(7, 5, 9), (20, 18, 40)])
def test_quadratures_in_turn(R, form, shape):
    p = W.random_slab(*shape, n_theta=4, n_phi=6, seed=3)
    p.src_order = int(form == "parabolic")
    prec = R.RT_DF64 if form == "df" else R.RT_FP64
    S = 0.5 + np.random.default_rng(1).random(p.B.shape)
    chi2 = p.chi[::-1].copy()
    one = (-np.linspace(0.2, 1.0, 5), np.arange(5.0), np.full(5, 0.2))
    with R.Solver(p, precision=prec) as s:
        s.formal_solution(S)
        for quad, chi in [(W.quadrature(16, 16), p.chi), (W.quadrature(16, 12), p.chi), (W.quadrature(2, 3), chi2),
                          (one, chi2), (W.quadrature(16, 16), chi2), (W.quadrature(4, 6), p.chi)]:
            R.rt_set_quadrature(s.ctx, *quad)
            R.rt_set_opacity(s.ctx, chi)
            J, L = s.formal_solution(S)
            q = W.Problem(p.nx, p.ny, p.nz, chi, p.eps, p.B, *quad, dx=p.dx, dy=p.dy, dz=p.dz,
                          top_bc=p.top_bc, bottom_bc=p.bottom_bc)
            q.src_order = p.src_order
            with R.Solver(q, precision=prec) as new:
                Jn, Ln = new.formal_solution(S)
            assert np.array_equal(J, Jn) and np.array_equal(L, Ln)
