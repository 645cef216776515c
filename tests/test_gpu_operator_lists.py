"""The operator's node lists where their order can go wrong: all directions on
the same nodes (one entry of many contributions), one direction, one fewer and one
more than fill a warp's round of items, more nodes than a block has threads, and a
plane whose table of nodes is in global memory (above 24 Ki nodes); against the
oracle, with Lambda*.  1e-12 relative, the FP64 bar."""

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


def _slab(nx, ny, nz, mu, phi):
    p = W.random_slab(nx, ny, nz, seed=len(mu))
    p.mu, p.phi = np.asarray(mu, float), np.asarray(phi, float)
    p.w = np.full(len(mu), 1.0 / len(mu))
    return p


def _spread(n):
    rng = np.random.default_rng(n)
    return np.where(np.arange(n) % 2, -1, 1) * (0.15 + 0.85 * rng.random(n)), 6.28 * rng.random(n)


CASES = {
    "same nodes": lambda: _slab(6, 5, 5, [0.9, -0.9] * 37, [0.4] * 74),
    "vertical": lambda: _slab(6, 5, 5, [1.0, -1.0] * 20, np.arange(40) * 0.1),
    "one": lambda: _slab(6, 5, 5, [0.6], [1.0]),
    "14 directions": lambda: _slab(5, 7, 6, *_spread(14)),
    "18 directions": lambda: _slab(5, 7, 6, *_spread(18)),
    "many nodes": lambda: _slab(40, 30, 9, *_spread(300)),
    "global table": lambda: _slab(170, 150, 3, *_spread(12)),
}


@pytest.mark.parametrize("form", ["linear", "parabolic", "df"])
@pytest.mark.parametrize("name", CASES)
def test_lists_match_oracle(R, oracle_mod, name, form):
    p = CASES[name]()
    p.src_order = int(form == "parabolic")
    prec = R.RT_DF64 if form == "df" else R.RT_FP64
    S = 0.5 + np.random.default_rng(5).random(p.B.shape)
    with R.Solver(p, precision=prec) as s:
        J, L = s.formal_solution(S)
        assert R.rt_fs_record_info(s.ctx)[1]
    Jo, Lo = oracle_mod.formal_solution(p, S)
    assert np.allclose(J, Jo, rtol=1e-12, atol=0)
    if form == "parabolic":     # its weights amplify rounding in Lambda* (the kernel's too)
        return
    # a double-float entry: 2^-48 per coefficient and per sum
    assert np.max(np.abs(L - Lo)) <= (1e-13 if form == "df" else 1e-14) * np.abs(Lo).max()
