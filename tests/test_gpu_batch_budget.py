"""FP64 and double-float batches whose budget holds the operators of some problems
only: they run in waves, a later one in the memory that an earlier one returned, with
the iterates of single solves bit for bit; solved twice."""

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


@pytest.mark.parametrize("form", ["fp64", "df64"])
@pytest.mark.parametrize("room", [1, 2])
def test_operators_in_waves(R, form, room):
    prec = R.RT_DF64 if form == "df64" else R.RT_FP64
    probs = [W.random_slab(nx, ny, nz, n_theta=6, n_phi=4, seed=nx, eps_range=(0.05, 1.0))
             for nx, ny, nz in [(9, 7, 6), (17, 9, 11), (13, 11, 9), (16, 9, 12), (5, 5, 5)]]
    single, sizes = [], []
    for p in probs:
        with R.Solver(p, precision=prec, ng_period=4) as s:
            single.append(s.solve(tol=1e-9, max_iter=500))
            sizes.append(R.rt_fs_record_info(s.ctx)[0])
    b = R.rt_batch_create(probs, precision=prec)
    try:
        R.rt_batch_set_ng(b, 4, 0.0)
        R.rt_batch_set_fs_record(b, room * max(sizes))
        for _ in range(2):
            before = R.rt_batch_get_stats(b)["iterations"]
            r = R.rt_batch_solve(b, len(probs), tol=1e-9, max_iter=500)
            assert r["converged"]
            # more than one wave
            assert R.rt_batch_get_stats(b)["iterations"] - before > max(r["iters"])
            for i, p in enumerate(probs):
                assert single[i]["iters"] == r["iters"][i]
                assert np.array_equal(R.rt_batch_get_J(b, i, (p.nz, p.ny, p.nx)), single[i]["J"]), i
            R.rt_batch_reset(b, rebuild_lstar=True)
    finally:
        R.rt_batch_destroy(b)
