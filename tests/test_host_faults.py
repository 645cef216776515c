"""Waits that gave up, on a device in host memory (fake_device.py): what the
host code keeps for the next call."""

import pytest

import fake_device


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_device.build(str(tmp_path_factory.mktemp("fake")))


def test_history_of_a_solve_that_timed_out_is_dropped(lib):
    """The third iteration of a batch gives up before it has copied its J to the
    history: the next solve repeats it and must not extrapolate in the fourth
    from what was copied; one without the time-out extrapolates there."""
    fake_device.run(lib, """
p = W.random_slab(5, 4, 6, n_theta=2, n_phi=4, seed=1)
for gave_up in (False, True):
    b = R.rt_batch_create([p, p], precision=0)
    R.rt_batch_set_ng(b, 4, 0.0)
    lib.fake_solves(5, 0.5)
    R.rt_batch_solve(b, 2, tol=0.0, max_iter=2)
    if gave_up:
        lib.fake_solves(-1, 0.5)
        try:
            R.rt_batch_solve(b, 2, tol=0.0, max_iter=4)
            raise SystemExit("no error")
        except R.RtError as e:
            assert e.code == R.RT_ETIMEOUT, e.code
    lib.fake_solves(5, 0.5)
    counts()
    r = R.rt_batch_solve(b, 2, tol=0.0, max_iter=4)
    assert r["iters"].tolist() == [4, 4]
    assert counts()["ng"] == (0 if gave_up else 2)
    R.rt_batch_destroy(b)
    assert lib.fake_live() == 0
""")
