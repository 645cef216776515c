"""The host code on a device in host memory (fake_device.py): waits that gave up,
numbers of sweeps up to the largest."""

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


def test_barrier_words_of_any_number_of_sweeps(lib):
    """The one-kernel solve has a word for each barrier (two a sweep for
    Gauss-Seidel) inside its allocation; numbers of sweeps that take too many
    run as a graph, up to the largest int."""
    fake_device.run(lib, """
p = W.random_slab(5, 4, 6, n_theta=2, n_phi=4, seed=1)
lib.fake_memory(400 * GB)
for method in (0, 1):
    for sweeps in (1, 1000, (1 << 21) + 1, (1 << 22) + 1, (1 << 30) - 1, 1 << 30, (1 << 31) - 3, (1 << 31) - 1):
        with R.Solver(p, os_method=method) as s:
            s.formal_solution(p.B)
            counts()
            for _ in range(2):
                s.os_step(p.B, p.B, max_sweeps=sweeps)
            n = counts()
            one = sweeps * (1 + method) <= 1 << 22
            assert n["outside"] == 0, (method, sweeps)
            assert (n["solves"], n["graphs"]) == ((2, 0) if one else (0, 2)), (method, sweeps, n)
    for sweeps in (1000, 1 << 20, (1 << 30) + 1):
        b = R.rt_batch_create([p] * 3, precision=0)
        R.rt_batch_set_os_method(b, method)
        counts()
        R.rt_batch_solve(b, 3, tol=0.0, max_iter=2, max_sweeps=sweeps)
        n = counts()
        one = 3 * sweeps * (1 + method) <= 1 << 22
        assert n["outside"] == 0 and (n["solves"] == 2) == one and (n["graphs"] == 2) != one, (method, sweeps, n)
        R.rt_batch_destroy(b)
""")
