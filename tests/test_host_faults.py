"""The host code on a device in host memory (fake_device.py): waits that gave up,
numbers of sweeps up to the largest, allocations that fail."""

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


@pytest.mark.parametrize("form", ["fp64", "df64", "parabolic", "short"])
def test_recording_that_gets_no_memory_marches(lib, form):
    """Each allocation of a first formal solution with recording fails in turn: the
    formal solution marches, or replays ray by ray, and the next one records."""
    fake_device.run(lib, f"""
form = {form!r}
p = W.random_slab(9, 8, 12, n_theta=4, n_phi=6, seed=1)
p.src_order = int(form == "parabolic")
kw = dict(precision=R.RT_DF64 if form == "df64" else R.RT_FP64,
          fs_method=R.RT_FS_SHORT if form == "short" else R.RT_FS_LONG)
n = tried = 0
while True:
    with R.Solver(p, record=0, **kw) as s:
        s.formal_solution(p.B)          # the buffers of every formal solution
        R.rt_set_fs_record(s.ctx, -1)
        counts()
        lib.fake_fail(n)
        s.formal_solution(p.B)
        if not lib.fake_failed():
            lib.fake_fail(-1)
            break
        first = counts()
        s.formal_solution(p.B)
        assert R.rt_fs_record_info(s.ctx)[1], n
        if form in ("fp64", "df64"):
            assert first["marches"] + first["replays"] == 1 and not first["applies"], (n, first)
            again = counts()
            assert again["applies"] == (first["marches"]) and again["replays"] == first["replays"], (n, again)
    n += 1
assert n >= (1 if form == "short" else 3), n
assert lib.fake_live() == 0
""")
