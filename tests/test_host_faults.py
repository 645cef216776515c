"""The host code on a device in host memory (fake_device.py): waits that gave up,
numbers of sweeps up to the largest, allocations that fail, budgets of batches,
chunks of a recording, blocks kept over a change of the quadrature."""

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


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_batch_keeps_its_budget(lib, form):
    """Problems of two sizes whose operators take more than their ray-by-ray
    recordings, under budgets from one such recording to several operators, solved
    three times: what is held never exceeds the budget, and every problem records."""
    fake_device.run(lib, f"""
prec = R.RT_DF64 if {form!r} == "df64" else R.RT_FP64
small = W.random_slab(16, 12, 10, n_theta=4, n_phi=6, seed=1)
large = W.random_slab(20, 16, 12, n_theta=4, n_phi=6, seed=2)
probs = [small, large, small, large, small, large]
sizes = []
for p in (small, large):
    with R.Solver(p, precision=prec) as s:
        s.formal_solution(p.B)
        sizes.append(R.rt_fs_record_info(s.ctx)[0])
        assert sizes[-1] > rays(p)
lib.fake_solves(5, 1e-9)
need = rays(large)
budgets = [need, need + 1000, sizes[1], sizes[1] + rays(small), sizes[1] + need, sizes[1] + sizes[0], 2 * sizes[1],
           2 * sizes[1] + need, 3 * sizes[1] + sizes[0], 20 * sizes[1]]
for budget in budgets:
    b = R.rt_batch_create(probs, precision=prec)
    R.rt_batch_set_fs_record(b, budget)
    lib.fake_large(int(0.8 * rays(small)))
    counts()
    for solve in range(3):
        lib.fake_solves(5, 1e-9)
        r = R.rt_batch_solve(b, len(probs))
        assert r["converged"]
        n = counts()
        assert n["marches"] == 0 and n["applies"] + n["replays"] == len(probs), (budget, solve, n)
        if budget >= sizes[1]:
            assert n["replays"] == 0, (budget, solve, n)
        held = lib.fake_large(int(0.8 * rays(small)))
        assert held <= budget, (budget, solve, held)
        R.rt_batch_reset(b, rebuild_lstar=True)
    R.rt_batch_destroy(b)
assert lib.fake_live() == 0
""")


def test_batch_that_stops_and_goes_on_keeps_its_budget(lib):
    """Problems that reach max_iter and go on in a later solve are admitted
    again, within the budget."""
    fake_device.run(lib, """
p = W.random_slab(16, 12, 10, n_theta=4, n_phi=6, seed=1)
with R.Solver(p) as s:
    s.formal_solution(p.B)
    one = R.rt_fs_record_info(s.ctx)[0]
b = R.rt_batch_create([p] * 5, precision=0)
R.rt_batch_set_fs_record(b, 2 * one)
lib.fake_large(int(0.8 * rays(p)))
lib.fake_solves(5, 0.5)
counts()
for it in (2, 3, 5):
    R.rt_batch_solve(b, 5, tol=0.0, max_iter=it)
n = counts()
assert n["marches"] == n["replays"] == 0 and n["applies"] == 25, n
assert lib.fake_large(1 << 60) <= 2 * one
R.rt_batch_destroy(b)
""")


@pytest.mark.parametrize("form", ["fp64", "df64", "fp32"])
def test_batch_automatic_budget_leaves_its_reserve(lib, form):
    """The automatic budget on devices with little room: 4 GiB stay free."""
    fake_device.run(lib, f"""
prec = dict(fp64=R.RT_FP64, df64=R.RT_DF64, fp32=R.RT_FP32_SWEEP)[{form!r}]
p = W.random_slab(16, 12, 10, n_theta=4, n_phi=6, seed=1)
lib.fake_solves(5, 1e-9)
recorded = []
for mb in (3, 8, 16, 32, 64, 128, 256):
    lib.fake_memory(400 * GB)
    b = R.rt_batch_create([p] * 6, precision=prec)
    total = lib.fake_live() + 4 * GB + (mb << 20)
    lib.fake_memory(total)
    lib.fake_peak(1)
    counts()
    for solve in range(2):
        assert R.rt_batch_solve(b, 6)["converged"]
        R.rt_batch_reset(b, rebuild_lstar=True)
    n = counts()
    recorded.append(n["applies"] + n["replays"])
    if recorded[-1]:
        assert total - lib.fake_peak(0) >= 4 * GB, (mb, recorded[-1])
    R.rt_batch_destroy(b)
assert recorded[-1] == 12 and recorded == sorted(recorded)
""")


def test_batch_uses_its_own_block_on_a_full_device(lib):
    """A pooled block that holds the recording takes no memory: it is used also where
    less than the reserve is free."""
    fake_device.run(lib, """
p = W.random_slab(16, 12, 10, n_theta=4, n_phi=6, seed=1)
lib.fake_solves(5, 1e-9)
lib.fake_memory(400 * GB)
b = R.rt_batch_create([p] * 3, precision=R.RT_FP32_SWEEP)
R.rt_batch_solve(b, 3)
assert counts()["replays"] == 3
R.rt_batch_reset(b, rebuild_lstar=True)
lib.fake_memory(lib.fake_live() + 3 * GB)
R.rt_batch_solve(b, 3)
assert counts()["replays"] == 3
R.rt_batch_destroy(b)
""")


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_operator_near_its_budget_is_recorded_in_large_chunks(lib, form):
    """33^3 with 256 directions, ray by ray 1.1 GiB, so an operator of up to 5.1 GiB: one
    of 4.6 records its 1 GiB of coefficients at once, not a few planes at a time;
    where max_bytes leaves less beside it, in chunks; above the budget ray by ray."""
    fake_device.run(lib, f"""
prec = R.RT_DF64 if {form!r} == "df64" else R.RT_FP64
p = W.slab_65(n=33, n_theta=16, n_phi=16)
own = lambda entries: entries * 33 * 35 * 32 * 8
for entries, record, chunks, applies in ((16704, -1, 1, 1), (16704, own(16704) + GB // 2, 14, 1),
                                         (18720, -1, 1, 0)):
    lib.fake_operator(entries, 3735, 1 << 40)
    with R.Solver(p, precision=prec, record=record) as s:
        counts()
        s.formal_solution(p.B)
        n = counts()
    assert n["applies"] == applies and n["replays"] == 1 - applies, (entries, record, n)
    assert n["chunks"] == 1 if chunks == 1 else n["chunks"] >= 12, (entries, record, n)
""")


def test_operator_is_kept_while_its_entries_are_worth_it(lib):
    """On both sides of the entries per step up to which the operator is the faster
    form: 7 in FP64, 7.5 in double-float, 8.5 for the parabolic source."""
    fake_device.run(lib, """
entries = 3200
lanes = entries * 33 * 35 * 32
for form, worth in (("fp64", 7.0), ("df64", 7.5), ("parabolic", 8.5)):
    p = W.slab_65(n=33, n_theta=16, n_phi=16)
    p.src_order = int(form == "parabolic")
    for ratio in (worth - 0.01, worth + 0.01, 1e6):
        lib.fake_operator(entries, 100, int(lanes / ratio))
        with R.Solver(p, precision=R.RT_DF64 if form == "df64" else R.RT_FP64) as s:
            counts()
            s.formal_solution(p.B)
            n = counts()
        kept = ratio < worth
        assert (n["applies"], n["replays"]) == ((1, 0) if kept else (0, 1)), (form, ratio, n)
""")


@pytest.mark.parametrize("form", ["fp64", "df64"])
def test_recording_keeps_its_blocks_over_a_quadrature(lib, form):
    """A quadrature of the same or a somewhat smaller size takes the blocks of the
    one before; a much smaller or a larger one its own; a grid frees them."""
    fake_device.run(lib, f"""
prec = R.RT_DF64 if {form!r} == "df64" else R.RT_FP64
p = W.random_slab(20, 18, 40, n_theta=32, n_phi=32, seed=1)
with R.Solver(p, precision=prec) as s:
    s.formal_solution(p.B)
    for n_theta, n_phi, new in ((32, 32, 0), (32, 24, 0), (32, 32, 0), (4, 2, 1), (32, 32, 1)):
        R.rt_set_quadrature(s.ctx, *W.quadrature(n_theta, n_phi))
        counts()
        s.formal_solution(p.B)
        n = counts()
        assert n["applies"] == 1
        # the recording's block itself where it has to grow; lists and working storage
        assert n["mallocs"] <= 1 if new == 0 else n["mallocs"] >= new, (n_theta, n_phi, n)
assert lib.fake_live() == 0
""")
