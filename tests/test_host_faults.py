"""The host code where memory, a thread or a place in a cache is not what a call
hoped for: over a CUDA runtime and launchers that run nothing (fake_device.cpp),
so no device is needed and none can fault.  A launch with another problem's
tables, or with memory that is not allocated, is noted there."""
import os
import subprocess
import sys
import textwrap
import time

import numpy as np
import pytest

import fake_device
from paper_1310_2078_gb300 import synth


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_device.build(str(tmp_path_factory.mktemp("fake")))


@pytest.fixture
def sl1m(lib):
    m = fake_device.binding(lib)
    m.fake.fake_reset()
    yield m
    m.fake.fake_reset()


def faults(m):
    return m.fake.fake_faults().decode()


def lattice(ctx, side=128, n_vis=30000, w_max=100.0):
    rng = np.random.default_rng(side)
    P = ctx.problem()
    P.set_visibilities(rng.uniform(-1, 1, (n_vis, 3)) * [1000.0, 1000.0, w_max])
    P.set_pixels(synth.regular_grid(side, 1e-3 * side))
    return P


def scattered(ctx, n_vis=900, n_pix=700, seed=3):
    rng = np.random.default_rng(seed)
    P = ctx.problem()
    P.set_visibilities(rng.uniform(-100, 100, (n_vis, 3)))
    P.set_pixels(rng.uniform(-0.1, 0.1, (n_pix, 2)))
    return P


def wait_for(cond, limit_s=60.0):
    t0 = time.monotonic()
    while not cond():
        assert time.monotonic() - t0 < limit_s
        time.sleep(0.001)


def in_a_child(lib, code):
    """Runs code in a process of its own, which an exception that crosses the C ABI ends."""
    pre = f"""
        import sys
        sys.path[:0] = {[os.path.dirname(os.path.abspath(__file__)), fake_device.b.ROOT]!r}
        import numpy as np
        import fake_device
        from paper_1310_2078_gb300 import synth
        sl1m = fake_device.binding({lib!r})
        """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(pre) + textwrap.dedent(code)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]


def serve(ctx, P):
    t = ctx.server_submit(P, 1.0, L=1.0, max_iter=5)
    return ctx.server_wait(t, P, 60)


@pytest.mark.parametrize("second", [dict(n_vis=300, n_pix=500), dict(n_vis=5000, n_pix=4000), None])
@pytest.mark.parametrize("first", ["scattered", "lattice"])
def test_a_new_problem_at_a_destroyed_ones_address_is_another_problem(sl1m, first, second):
    """A running server keeps the tables of the last set of problems it ran."""
    ctx = sl1m.Context(0)
    ctx.server_start()
    A = scattered(ctx) if first == "scattered" else lattice(ctx)
    address = A.h.value
    serve(ctx, A)
    A.close()
    B = lattice(ctx) if second is None else scattered(ctx, **second)
    assert B.h.value == address
    sl1m.fake.fake_reset()
    serve(ctx, B)
    kinds = [sl1m.fake.fake_count(i) > 0 for i in range(4)]
    assert kinds == ([False, False, True, True] if second is None else [True, True, False, False])
    assert faults(sl1m) == ""
    ctx.close()


@pytest.mark.parametrize("call", ["forward", "adjoint", "solve"])
def test_a_call_after_one_that_ran_out_of_memory_starts_afresh(sl1m, call):
    """The allocation that fails is that of the partial sums, once the tables are made."""
    ctx = sl1m.Context(0)
    P = scattered(ctx)
    run = {"forward": lambda: P.forward(np.zeros(P.n_pix)), "adjoint": lambda: P.adjoint(np.zeros(P.n_vis, complex)),
           "solve": lambda: P.solve(1.0, L=1.0, max_iter=3)}[call]
    sl1m.fake.fake_fail(150_000, 1)
    with pytest.raises(sl1m.SL1MError) as e:
        run()
    assert e.value.status == sl1m.ERR_OOM
    run()
    assert faults(sl1m) == ""
    ctx.close()


# the workspace of the large lattice is above, every other allocation below (but the small one's workspace at 1 MB)
WORKSPACE = 20_000_000


@pytest.mark.parametrize("at_least,times", [(WORKSPACE, 2), (1_000_000, 3)])
def test_a_workspace_that_cannot_grow_is_left_to_those_who_use_it(sl1m, at_least, times):
    """... and the problem that asked for more takes the pair kernels.  Three
    failures: the old workspace is lost, too, and made again by its user."""
    ctx = sl1m.Context(0)
    A, B = lattice(ctx), lattice(ctx, 256, 60000)
    A.forward(np.zeros(A.n_pix))
    B.forward(np.zeros(B.n_pix), sl1m.FP64)                # laid out; the workspace comes with the first mixed call
    sl1m.fake.fake_reset()
    sl1m.fake.fake_fail(at_least, times)
    B.forward(np.zeros(B.n_pix))
    assert sl1m.fake.fake_count(0) == 1 and sl1m.fake.fake_count(2) == 0
    for P in (A, B):
        P.adjoint(np.zeros(P.n_vis, complex))
    assert sl1m.fake.fake_count(3) == 1 and sl1m.fake.fake_count(1) == 1
    assert faults(sl1m) == ""
    ctx.close()


def test_two_lattices_of_a_server_with_room_for_one(sl1m):
    ctx = sl1m.Context(0)
    A, B = lattice(ctx), lattice(ctx, 256, 60000)
    for P in (A, B):
        P.forward(np.zeros(P.n_pix), sl1m.FP64)
    sl1m.fake.fake_fail(WORKSPACE, 100)
    ctx.server_start(max_pairs_per_tick=1e12)
    sl1m.fake.fake_hold(1)
    tickets = [ctx.server_submit(P, 1.0, L=1.0, max_iter=5) for P in (A, B)]
    wait_for(lambda: ctx.server_info()["active"] == 2)
    sl1m.fake.fake_hold(0)
    for t, P in zip(tickets, (A, B)):
        ctx.server_wait(t, P, 60)
    assert sl1m.fake.fake_count(2) > 0 and faults(sl1m) == ""
    ctx.close()


def test_a_running_lattice_solve_stays_one_when_the_workspace_cannot_grow(sl1m):
    """Its residual has no polar form, so the pair kernels cannot take it over."""
    ctx = sl1m.Context(0)
    A, B = lattice(ctx), lattice(ctx, 256, 60000)
    B.forward(np.zeros(B.n_pix), sl1m.FP64)
    ctx.server_start(max_pairs_per_tick=1e12)
    sl1m.fake.fake_hold(1)
    tickets = [ctx.server_submit(A, 1.0, L=1.0, max_iter=5)]
    wait_for(lambda: ctx.server_info()["rounds"] > 3)
    sl1m.fake.fake_fail(WORKSPACE, 100)
    tickets.append(ctx.server_submit(B, 1.0, L=1.0, max_iter=5))
    wait_for(lambda: ctx.server_info()["active"] == 2)
    r = ctx.server_info()["rounds"]
    wait_for(lambda: ctx.server_info()["rounds"] > r + 3)
    before = [sl1m.fake.fake_count(i) for i in range(4)]
    r = ctx.server_info()["rounds"]
    wait_for(lambda: ctx.server_info()["rounds"] > r + 3)
    assert all(sl1m.fake.fake_count(i) > before[i] for i in range(4))      # A lattice, B pairs
    sl1m.fake.fake_hold(0)
    for t, P in zip(tickets, (A, B)):
        ctx.server_wait(t, P, 60)
    assert faults(sl1m) == ""
    ctx.close()


def test_a_lattice_without_memory_for_its_sums_takes_the_pair_kernels(sl1m):
    ctx = sl1m.Context(0)
    A, B = lattice(ctx), lattice(ctx, n_vis=60000)         # one workspace, more sums
    A.forward(np.zeros(A.n_pix))
    B.forward(np.zeros(B.n_pix), sl1m.FP64)
    sl1m.fake.fake_reset()
    sl1m.fake.fake_fail(900_000, 2)
    B.forward(np.zeros(B.n_pix))
    assert sl1m.fake.fake_count(0) == 1 and sl1m.fake.fake_count(2) == 0
    A.forward(np.zeros(A.n_pix))
    assert sl1m.fake.fake_count(2) == 1 and faults(sl1m) == ""
    ctx.close()


def test_a_lattice_of_many_passes_holds_the_sums_of_one(sl1m):
    sl1m.fake.fake_total(400 << 20)                        # 120 of its 648 planes
    ctx = sl1m.Context(0)
    P = lattice(ctx, n_vis=60000, w_max=20000.0)
    P.adjoint(np.zeros(P.n_vis, complex))
    assert sl1m.fake.fake_count(3) == 1 and faults(sl1m) == ""
    ctx.close()


def test_a_gains_layout_where_no_thread_can_be_had(lib):
    """The orders that threads of their own would try are tried by the caller: the same layout."""
    in_a_child(lib, """
        rng = np.random.default_rng(1)
        uvw, ant = synth.uvw_tracks(synth.antennas(rng, 12, 800.0, 20.0), -30.0, 16)
        lm = rng.uniform(-0.2, 0.2, (700, 2))
        shares = []
        for no_threads in (0, 1):
            ctx = sl1m.Context(0)
            P = ctx.problem()
            P.set_visibilities(uvw, None, None, ant)
            P.set_pixels(lm)
            P.set_gains(synth.beam_gains(rng, lm, 12))
            sl1m.fake.fake_no_threads(no_threads)
            P.forward(np.zeros(700))
            assert sl1m.fake.fake_faults() == b""
            shares.append((P.exact_tile_share(), P.bytes()))
            ctx.close()
        assert shares[0] == shares[1]
        """)


LATTICE_WS = 8 * (128 + 256) * 256 * 16                    # of lattice()'s 16 planes


def held(ctx, sl1m, problems, budget=0):
    """The server's info while it runs the problems' solves, which then end."""
    ctx.server_start(mem_budget_bytes=budget, max_pairs_per_tick=1e12)
    sl1m.fake.fake_hold(1)
    tickets = [ctx.server_submit(P, 1.0, L=1.0, max_iter=5) for P in problems]
    wait_for(lambda: ctx.server_info()["active"] == len(problems))
    info = ctx.server_info()
    sl1m.fake.fake_hold(0)
    for t, P in zip(tickets, problems):
        ctx.server_wait(t, P, 60)
    assert ctx.server_info()["bytes_in_use"] == 0 and faults(sl1m) == ""
    ctx.server_stop()
    return info


@pytest.mark.parametrize("first", ["laid out before", "laid out by the server"])
def test_a_lattice_operator_counts_against_the_servers_budget(sl1m, first):
    """Without room for it the solve takes the pair kernels, there only."""
    ctx = sl1m.Context(0)
    P = lattice(ctx)
    if first == "laid out before":
        P.forward(np.zeros(P.n_pix))
        assert sl1m.fake.fake_count(2) == 1
    sl1m.fake.fake_reset()
    budget = 16 << 20                                      # the solve's 11 MB, not its lattice's 17, or 10 by halves
    info = held(ctx, sl1m, [P], budget)
    assert sl1m.fake.fake_count(0) > 0 and sl1m.fake.fake_count(2) == 0
    assert 0 < info["bytes_in_use"] <= budget
    sl1m.fake.fake_reset()
    P.forward(np.zeros(P.n_pix))
    assert sl1m.fake.fake_count(2) == 1 and faults(sl1m) == ""
    ctx.close()


def test_lattice_solves_of_a_server_share_one_workspace(sl1m):
    ctx = sl1m.Context(0)
    A, B = lattice(ctx), lattice(ctx)
    one, two = (held(ctx, sl1m, ps)["bytes_in_use"] for ps in ([A], [A, B]))
    assert two - LATTICE_WS == 2 * (one - LATTICE_WS) > 0
    ctx.close()


def test_the_lattice_workspace_goes_with_the_last_lattice_problem(sl1m):
    ctx = sl1m.Context(0)
    A, B, S = lattice(ctx), lattice(ctx), scattered(ctx)
    for P in (S, A, B):
        P.forward(np.zeros(P.n_pix))
    A.close()
    before, own = sl1m.fake.fake_held(), B.bytes()
    B.close()
    assert before - sl1m.fake.fake_held() >= own + LATTICE_WS
    C = lattice(ctx)
    for P in (S, C):
        P.forward(np.zeros(P.n_pix))
    assert sl1m.fake.fake_count(2) == 3 and faults(sl1m) == ""
    ctx.close()


@pytest.mark.parametrize("gains", [False, True])
@pytest.mark.parametrize("scales", [1, 4])
def test_admission_counts_what_a_laid_out_problem_holds(sl1m, scales, gains):
    """Gaussian pixels of few scales, every buffer there is, in FP64."""
    rng = np.random.default_rng(2)
    uvw, ant = synth.uvw_tracks(synth.antennas(rng, 24, 800.0, 20.0), -30.0, 10)
    lm = rng.uniform(-0.2, 0.2, (1024, 2))
    ctx = sl1m.Context(0)
    P = ctx.problem()
    P.set_visibilities(uvw, None, None, ant)
    P.set_pixels(lm, np.resize(1e-3 * np.arange(1, scales + 1), 1024), np.full(1024, 2, np.int32))
    if gains:
        P.set_gains(synth.beam_gains(rng, lm, 24))
    for prec in (sl1m.FP64, sl1m.MIXED):
        P.forward(np.zeros(1024), prec)
        P.adjoint(np.zeros(len(uvw), complex), prec)
    P.solve(1.0, L=1.0, max_iter=1)
    ctx.server_start(precision=sl1m.FP64)
    sl1m.fake.fake_hold(1)
    t = ctx.server_submit(P, 1.0, L=1.0, max_iter=5)
    wait_for(lambda: ctx.server_info()["active"] == 1)
    in_use, holds = ctx.server_info()["bytes_in_use"], P.bytes()
    sl1m.fake.fake_hold(0)
    ctx.server_wait(t, P, 60)
    assert in_use >= holds
    ctx.close()


def test_the_fp64_tables_are_written_for_the_first_context(sl1m):
    """Another context's kernels may be reading them."""
    fills = lambda: sl1m.fake.fake_count(4)  # noqa: E731
    a, b = sl1m.Context(0), sl1m.Context(0)
    assert fills() == 1
    a.close()
    c = sl1m.Context(0)
    assert fills() == 1
    b.close()
    c.close()
    d = sl1m.Context(0)
    assert fills() == 2
    d.close()


def test_a_lattice_whose_tables_do_not_fit_host_memory_takes_the_pair_kernels(lib):
    """4,096 tiles by 1,600 planes of offsets, 25 MB; everything else is below 20."""
    in_a_child(lib, """
        rng = np.random.default_rng(1)
        for limit in (0, 20_000_000):
            ctx = sl1m.Context(0)
            P = ctx.problem()
            P.set_visibilities(rng.uniform(-1, 1, (200_000, 3)) * [1000.0, 1000.0, 12000.0])
            P.set_pixels(synth.regular_grid(512, 0.25))
            sl1m.fake.fake_reset()
            if limit:
                sl1m.fake.fake_host_limit(limit)
            P.forward(np.zeros(P.n_pix))
            sl1m.fake.fake_host_limit(1 << 60)
            assert (sl1m.fake.fake_count(0), sl1m.fake.fake_count(2)) == ((1, 0) if limit else (0, 1))
            assert sl1m.fake.fake_faults() == b""
            ctx.close()
        """)
