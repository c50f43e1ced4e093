"""The host code where memory, a thread or a place in a cache is not what a call
hoped for: over a CUDA runtime and launchers that run nothing (fake_device.cpp),
so no device is needed and none can fault.  A launch with another problem's
tables, or with memory that is not allocated, is noted there."""
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
