"""The lattice operator over the range of its inputs: as near FP64 for values near
the smallest FP32 takes as for others, one call's huge inputs without a trace in
the next one's small ones, and the same in a solve.

Tolerance: that of tests/test_gpu_lattice.py, 6e-7 in the 2-norm."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 6e-7


def rel2(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def problem(gpu_lib):
    ctx = gpu_lib.Context(0)
    rng = np.random.default_rng(1)
    uvw = rng.uniform(-1, 1, (30000, 3)) * [1000.0, 1000.0, 100.0]
    P = ctx.problem()
    P.set_visibilities(uvw)
    P.set_pixels(synth.regular_grid(256, 0.2))
    P.forward(np.zeros(P.n_pix))
    ctx.counters_reset()
    P.forward(np.zeros(P.n_pix))
    assert ctx.counters()["launches"] == 5              # the lattice operator
    O = oracle.Problem(uvw, synth.regular_grid(256, 0.2), threads=8)
    yield P, O, rng
    ctx.close()


@pytest.mark.parametrize("scales", [(1e-36,), (1e-33, 1e30, 1e-36, 1.0), (1e35,), (2.0 ** 40, 1.0), (0.5 * 2.0 ** 40,)])
def test_operators_keep_their_accuracy_at_every_scale(problem, scales):
    P, O, rng = problem
    x, r = rng.random(P.n_pix), rng.normal(size=P.n_vis) + 1j * rng.normal(size=P.n_vis)
    rows, cols = rng.choice(P.n_vis, 200, replace=False), rng.choice(P.n_pix, 200, replace=False)
    f, a = oracle.forward(O, x, rows=rows), oracle.adjoint(O, r, cols=cols)
    for s in scales:
        assert rel2(P.forward(s * x)[rows] / s, f) <= TOL
        assert rel2(P.adjoint(s * r)[cols] / s, a) <= TOL


def test_solves_are_the_same_at_every_scale(problem, gpu_lib):
    """Data, lambda and the starting image scaled together scale the image."""
    P, O, rng = problem
    sky = np.zeros(P.n_pix)
    sky[rng.choice(P.n_pix, 40, replace=False)] = 1.0 + rng.random(40)
    V = P.forward(sky, gpu_lib.FP64)
    lam = 0.05 * P.adjoint(V, gpu_lib.FP64).max()
    images = []
    for s in (1.0, 2.0 ** -110, 2.0 ** 50):
        P.set_vis_data(s * V)
        images.append([P.solve(s * lam, max_iter=12, x0=s * sky * (k > 0), algorithm=algo)[0] / s
                       for algo in ("fista", "mfista") for k in range(2)])
    for other in images[1:]:
        for img, want in zip(other, images[0]):
            assert want.max() > 0.5 and np.max(np.abs(img - want)) <= 1e-5 * want.max()
