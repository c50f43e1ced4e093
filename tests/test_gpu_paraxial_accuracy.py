"""Paraxial Gaussian pixels far from the phase centre under a large w: their phase
term -w nu, nu = n - 1 + r^2/2, is w times a number that the products w (n - 1) and
w r^2/2 cancel to, so either alone may not be rounded.

Tolerance.  The mixed path rounds a pair's phase to about 2e-7 rad rms and its sine
and cosine to as much again; 6e-7 of the result's 2-norm leaves a third over the
3.5e-7 to 4.5e-7 that Dirac and wide-field pixels measure, and is asked of
wide-field pixels at the same places too."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 6e-7


def rel2(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("kind", [1, 2])
@pytest.mark.parametrize("gains", [False, True])
@pytest.mark.parametrize("spread", [15.0, 1000.0])         # tiles by the linear form, and by the exact one
def test_paraxial_error_is_that_of_wide_field_pixels(gpu_lib, kind, gains, spread):
    rng = np.random.default_rng(int(spread) + gains)
    n_vis, n_pix, n_ant = 3000, 1500, 12
    uvw = np.array([600.0, -500.0, 900.0]) * (spread < 100) + rng.uniform(-spread, spread, (n_vis, 3))
    lm = np.array([0.2, 0.15]) + rng.uniform(-0.08, 0.08, (n_pix, 2))
    sigma, kinds = np.full(n_pix, 1e-4), np.full(n_pix, kind, np.int32)
    ant = rng.integers(0, n_ant, (n_vis, 2)).astype(np.int32)
    g = synth.beam_gains(rng, lm, n_ant, theta=(0.5, 0.8)) if gains else None
    ctx = gpu_lib.Context(0)
    P = ctx.problem()
    P.set_visibilities(uvw, None, None, ant)
    P.set_pixels(lm, sigma, kinds)
    if gains:
        P.set_gains(g)
    x = rng.random(n_pix)
    f = P.forward(x)
    share = P.exact_tile_share()[0]
    assert share == 0.0 if spread < 100 else share > 0.5
    r = rng.normal(size=n_vis) + 1j * rng.normal(size=n_vis)
    a = P.adjoint(r)
    O = oracle.Problem(uvw, lm, sigma, kinds, None, ant, g, threads=8)
    assert rel2(f, oracle.forward(O, x)) <= TOL
    assert rel2(a, oracle.adjoint(O, r)) <= TOL
    ctx.close()
