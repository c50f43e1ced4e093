"""The FP64 kernels take sine, cosine and powers of two from tables of 2048
points and Taylor polynomials of the rest, and split the work by single
streamed elements: against the FP64 oracle, entry for entry.

Tolerance.  With the terms of every phase summing to less than PHI turns (u l +
v m + w (n - 1) below 45, the Gaussian terms gam t and id beta s^2 (u^2 + v^2) / 2
below 30 and 70), either side rounds a phase four or five times (2^-53 PHI
turns each) and everything else to a few 2^-53, so an output is off by less
than 2 * 2 pi * 5 * 2^-53 * PHI of the sum of its terms' magnitudes."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu

PHI = 160.0
TOL = 4 * np.pi * 5 * 2.0 ** -53 * PHI


@pytest.mark.parametrize("nv,npx", [(1, 1), (3, 64), (64, 65), (513, 31), (700, 1100)])
@pytest.mark.parametrize("kinds", [(0,), (1,), (2,), (0, 1, 2)])
@pytest.mark.parametrize("gains", [False, True])
def test_fp64_matches_oracle_to_rounding(gpu_lib, nv, npx, kinds, gains):
    # Gaussian amplitudes from 1 down to below the smallest double
    d = synth.random_problem(nv + npx, nv, npx, kinds=kinds, gains=gains, n_ant=7, uv_max=100, w_max=100,
                             extent=0.3, sigma_max=0.12)
    if gains:
        d["gains"] = np.exp(2j * np.pi * np.random.default_rng(1).random((npx, 7)))   # magnitude 1
    O = oracle.Problem(d["uvw"], d["lm"], d["sigma"], d["kind"], None, d["ant_pair"], d["gains"], threads=8)
    ctx = gpu_lib.Context(0)
    P = ctx.problem()
    P.set_visibilities(d["uvw"], None, None, d["ant_pair"])
    P.set_pixels(d["lm"], d["sigma"], d["kind"])
    if gains:
        P.set_gains(d["gains"])
    rng = np.random.default_rng(nv)
    inv_n = 1.0 / np.sqrt(1.0 - (d["lm"] ** 2).sum(axis=1))
    x = rng.normal(size=npx)
    assert np.max(np.abs(P.forward(x, gpu_lib.FP64) - oracle.forward(O, x))) <= TOL * np.sum(np.abs(x) * inv_n)
    r = rng.normal(size=nv) + 1j * rng.normal(size=nv)
    r[::5] = 0.0                                        # no argument
    r[1::7] = -np.abs(r[1::7])                          # argument 1/2 turn
    a, ao = P.adjoint(r, gpu_lib.FP64), oracle.adjoint(O, r)
    assert np.all(np.abs(a - ao) <= TOL * np.sum(np.abs(r)) * inv_n)
    ctx.close()
