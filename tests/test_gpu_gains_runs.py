"""The gains kernels over what their layout can give them: granules of whole runs
of a pair's samples (16, 8 or 4 of them), runs cut short, pairs in any order;
pair tables of 16, 32 and 64 pixels per chunk and the gathers beyond them; up
to and beyond the number of Gaussian scales whose constants are tabulated.
Against the FP64 oracle at the mixed path's tolerance (1e-5 of the largest
output)."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def sky(rng, n_pix, scales, kinds):
    lm = rng.uniform(-0.2, 0.2, (n_pix, 2))
    sigma = np.resize(np.array(scales), n_pix)
    kind = np.where(sigma == 0.0, 0, np.resize(np.array(kinds, np.int32), n_pix)).astype(np.int32)
    return lm, sigma, kind


@pytest.mark.parametrize("n_ant,n_times,shuffle", [
    (8, 16, False),        # 28 pairs of 16: granules of 4 pairs, 64-pixel chunks
    (12, 10, False),       # 66 pairs of 10: runs of 8 and singles
    (20, 5, False),        # 190 pairs of 5: runs of 4 and singles
    (12, 16, True),        # the same pairs in no order
    (40, 1, False),        # every visibility its own pair: gathers
    (7, 9, False),         # 21 pairs of 9: a last granule with padding
])
@pytest.mark.parametrize("scales,kinds", [
    ([0.0], (0,)),                                              # Dirac
    ([0.0, 2e-3, 4e-3], (2, 2, 1)),                             # tabulated scales, paraxial among them
    ([1e-3, 2e-3, 3e-3, 4e-3], (2,)),                           # as many as the table takes
    ([1e-3, 2e-3, 3e-3, 4e-3, 5e-3, 6e-3], (2, 1)),             # more: formed in the kernels
])
def test_gains_orders_and_scales(gpu_lib, n_ant, n_times, shuffle, scales, kinds):
    rng = np.random.default_rng(n_ant * 100 + n_times + len(scales))
    uvw, ant = synth.uvw_tracks(synth.antennas(rng, n_ant, 800.0, 20.0), -30.0, n_times)
    if shuffle:
        p = rng.permutation(len(uvw))
        uvw, ant = uvw[p], ant[p]
    lm, sigma, kind = sky(rng, 700, scales, kinds)
    gains = synth.beam_gains(rng, lm, n_ant, theta=(0.3, 0.5), ramp=0.5)
    gains[::7, 0] = 0.0                                         # a dead antenna: log2 |G| = -inf
    O = oracle.Problem(uvw, lm, sigma, kind, None, ant, gains, threads=8)
    ctx = gpu_lib.Context(0)
    P = ctx.problem()
    P.set_visibilities(uvw, None, None, ant)
    P.set_pixels(lm, sigma, kind)
    P.set_gains(gains)
    x = rng.normal(size=len(lm))
    f, fo = P.forward(x), oracle.forward(O, x)
    assert np.max(np.abs(f - fo)) <= TOL * np.max(np.abs(fo))
    r = rng.normal(size=len(uvw)) + 1j * rng.normal(size=len(uvw))
    r[::9] = 0.0
    a, ao = P.adjoint(r), oracle.adjoint(O, r)
    assert np.max(np.abs(a - ao)) <= TOL * np.max(np.abs(ao))
    ctx.close()
