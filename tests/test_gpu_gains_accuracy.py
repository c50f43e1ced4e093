"""How the visibilities are ordered for the gains kernels does not cost accuracy: the
same visibilities and pixels, with gains of one, once with the antenna pairs of the
tracks (granules of whole runs of a pair's samples) and once with pairs dealt at
random (granules of neighbours), are equally far from FP64.

Bound.  Either error is the root mean square of some 10^8 pairs' roundings; the two
estimates agree to a few per cent, 1.04 here, when the roundings are of the same size.
Granules of runs that measure their offsets from one centre made it 1.06 to 1.14."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [5, 6, 7])
def test_runs_of_a_pair_are_as_accurate_as_neighbours(gpu_lib, seed):
    rng = synth.rng_for(seed)
    uvw, ant = synth.uvw_tracks(synth.antennas(rng, 64, 1000.0, 20.0), -30.0, 16)
    uvw, ant = uvw[:32000], ant[:32000]
    side, extent = 128, 0.25
    delta = 2 * extent / side
    lm = synth.regular_grid(side, extent)
    lm = np.concatenate([lm + rng.uniform(-0.3 * delta, 0.3 * delta, lm.shape)] * 4)
    sigma = np.repeat([0.0, delta, 2 * delta, 4 * delta], side * side)
    kind = np.where(sigma == 0, 0, 2).astype(np.int32)
    x = rng.exponential(1.0, len(lm)) * (rng.random(len(lm)) < 0.01)
    r = rng.normal(size=len(uvw)) + 1j * rng.normal(size=len(uvw))
    err = []
    for pairs in (ant, rng.permutation(ant)):
        ctx = gpu_lib.Context(0)
        P = ctx.problem()
        P.set_visibilities(uvw, None, None, pairs)
        P.set_pixels(lm, sigma, kind)
        P.set_gains(np.ones((len(lm), 64), complex))
        want = P.forward(x, gpu_lib.FP64), P.adjoint(r, gpu_lib.FP64)
        err.append([np.linalg.norm(g - w) / np.linalg.norm(w) for g, w in zip((P.forward(x), P.adjoint(r)), want)])
        ctx.close()
    ratio = np.array(err[0]) / np.array(err[1])
    print("errors", err, "ratio", ratio)
    assert np.all(ratio <= 1.04), ratio


@pytest.mark.parametrize("n_times", [16, 13, 9])              # runs that all begin at multiples of 4, and others
@pytest.mark.parametrize("kinds,tol", [((0,), 6e-7), ((2,), 6e-7), ((0, 2), 6e-7), ((1,), 3e-6)])
def test_own_centres_of_every_pixel_kind(gpu_lib, n_times, kinds, tol):
    """Layouts most of whose granules measure from their pairs' own centres (24 antennas,
    small pixel granules), against the oracle.  A pair's phase is rounded to about 2e-7
    rad rms and its sine and cosine to as much again: 6e-7 of the 2-norm; paraxial
    pixels add w nu of their granule's offsets.  A wrong centre is an error of order 1."""
    rng = synth.rng_for(n_times)
    uvw, ant = synth.uvw_tracks(synth.antennas(rng, 24, 1000.0, 20.0), -30.0, n_times)
    lm = synth.regular_grid(64, 0.25)
    lm = lm + rng.uniform(-0.002, 0.002, lm.shape)
    kind = np.resize(np.array(kinds, np.int32), len(lm))
    sigma = np.where(kind == 0, 0.0, 1e-3)
    gains = synth.beam_gains(rng, lm, 24, theta=(0.3, 0.5), ramp=0.5)
    O = oracle.Problem(uvw, lm, sigma, kind, None, ant, gains, threads=8)
    ctx = gpu_lib.Context(0)
    P = ctx.problem()
    P.set_visibilities(uvw, None, None, ant)
    P.set_pixels(lm, sigma, kind)
    P.set_gains(gains)
    x = rng.normal(size=len(lm))
    r = rng.normal(size=len(uvw)) + 1j * rng.normal(size=len(uvw))
    for got, want in ((P.forward(x), oracle.forward(O, x)), (P.adjoint(r), oracle.adjoint(O, r))):
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
    ctx.close()
