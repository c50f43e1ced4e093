"""How the visibilities are ordered for the gains kernels does not cost accuracy: the
same visibilities and pixels, with gains of one, once with the antenna pairs of the
tracks (granules of whole runs of a pair's samples) and once with pairs dealt at
random (granules of neighbours), are equally far from FP64.

Bound.  Either error is the root mean square of some 10^8 pairs' roundings; the two
estimates agree to a few per cent, 1.04 here, when the roundings are of the same size.
Granules of runs that measure their offsets from one centre made it 1.06 to 1.14."""
import numpy as np
import pytest

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
