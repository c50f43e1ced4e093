"""The lattice operator (gridding and FFT) that the mixed path takes for Dirac
pixels on a regular (l, m) lattice: against the FP64 oracle for every transform
length, odd and ragged lattices, holes, any pixel order, negative and zero w;
and the pixel sets that must keep the pair kernels.

Tolerance.  A kernel of 8 cells at twice the band interpolates to 2e-7 of the
result's norm per axis (three axes: u, v, w), which bounds the FP32 rounding of
the transforms as well: 6e-7 in the 2-norm, over all outputs or a sample."""
import numpy as np
import pytest

import oracle
from paper_1310_2078_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 6e-7
LATTICE_LAUNCHES, PAIR_LAUNCHES = 5, 3        # of one forward call, one pass over the planes


def lattice(nx, ny, dl, dm, l0=0.0, m0=0.0, keep=1.0, seed=0):
    """Lattice points in random order, a share `keep` of them."""
    rng = np.random.default_rng(seed)
    s, t = np.meshgrid(np.arange(nx) - nx // 2, np.arange(ny) - ny // 2)
    lm = np.stack([l0 + s.ravel() * dl, m0 + t.ravel() * dm], axis=1)
    pick = rng.permutation(lm.shape[0])[:max(1, int(keep * lm.shape[0]))]
    return lm[pick]


def tracks(nv, uv_max, w_max, seed=1, w_sign=None):
    rng = np.random.default_rng(seed)
    uvw = np.stack([rng.uniform(-uv_max, uv_max, nv), rng.uniform(-uv_max, uv_max, nv),
                    rng.uniform(-w_max, w_max, nv)], axis=1)
    if w_sign is not None:
        uvw[:, 2] = w_sign * np.abs(uvw[:, 2])
    return uvw


def problem(ctx, uvw, lm, vis=None, **kw):
    P = ctx.problem()
    P.set_visibilities(uvw, vis, kw.get("weights"), kw.get("ant_pair"))
    P.set_pixels(lm, kw.get("sigma"), kw.get("kind"))
    if kw.get("gains") is not None:
        P.set_gains(kw["gains"])
    return P


def forward_launches(ctx, P):
    P.forward(np.zeros(P.n_pix))
    ctx.counters_reset()
    P.forward(np.zeros(P.n_pix))
    return ctx.counters()["launches"]


def rel2(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = gpu_lib.Context(0)
    yield c
    c.close()


# transform lengths 64 .. 4096 on either axis, odd and even sizes, coarse and fine spacings
LATTICES = [
    ("64x2048", lattice(32, 600, 2e-3, 1e-3), tracks(30000, 1000, 100)),
    ("2048x64 odd", lattice(701, 31, 1e-3, 9e-3), tracks(20001, 1500, 50)),
    ("256x256 odd", lattice(127, 97, 3e-3, 2e-3), tracks(12001, 2000, 300)),
    ("512x256 holes", lattice(255, 128, 1e-3, 2e-3, keep=0.6), tracks(9973, 1500, 150)),
    ("256x1024 off centre", lattice(100, 300, 5e-4, 1e-3, 0.2, -0.3), tracks(20000, 900, 60)),
    ("1024x512 w < 0", lattice(400, 250, 1e-3, 1e-3), tracks(3001, 1000, 60, w_sign=-1)),
    ("2048x64", lattice(1024, 32, 5e-4, 5e-3), tracks(5003, 1000, 100)),
    ("64x4096 w = 0", lattice(20, 2000, 1e-3, 3e-4), tracks(6000, 800, 0)),
    ("4096x128", lattice(1500, 40, 4e-4, 2e-3), tracks(4001, 2500, 20)),
    ("128x2048 narrow", lattice(50, 900, 1e-6, 1e-6), tracks(5000, 200000, 50000)),
]


@pytest.mark.parametrize("name,lm,uvw", LATTICES, ids=[c[0] for c in LATTICES])
def test_lattice_operator_matches_oracle(ctx, name, lm, uvw):
    P = problem(ctx, uvw, lm)
    assert forward_launches(ctx, P) == LATTICE_LAUNCHES
    O = oracle.Problem(uvw, lm, threads=8)
    rng = np.random.default_rng(7)
    x = rng.normal(size=len(lm))
    rows = rng.choice(len(uvw), 200, replace=False)
    assert rel2(P.forward(x)[rows], oracle.forward(O, x, rows=rows)) <= TOL
    r = rng.normal(size=len(uvw)) + 1j * rng.normal(size=len(uvw))
    cols = rng.choice(len(lm), 200, replace=False)
    assert rel2(P.adjoint(r)[cols], oracle.adjoint(O, r, cols=cols)) <= TOL


def test_planes_in_several_passes(ctx):
    """More planes than the workspace holds at once: the passes add up."""
    lm = lattice(1024, 1024, 5e-4, 5e-4)
    uvw = tracks(200_000, 1000, 3000)
    P = problem(ctx, uvw, lm)
    n = forward_launches(ctx, P)
    assert n > LATTICE_LAUNCHES and (n - 2) % 3 == 0
    O = oracle.Problem(uvw, lm, threads=8)
    rng = np.random.default_rng(3)
    x = rng.random(len(lm)) * (rng.random(len(lm)) < 0.01)
    rows = rng.choice(len(uvw), 100, replace=False)
    assert rel2(P.forward(x)[rows], oracle.forward(O, x, rows=rows)) <= TOL
    r = rng.normal(size=len(uvw)) + 1j * rng.normal(size=len(uvw))
    cols = rng.choice(len(lm), 30, replace=False)
    assert rel2(P.adjoint(r)[cols], oracle.adjoint(O, r, cols=cols)) <= TOL


def _jitter(lm):
    out = lm.copy()
    out[5, 0] += 1e-6
    return out


def _rotated(lm):
    c, s = np.cos(0.3), np.sin(0.3)
    return lm @ np.array([[c, s], [-s, c]])


OTHERS = {
    "one pixel off the lattice": lambda lm: (_jitter(lm), {}),
    "rotated": lambda lm: (_rotated(lm), {}),
    "two pixels at one place": lambda lm: (np.concatenate([lm, lm[:1]]), {}),
    "Gaussian": lambda lm: (lm, dict(sigma=np.full(len(lm), 1e-3), kind=np.full(len(lm), 2, np.int32))),
    "gains": lambda lm: (lm, dict(gains=np.ones((len(lm), 3), complex))),
    "few pairs": lambda lm: (lm[:200], {}),
}


@pytest.mark.parametrize("which", sorted(OTHERS))
def test_other_pixel_sets_keep_the_pair_kernels(ctx, which):
    lm, kw = OTHERS[which](lattice(128, 100, 2e-3, 2e-3, seed=4))
    uvw = tracks(10000, 1000, 100)
    ant = np.stack([np.zeros(10000), np.ones(10000)], axis=1).astype(np.int32)
    P = problem(ctx, uvw, lm, ant_pair=ant, **kw)
    assert forward_launches(ctx, P) == PAIR_LAUNCHES
    x = np.random.default_rng(0).random(len(lm))
    rows = np.arange(0, 10000, 97)
    O = oracle.Problem(uvw, lm, kw.get("sigma"), kw.get("kind"), None, ant, kw.get("gains"), threads=8)
    want = oracle.forward(O, x, rows=rows)
    assert np.max(np.abs(P.forward(x)[rows] - want)) <= 1e-5 * np.max(np.abs(want))


def test_inputs_keep_their_range(ctx):
    """Inputs near the ends of FP32's range, summed coherently: no overflow in
    the transforms, no loss below."""
    lm = lattice(128, 128, 1e-5, 1e-5)
    uvw = tracks(10000, 100, 10)
    P = problem(ctx, uvw, lm)
    one_f, one_a = P.forward(np.ones(len(lm))), P.adjoint(np.ones(10000, complex))
    for scale in (2.0 ** 100, 2.0 ** -80):
        assert rel2(P.forward(np.full(len(lm), scale)) / scale, one_f) <= TOL
        assert rel2(P.adjoint(np.full(10000, scale, complex)) / scale, one_a) <= TOL


def test_solve_on_a_lattice_repeats_and_matches_fp64(gpu_lib):
    """A solve's captured step bakes in the shared workspace: a larger lattice
    in between reallocates it, and the image is the same bit for bit; a new
    layout of the same problem is taken up."""
    c = gpu_lib.Context(0)
    w = synth.config2(n_side=128)
    P = problem(c, w.uvw, w.lm)
    assert forward_launches(c, P) == LATTICE_LAUNCHES
    P.set_vis_data(P.forward(w.x_true, gpu_lib.FP64) + w.noise[:w.n_vis])
    L, _ = P.max_eig(precision=gpu_lib.FP64)
    lam = 0.02 * P.dirty_image(gpu_lib.FP64)[1]
    ref, _ = P.solve(lam, L=L, max_iter=30, precision=gpu_lib.FP64)
    for algo in ("fista", "mfista"):
        a, _ = P.solve(lam, L=L, max_iter=30, algorithm=algo)
        Q = problem(c, tracks(20000, 1500, 300), lattice(400, 400, 1e-3, 1e-3))
        Q.forward(np.ones(Q.n_pix))
        b, _ = P.solve(lam, L=L, max_iter=30, algorithm=algo)
        assert np.array_equal(a, b)
        if algo == "fista":
            assert np.max(np.abs(a - ref)) <= 1e-4 * ref.max()
    keep = np.arange(0, w.n_pix, 2)                 # every other column: another lattice
    P.set_pixels(w.lm[keep])
    want = P.forward(w.x_true[keep], gpu_lib.FP64)
    assert rel2(P.forward(w.x_true[keep]), want) <= TOL
    c.close()


def test_server_mixes_lattice_and_pair_problems(gpu_lib):
    c = gpu_lib.Context(0)
    w = synth.config2(n_side=128)
    d = synth.random_problem(5, 900, 700, kinds=(2,), uv_max=150, w_max=40, extent=0.15, sigma_max=0.005)
    P = problem(c, w.uvw, w.lm)
    Q = problem(c, d["uvw"], d["lm"], sigma=d["sigma"], kind=d["kind"])
    xq = np.zeros(700)
    xq[::100] = 1.0
    alone = []
    for p, x in ((P, w.x_true), (Q, xq)):
        p.set_vis_data(p.forward(x, gpu_lib.FP64))
        lam = 0.02 * p.dirty_image(gpu_lib.FP64)[1]
        alone.append((lam, p.solve(lam, max_iter=25)[0]))
    c.server_start(ticks_per_round=2)
    for _ in range(2):
        t = [c.server_submit(p, lam, max_iter=25) for p, (lam, _) in zip((P, Q), alone)]
        for ticket, p, (_, img) in zip(t, (P, Q), alone):
            got, st = c.server_wait(ticket, p, 60)
            assert st["iters"] == 25 and np.max(np.abs(got - img)) <= 1e-6 * img.max()
    c.server_stop()
    c.close()
