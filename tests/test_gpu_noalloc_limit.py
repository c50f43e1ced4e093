"""sl1m_forward_noalloc near its 32 MiB: what a split of the work by granules of
64 pixels lets in is let in, also in FP64, whose split is by single pixels."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_blk,prec", [(2031, 0), (2031, 1), (1900, 0)])
def test_few_pixels_and_as_many_visibilities_as_fit(gpu_lib, n_blk, prec):
    import torch
    n_vis, n_pix = 512 * n_blk, 50                 # output and one partial slot a block: 16,384 bytes each a block
    rng = np.random.default_rng(n_blk)
    uvw, lm = rng.uniform(-50, 50, (n_vis, 3)), rng.uniform(-0.1, 0.1, (n_pix, 2))
    ctx = gpu_lib.Context(0, stream=torch.cuda.Stream())
    P = ctx.problem()
    P.set_visibilities(uvw)
    P.set_pixels(lm)
    xh = rng.random(n_pix)
    want = P.forward(xh, prec)
    x = torch.as_tensor(xh, device="cuda")
    got = torch.zeros((n_vis, 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    P.forward_noalloc(x, got, prec)
    torch.cuda.synchronize()
    g = got.cpu().numpy()
    g = g[:, 0] + 1j * g[:, 1]
    assert np.max(np.abs(g - want)) <= (1e-12 if prec == 0 else 1e-6) * np.max(np.abs(want))
    rows = rng.choice(n_vis, 50, replace=False)
    o = oracle.forward(oracle.Problem(uvw, lm, threads=8), xh, rows=rows)
    assert np.max(np.abs(g[rows] - o)) <= (1e-10 if prec == 0 else 1e-5) * np.max(np.abs(o))
    ctx.close()
