"""The density view at the edges of its tiles (32 pixels), chunks (1024 points
per CTA and step) and cluster sizes, against the FP64 oracle within the parity
bounds of tests/test_gpu_parity.py (f 1e-5 relative, the shares 1e-5)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,W,H", [(1, 1, 33), (1023, 31, 32), (1025, 33, 65), (8191, 32, 31), (8192, 64, 1),
                                   (8193, 97, 40), (16400, 800, 800)])
@pytest.mark.parametrize("cutoff,sorted_by", [(4.0, False), (1.5, True), (0.0, False)])
def test_kde_tile_and_chunk_edges(N, W, H, cutoff, sorted_by):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as at
    if W * H * N > 4e8 and cutoff == 0.0:
        N, W, H = 16400, 90, 70
    rng = np.random.default_rng(N + W)
    c = rng.integers(0, 5, N)
    if sorted_by:
        c = np.sort(c)
    Y = (np.stack([c * 2.0, (c % 3) * 1.5], 1) + rng.normal(scale=0.4, size=(N, 2))).astype(np.float32)
    rho, sel = rng.random(N).astype(np.float32), (c == 2).astype(np.uint8)
    x0, y0, px, h = -1.5, -1.0, 11.0 / W, 0.3
    g = at.atsne_kde_map(torch.from_numpy(Y).cuda(), x0, y0, px, W, H, h, cutoff=cutoff, lens_k=2.0,
                         rho=torch.from_numpy(rho).cuda(), selected=torch.from_numpy(sel).cuda())
    of, os_, oa, oal = oracle.kde(Y, x0, y0, px, W, H, h, cutoff=cutoff, k=2.0, rho=rho, selected=sel)
    gf, gs, ga, gal = [t.cpu().numpy().astype(np.float64) for t in g]
    assert np.all(np.abs(gf - of) <= 1e-5 * np.abs(of) + 1e-12)
    live = of > 1e-9
    for u, v in ((gs, os_), (ga, oa), (gal, oal)):
        assert np.abs(u - v)[live].max(initial=0.0) <= 1e-5


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_precision_out_of_reach_does_not_count(bad):
    # a point's rho enters the pixels within cutoff * h of it and no other, whatever its value
    import paper_1512_01655_gb300 as at
    rng = np.random.default_rng(7)
    N, W, H, h, cutoff, px = 2000, 70, 50, 0.3, 2.0, 0.1
    Y = (rng.random((N, 2)) * [7.0, 5.0]).astype(np.float32)
    rho = rng.random(N).astype(np.float32)
    Y[11] = (3.02, 2.04)
    args = (0.0, 0.0, px, W, H, h)
    a0 = at.atsne_kde_map(torch.from_numpy(Y).cuda(), *args, cutoff=cutoff, rho=torch.from_numpy(rho).cuda())[2].cpu().numpy()
    rho[11] = bad
    a1 = at.atsne_kde_map(torch.from_numpy(Y).cuda(), *args, cutoff=cutoff, rho=torch.from_numpy(rho).cuda())[2].cpu().numpy()
    # the decision as the interface states it: centres and distances in FP32, each operation rounded once
    f = np.float32
    cx = (np.arange(W, dtype=np.float64) + 0.5) * float(f(px))
    cy = (np.arange(H, dtype=np.float64) + 0.5) * float(f(px))
    dx, dy = (cx.astype(f) - Y[11, 0]).astype(f), (cy.astype(f) - Y[11, 1]).astype(f)
    d2 = (dx.astype(np.float64)[None, :] ** 2 + (dy * dy).astype(np.float64)[:, None]).astype(f)
    r = f(cutoff) * f(h)
    near = d2 <= r * r
    assert near.any() and not np.isfinite(a1[near]).any()
    assert np.array_equal(a1[~near], a0[~near])
