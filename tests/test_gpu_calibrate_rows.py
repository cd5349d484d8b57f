"""The bandwidth search with eight lanes per row at the edges of its layout
(neighbours per lane, rows per warp), against the FP64 oracle within the parity
bound of P (1e-5 absolute), and on rows whose perplexity is out of reach, where
it has to give what the bisection gives."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def at():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as pkg
    return pkg


@pytest.mark.parametrize("k", [2, 7, 8, 9, 32, 33, 64, 65, 96, 97, 128, 129, 192, 193, 256, 257])
@pytest.mark.parametrize("rows,scale", [(1, 1.0), (5, 1e-8), (18, 1e6)])
def test_lane_and_row_edges(at, k, rows, scale):
    rng = np.random.default_rng(k * 100 + rows)
    d2 = np.sort(scale * (1.0 + rng.gamma(2.0, 1.0, size=(rows, k))), axis=1).astype(np.float32)
    perp = max(1.5, k / 3.0)
    P, beta = at.atsne_calibrate_P(torch.from_numpy(d2).cuda(), perp)
    at.atsne_check()
    o_P, o_beta, _, _ = oracle.calibrate(d2.astype(np.float64), perp)
    assert np.abs(P.cpu().numpy() - o_P).max() <= 1e-5
    assert np.abs(beta.cpu().numpy() / o_beta - 1).max() <= 1e-3


def test_rows_out_of_reach_equal_the_bisection(at):
    k, perp = 40, 12.0
    rng = np.random.default_rng(5)
    d2 = np.sort(rng.random((9, k)), axis=1).astype(np.float32)
    d2[1, :] = 3.0                    # equal distances
    d2[2, :20] = 0.0                  # more nearest neighbours than the perplexity
    d2[3, :12] = d2[3, 0]             # as many
    d2[4, 30:] = np.inf               # absent entries
    d2[5, 12:] = np.inf               # as many present as the perplexity
    d2[6, :] = np.inf                 # no neighbour
    d2[7, :] *= 1e37                  # near the end of the range
    d2[8, :] *= 1e-37
    d = torch.from_numpy(d2).cuda()
    P, beta = at.atsne_calibrate_P(d, perp)
    # another tolerance takes the bisection kernel
    bP, bb = at.atsne_calibrate_P(d, perp, tol=1.0001e-5)
    at.atsne_check()
    assert (P - bP).abs().max().item() <= 1e-5
    out = [1, 2, 3, 5, 6]
    assert torch.equal(beta[out], bb[out])
    assert ((beta[[0, 4, 7, 8]] / bb[[0, 4, 7, 8]]) - 1).abs().max().item() <= 1e-3
