"""The CSR P at the edges of the merge's row classes (64, 128, 256, 512 and 1024
entries, hub rows beyond), with mutual and absent entries, and with a corpus
whose columns need 64-bit sort keys, against the FP64 oracle (columns equal,
values within 1e-5 / N)."""
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


def lists(N, k, refs, rng):
    """Random lists; row t (t < len(refs)) is referred to by refs[t] rows, part
    of them its own neighbours."""
    idx = np.empty((N, k), np.int32)
    for i in range(N):
        hubs = [t for t, n in enumerate(refs) if t != i and (i - t - 1) % N < n]
        rest = rng.choice(np.setdiff1d(np.arange(len(refs), N), [i]), size=k - len(hubs), replace=False)
        idx[i] = np.concatenate([hubs, rest])
    return idx


@pytest.mark.parametrize("N,k,refs", [
    (700, 20, [43, 44, 45, 107, 108, 109, 235, 236, 237, 491, 492, 493]),
    (3000, 30, [481, 482, 483, 993, 994, 995, 2000, 2999]),
    (40, 32, [31, 32, 33, 39]), (600, 512, [20]), (2, 1, [])])
def test_row_classes(at, N, k, refs):
    rng = np.random.default_rng(N)
    idx = lists(N, k, refs, rng)
    P = rng.random((N, k)).astype(np.float32)
    P /= P.sum(1, keepdims=True)
    rp, col, val = at.atsne_symmetrize(torch.from_numpy(idx).cuda(), torch.from_numpy(P).cuda())
    at.atsne_check()
    e_rp, e_col, e_val = oracle.symmetrize(idx, P.astype(np.float64))
    assert np.array_equal(rp.cpu().numpy(), e_rp) and np.array_equal(col.cpu().numpy(), e_col)
    assert np.abs(val.cpu().numpy() - e_val).max() * N <= 1e-5


def test_absent_entries_and_a_column_listed_twice(at):
    rng = np.random.default_rng(3)
    N, k = 900, 12
    idx = lists(N, k, [700], rng)
    P = rng.random((N, k)).astype(np.float32)
    idx[::7, 8:], P[::7, 8:] = -1, 0.0
    rp, col, val = [t.cpu().numpy() for t in at.atsne_symmetrize(torch.from_numpy(idx).cuda(), torch.from_numpy(P).cuda())]
    at.atsne_check()
    W = np.zeros((N, N))
    M = np.zeros((N, N), bool)
    for i in range(N):
        j = idx[i][idx[i] >= 0]
        W[i, j], M[i, j] = P[i][idx[i] >= 0], True
    S, M = (W + W.T) / (2 * N), M | M.T
    assert np.array_equal(rp, np.concatenate([[0], M.sum(1).cumsum()]))
    assert np.array_equal(col, np.nonzero(M)[1]) and np.abs(val - S[M]).max() * N <= 1e-5
    for row in (1, 0):  # an ordinary row and the hub
        bad = idx.copy()
        bad[row, 1] = bad[row, 2]
        at.atsne_symmetrize(torch.from_numpy(bad).cuda(), torch.from_numpy(P).cuda())
        with pytest.raises(at.AtsneError):
            at.atsne_check()


def test_columns_beyond_32_bit_keys(at):
    # more than 2^21 rows, k = 2: i's neighbours are i + 1 and row 0 or 5 (hubs
    # whose bitmap spans several column ranges)
    N = (1 << 21) + 3
    i = torch.arange(N, device="cuda")
    idx = torch.stack([(i + 1) % N, torch.where((i % 1000 == 7) & (i != 4), 5, (i + 2) % N)], 1).int().contiguous()
    P = torch.rand((N, 2), device="cuda")
    rp, col, val = at.atsne_symmetrize(idx, P)
    at.atsne_check()
    key, p = torch.cat([i.repeat_interleave(2) * N + idx.flatten(), idx.flatten().long() * N + i.repeat_interleave(2)]), P.double().flatten().repeat(2)
    u, inv = key.unique(return_inverse=True)
    s = torch.zeros(u.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, p) / (2 * N)
    assert torch.equal(col.long(), u % N) and torch.equal(rp[1:], (u // N).bincount(minlength=N).cumsum(0))
    assert ((val - s).abs().max() * N).item() <= 1e-5


@pytest.mark.parametrize("N", [(1 << 21) - 1, 1 << 21, (1 << 21) + 5])
def test_every_key_differs_from_the_mark_for_none(at, N):
    # the largest column in the last slot of a row of 1024 entries, with 21
    # column bits the largest key of all; and such rows with wider keys: four
    # rows are listed by 1,020 others, row N - 1 (whose entry is placed last,
    # or near it) among them
    k = 4
    i = torch.arange(N, device="cuda")
    idx = torch.stack([(i + t) % N for t in range(1, k + 1)], 1)
    at_row = torch.tensor([100000, 200000, 300000, 400000], device="cuda")
    for t in range(4):
        idx[500000 + 4 * t + 16 * torch.arange(1015, device="cuda"), 3] = at_row[t]
    idx[N - 1] = at_row
    P = torch.rand((N, k), device="cuda")
    rp, col, val = at.atsne_symmetrize(idx.int().contiguous(), P)
    at.atsne_check()
    src = i.repeat_interleave(k)
    assert torch.equal((idx.flatten() == at_row[:, None]).sum(1), torch.full((4,), 1024 - k, device="cuda"))
    key = torch.cat([src * N + idx.flatten(), idx.flatten() * N + src])
    u, inv = key.unique(return_inverse=True)
    s = torch.zeros(u.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, P.double().flatten().repeat(2)) / (2 * N)
    assert torch.equal(col.long(), u % N) and torch.equal(rp[1:], (u // N).bincount(minlength=N).cumsum(0))
    assert ((val - s).abs().max() * N).item() <= 1e-5


@pytest.mark.parametrize("N,k", [(1100, 12), (1200, 200)])
def test_a_mutual_column_listed_twice_in_a_hub_row(at, N, k):
    rng = np.random.default_rng(5)
    idx = lists(N, k, [N - 1], rng)  # every row lists row 0, which lists each of its neighbours mutually
    P = torch.full((N, k), 1.0 / k, device="cuda")
    at.atsne_symmetrize(torch.from_numpy(idx).cuda(), P)
    at.atsne_check()
    idx[0, k - 1] = idx[0, 0]
    at.atsne_symmetrize(torch.from_numpy(idx).cuda(), P)
    with pytest.raises(at.AtsneError):
        at.atsne_check()
