"""Row lists around the size up to which a block merges a single row, and lists
long enough that sampled thresholds come out too low for some of their rows. On
small whole numbers every key is exact in BF16, so that the approximate mode's
lists too are the true ones, compared with an integer oracle."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def at():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as pkg
    return pkg


def oracle(X, q, k):
    """Nearest k by (distance, index), in whole numbers held exactly by FP64."""
    Xd = X.double()
    n = (Xd * Xd).sum(1)
    idx, d2 = [], []
    for c in q.split(2048):
        d = n[c][:, None] + n[None] - 2.0 * (Xd[c] @ Xd.T)
        d[torch.arange(len(c), device=d.device), c] = float("inf")
        key, order = (d * X.shape[0] + torch.arange(X.shape[0], device=d.device)).topk(k, largest=False)
        idx.append(order.int())
        d2.append(d.gather(1, order).float())
    return torch.cat(idx), torch.cat(d2)


@pytest.mark.parametrize("precision", ["fp32", "bf16", "bf16_approx"])
@pytest.mark.parametrize("over", [None, 0, 1])
@pytest.mark.parametrize("N,D", [(9000, 24), (1500, 85)])
def test_lists_around_one_row_per_block(at, precision, over, N, D):
    g = torch.Generator(device="cuda").manual_seed(N + D)
    X = torch.randint(0, 256, (N, D), generator=g, device="cuda").float()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Q = 1 if over is None else 4 * sms + over
    q = torch.randperm(N, generator=g, device="cuda")[:Q]
    i, d = at.atsne_knn(X, 12, queries=q.int(), precision=precision)
    at.atsne_check()
    ri, rd = oracle(X, q, 12)
    assert torch.equal(i, ri) and torch.equal(d, rd)


def test_rows_given_up_start_from_the_wider_rank(at):
    N = 40000
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randint(0, 256, (N, 24), generator=g, device="cuda").float()
    q = torch.randperm(N, generator=g, device="cuda")[:20000]
    i, d = at.atsne_knn(X, 12, queries=q.int(), precision="bf16_approx")
    at.atsne_check()
    ri, rd = oracle(X, q, 12)
    assert torch.equal(i, ri) and torch.equal(d, rd)


@pytest.mark.parametrize("D", [2, 6, 48, 50, 51, 98, 785])
@pytest.mark.parametrize("offset", [0, 1, 2])
def test_row_widths_and_alignments(at, D, offset):
    """Rows whose widths and first addresses admit 16-byte, 8-byte or 4-byte
    loads, of values that the BF16 copies hold exactly or not."""
    N, k = 1800, 12
    g = torch.Generator(device="cuda").manual_seed(D)
    for top in (256, 1024):
        flat = torch.randint(0, top, (N * D + offset,), generator=g, device="cuda").float()
        X = flat[offset:].view(N, D)
        i, d = at.atsne_knn(X, k, precision="fp32")
        at.atsne_check()
        ri, rd = oracle(X, torch.arange(N, device="cuda"), k)
        assert torch.equal(i, ri)
        assert torch.equal(d, rd) if D * top * top < 2 ** 24 else torch.allclose(d, rd, rtol=(D / 8 + 12) * 2.0 ** -24)
