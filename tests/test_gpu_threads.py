"""Calls of different sizes from two threads, each on its own stream: a launch's
shared memory is not refused for what the other thread's call asked for, and the
results are those of one thread."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def at():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as pkg
    return pkg


def run_threads(calls, repeats=1500):
    """calls[i]() many times in thread i, on its own stream; the errors, and each call's last results."""
    errors, results, start = [], [None] * len(calls), threading.Barrier(len(calls))

    def work(i):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            with torch.cuda.stream(stream):
                for _ in range(repeats):
                    results[i] = calls[i]()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors, results


def check(at, calls):
    want = [[t.clone() for t in c()] for c in calls]
    torch.cuda.synchronize()
    errors, got = run_threads(calls)
    assert not errors, errors
    at.atsne_check()
    for w, g in zip(want, got):
        assert all(torch.equal(a, b) for a, b in zip(w, g))


def test_symmetrize(at):
    def call(N, k=2):
        i = torch.arange(N, device="cuda")
        idx = torch.stack([(i + 1) % N, (i + 2) % N], 1).int().contiguous()
        P = torch.rand((N, k), device="cuda")
        out = (torch.empty(N + 1, dtype=torch.int64, device="cuda"), torch.zeros(2 * N * k, dtype=torch.int32, device="cuda"),
               torch.zeros(2 * N * k, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda"))
        ws = torch.empty(at.workspace_bytes(at.OP_SYMMETRIZE, N, 0, k), dtype=torch.uint8, device="cuda")
        return lambda: at.atsne_symmetrize(idx, P, trim=False, out=out, workspace=ws)

    check(at, [call(300), call(600000)])


@pytest.mark.parametrize("N", [1500, 400])  # a row of the merge by a warp, and by a block
def test_approximate_knn(at, N):
    X = torch.randn((2000, 16), device="cuda")
    queries = torch.arange(N, dtype=torch.int32, device="cuda")

    def call(k):
        opts = at.knn_opts(precision="bf16_approx")
        return lambda: at.atsne_knn(X, k, queries=queries, opts=opts)

    check(at, [call(10), call(100)])
