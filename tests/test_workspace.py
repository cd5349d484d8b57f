"""Workspaces do not grow: a program that keeps a buffer of the size an earlier
version of the library asked for is not refused, and a problem that fitted the
device still fits. Each line: the call, the bytes it asked for then."""
import pytest

SYMMETRIZE = [  # N, k, bytes
    (2, 1, 3328), (40, 32, 23040), (2000, 90, 2938368), (5021, 150, 12192512), (70000, 90, 102761728),
    (300000, 90, 440402176), (1000000, 90, 1468002816), (2097152, 4, 192942848)]


@pytest.fixture(scope="module")
def at():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as pkg
    return pkg


@pytest.mark.parametrize("N,k,was", SYMMETRIZE)
def test_symmetrize(at, N, k, was):
    assert at.workspace_bytes(at.OP_SYMMETRIZE, N, 0, k) <= was
