"""Workspaces do not grow: a program that keeps a buffer of the size an earlier
version of the library asked for is not refused, and a problem that fitted the
device still fits. Each line: the call, the bytes it asked for then."""
import pytest

SYMMETRIZE = [  # N, k, bytes
    (2, 1, 3328), (40, 32, 23040), (2000, 90, 2938368), (5021, 150, 12192512), (70000, 90, 102761728),
    (300000, 90, 440402176), (1000000, 90, 1468002816), (2097152, 4, 192942848)]

KNN = [  # the call, N (of the corpus), D, S (listed or other rows; 0: all), k, precision, bytes
    ("knn", 2000, 64, 0, 90, "fp32", 41968896),
    ("knn", 70000, 784, 0, 90, "fp32", 1705200640),
    ("knn", 50021, 50, 0, 150, "fp32", 1359372032),
    ("knn", 1000000, 128, 0, 90, "bf16_approx", 66916384256),
    ("knn", 200000, 128, 0, 90, "fp32", 4823330048),
    ("knn", 1000000, 128, 0, 90, "fp8", 66760380160),
    ("knn", 1025, 17, 0, 30, "fp32", 14688000),
    ("knn", 800, 784, 0, 90, "bf16", 12465664),
    ("knn", 800, 300, 0, 30, "bf16_approx", 8369664),
    ("knn", 20000, 1500, 0, 30, "fp32", 2282080768),
    ("knn", 60000, 100, 0, 30, "bf16", 727204864),
    ("knn", 4000, 4096, 0, 30, "fp32", 181344768),
    ("knn", 107013, 50, 7013, 90, "fp32", 3178598912),
    ("knn", 100000, 50, 50, 90, "fp32", 77879296),
    ("refine", 70000, 784, 500, 90, None, 590509824),
    ("refine", 500000, 256, 20000, 90, None, 5949041152),
    ("refine", 3000, 32, 200, 30, None, 5308416),
    ("refine_batch", 500000, 256, 270000, 90, None, 8085304320),
    ("refine_batch", 3000, 32, 500, 30, None, 12028160),
    ("refine_batch", 900, 16, 400, 30, None, 3385344),
    ("refine_batch", 50000, 64, 100, 30, None, 44032),
    ("knn_cross", 100000, 50, 2500, 90, "fp32", 2541501440),
    ("knn_cross", 1500, 50, 2500, 20, "fp32", 33675520),
    ("knn_cross_radius", 7013, 50, 100000, 90, "fp32", 236336896),
    ("knn_cross_radius", 7013, 50, 100000, 90, "bf16", 429267712),
    ("knn_cross_radius", 100000, 50, 100000, 90, "fp32", 262001152),
    ("knn_cross_radius", 20000, 50, 20000, 90, "fp32", 592880896),
    ("knn_cross_radius", 500, 16, 3000, 30, "fp32", 7171072)]


@pytest.fixture(scope="module")
def at():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as pkg
    return pkg


@pytest.mark.parametrize("N,k,was", SYMMETRIZE)
def test_symmetrize(at, N, k, was):
    assert at.workspace_bytes(at.OP_SYMMETRIZE, N, 0, k) <= was


def check_knn(at, call, N, D, S, k, precision, was):
    opts = at.knn_opts(precision=precision) if precision else None
    assert at.workspace_bytes(getattr(at, "OP_" + call.upper()), N, D, k, S, opts) <= was


@pytest.mark.parametrize("call,N,D,S,k,precision,was", KNN)
def test_knn(at, call, N, D, S, k, precision, was):
    check_knn(at, call, N, D, S, k, precision, was)


@pytest.mark.gpu  # the plans count the device's SMs
@pytest.mark.parametrize("call,N,D,S,k,precision,was", KNN)
def test_knn_on_the_device(at, call, N, D, S, k, precision, was):
    check_knn(at, call, N, D, S, k, precision, was)
