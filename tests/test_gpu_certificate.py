"""The certified one-pass BF16 kNN on values that BF16 rounds by its full unit
roundoff (2^-8): neighbours closer together than the rounding, where a bound on
the key error that is too small would certify wrong lists (Eq. 8, against the
oracle)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [10, 90])
def test_certified_bf16_lists_of_values_between_bf16_numbers(k):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1512_01655_gb300 as at
    X = np.repeat(np.arange(6000, dtype=np.float32)[:, None], 3, axis=1)
    idx, d2 = at.atsne_knn(torch.from_numpy(X).cuda(), k, precision="bf16")
    at.atsne_check()
    rows = np.arange(200, 5800, 7, dtype=np.int32)
    o_idx, o_d2 = oracle.knn_exact(X, k, queries=rows)
    # squared distances are integers below 2^24: exact in FP32, ties by index
    assert np.array_equal(idx.cpu().numpy()[rows], o_idx)
    assert np.array_equal(d2.cpu().numpy()[rows].astype(np.float64), o_d2)
