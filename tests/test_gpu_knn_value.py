"""The KNN filter without a spatial term (lambda = 0: the window sorted by
value) against the heap search, which keys every candidate: the same
neighbours in the same order, O and labels bit for bit, on maps with exact
ties, equal rounded distances of different values, one value only, and
negative values; windows from one row to the largest the sort takes."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def maps(kind, H, W, k, seed):
    rng = np.random.default_rng(seed)
    I = rng.random((H, W))
    if kind == "grey":  # 9 levels: ties by index, both sides at one distance
        I = np.round(I * 8) / 8
    elif kind == "flat":
        I = np.full((H, W), 0.25)
    elif kind == "tiny":  # many values at one rounded distance from the large ones
        I = np.where(rng.random((H, W)) < 0.5, 1e-9 * I, 0.75 + I)
    elif kind == "signed":
        I = (I - 0.5) * 3
        I[0, 0] = -0.0
        I[0, 1] = 0.0
    P = rng.random((k, H, W))
    return I.astype(np.float32), (P / P.sum(axis=0)).astype(np.float32)


@pytest.mark.parametrize("kind", ["random", "grey", "flat", "tiny", "signed"])
@pytest.mark.parametrize("H,W,K,R,k", [(1, 70, 5, 1, 4), (2, 2, 4, 7, 1), (9, 33, 16, 7, 4),
                                       (14, 64, 64, 32, 8), (20, 513, 40, 14, 3)])
def test_value_order_equals_heap(hsc, ctx, kind, H, W, K, R, k):
    import torch
    K = min(K, min((R + 1) // 2, H) * W)
    I, P = maps(kind, H, W, k, H * W + K)
    It, Pt = torch.as_tensor(I, device="cuda"), torch.as_tensor(P, device="cuda")
    out = []
    for search in (hsc.HSC_KNN_SEARCH_AUTO, hsc.HSC_KNN_SEARCH_HEAP):
        O = torch.full_like(Pt, -1.0)
        lab = torch.full((H, W), -1, dtype=torch.int32, device="cuda")
        nbr = torch.full((H, W, K), -2, dtype=torch.int32, device="cuda")
        hsc.hsc_knn_filter(ctx, It, Pt, K, R, 0.0, out_probs=O, labels=lab, nbr_idx=nbr,
                           search=search)
        ctx.sync()
        out.append([t.cpu().numpy() for t in (nbr, O, lab)])
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
