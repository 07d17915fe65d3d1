"""The KNN filter without a spatial term at the edges of its value sort:
windows of exactly the largest size it sorts (128 KB of shared memory) and one
above (the full scan), maps whose squared distances underflow to zero or
overflow to infinity for most of the window (one group of many values), and
maps with NaN or infinite entries. Against the heap search, bit for bit (where
its keys overflow too, against a sort by (squared distance, index))."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(hsc, ctx, I, P, K, R, search):
    import torch
    k, H, W = P.shape
    O = torch.full((k, H, W), -1.0, device="cuda")
    lab = torch.full((H, W), -1, dtype=torch.int32, device="cuda")
    nbr = torch.full((H, W, K), -2, dtype=torch.int32, device="cuda")
    hsc.hsc_knn_filter(ctx, I, P, K, R, 0.0, out_probs=O, labels=lab, nbr_idx=nbr, search=search)
    ctx.sync()
    return O, lab, nbr


def by_value(I, K, R):
    H, W = I.shape
    out = np.empty((H, W, K), dtype=np.int32)
    for r in range(H):
        lo, hi = max(0, r - R // 2), min(H, r + (R + 1) // 2)
        win = I[lo:hi].reshape(-1)
        with np.errstate(over="ignore"):
            e = (I[r][:, None] - win[None]) ** 2
        out[r] = lo * W + np.argsort(e, axis=1, kind="stable")[:, :K]
    return out


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def probs(rng, k, H, W):
    P = rng.random((k, H, W))
    return dev(P / P.sum(axis=0))


@pytest.mark.parametrize("H,W,R", [(17, 1024, 16),   # 16384 candidates: the largest sorted
                                   (16, 1025, 16),   # 16400: the scan
                                   (4, 4096, 4), (6, 4096, 5)])
def test_largest_windows(hsc, ctx, H, W, R):
    import torch
    rng = np.random.default_rng(W)
    I, P = dev(rng.random((H, W))), probs(rng, 3, H, W)
    a = run(hsc, ctx, I, P, 12, R, hsc.HSC_KNN_SEARCH_AUTO)
    b = run(hsc, ctx, I, P, 12, R, hsc.HSC_KNN_SEARCH_HEAP)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


MAPS = {
    "underflow": lambda rng, s: 1e-24 * rng.random(s),
    "overflow": lambda rng, s: 1e20 * rng.standard_normal(s),
    "half": lambda rng, s: np.where(rng.random(s) < 0.5, 1e-24, 1.0) * rng.random(s),
    "far": lambda rng, s: np.where(rng.random(s) < 0.02, 0.0, 1e8 + rng.random(s)),
}


@pytest.mark.parametrize("kind", list(MAPS))
@pytest.mark.parametrize("H,W,K,R", [(1, 700, 9, 1), (20, 300, 40, 14), (11, 64, 64, 7)])
def test_one_group_of_many_values(hsc, ctx, kind, H, W, K, R):
    import torch
    rng = np.random.default_rng(K)
    I, P = dev(MAPS[kind](rng, (H, W))), probs(rng, 4, H, W)
    a = run(hsc, ctx, I, P, K, R, hsc.HSC_KNN_SEARCH_AUTO)
    if kind == "overflow":
        np.testing.assert_array_equal(a[2].cpu().numpy(), by_value(I.cpu().numpy(), K, R))
        return
    b = run(hsc, ctx, I, P, K, R, hsc.HSC_KNN_SEARCH_HEAP)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


def test_many_values_in_one_group_take_no_longer(hsc, ctx):
    """A pixel of such a group stops at its K-th index, as the others do at
    their K-th value: within a factor of 10 of an ordinary map's time (it was
    230 when each pixel ran through the group)."""
    import torch
    rng = np.random.default_rng(3)
    H, W = 1, 4096
    P = probs(rng, 4, H, W)
    us = []
    for kind in (lambda s: rng.random(s), lambda s: 1e-24 * rng.random(s)):
        I = dev(kind((H, W)))
        t = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            hsc.hsc_knn_filter(ctx, I, P, 16, 7, 0.0)
            b.record()
            ctx.sync()
            t.append(a.elapsed_time(b))
        us.append(min(t))
    assert us[1] < 10 * us[0], us


@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf])
def test_nonfinite_maps_are_reported(hsc, ctx, bad):
    rng = np.random.default_rng(1)
    H, W = 12, 90
    I = rng.random((H, W)).astype(np.float32)
    I[5, 7:20] = bad
    P = probs(rng, 4, H, W)
    with pytest.raises(hsc.HscError) as e:
        run(hsc, ctx, dev(I), P, 24, 7, hsc.HSC_KNN_SEARCH_AUTO)
    assert e.value.status == hsc.HSC_ERR_NONFINITE
    run(hsc, ctx, dev(rng.random((H, W))), P, 24, 7, hsc.HSC_KNN_SEARCH_AUTO)
