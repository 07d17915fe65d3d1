"""The tiled pruned walk (compile-time disk patterns, the shell picked in
registers, border pixels and undecided lanes by themselves) against the
full-window search, which keys every candidate: the same O and labels bit for
bit, where the tiles have edges and remainders, at each of the 13 shells that
K <= 64 can end in, and on maps that leave many keys undecided."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one K in each shell s_K = 0, 1, 2, 4, 5, 8, 9, 10, 13, 16, 17, 18, 20
SHELL_KS = (1, 4, 9, 12, 16, 24, 28, 33, 40, 47, 50, 60, 64)


def maps(kind, H, W, k, seed):
    rng = np.random.default_rng(seed)
    if kind == "smooth":  # every pixel decided by the shell
        I = 0.5 + 0.1 * rng.random((H, W))
    elif kind == "steps":  # jumps beside flat parts: undecided lanes, exact ties
        I = np.where(rng.random((H, W)) < 0.02, 1.0, 0.0) + np.round(rng.random((H, W)) * 8) / 64
    else:  # raw scale: e far above the shells' steps
        I = 40.0 * rng.random((H, W))
    P = rng.random((k, H, W))
    return I.astype(np.float32), (P / P.sum(axis=0)).astype(np.float32)


def both(hsc, ctx, I, P, K, R, lam):
    import torch
    It, Pt = torch.as_tensor(I, device="cuda"), torch.as_tensor(P, device="cuda")
    out = []
    for search in (hsc.HSC_KNN_SEARCH_PRUNED, hsc.HSC_KNN_SEARCH_FULL):
        O = torch.full_like(Pt, -1.0)
        lab = torch.full(It.shape, -1, dtype=torch.int32, device="cuda")
        hsc.hsc_knn_filter(ctx, It, Pt, K, R, lam, out_probs=O, labels=lab, search=search)
        ctx.sync()
        out.append((O.cpu().numpy(), lab.cpu().numpy()))
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("K", SHELL_KS)
@pytest.mark.parametrize("kind", ["smooth", "steps"])
def test_every_shell(hsc, ctx, K, kind):
    I, P = maps(kind, 27, 71, 4, K)
    both(hsc, ctx, I, P, K, 14, 1.0)


@pytest.mark.parametrize("H,W", [(8, 7), (9, 40), (10, 33), (11, 31), (12, 64), (7, 65), (64, 7)])
def test_tile_edges(hsc, ctx, H, W):
    """K = 40 reaches 3 rows and columns: maps with no tile, one row group,
    an odd row left over, one column inside, partial column tiles."""
    I, P = maps("smooth", H, W, 3, H * W)
    both(hsc, ctx, I, P, 40 if min(7, H) * W >= 40 else 16, 14, 1.0)


@pytest.mark.parametrize("k", [1, 2, 5, 7, 8])
def test_class_counts(hsc, ctx, k):
    I, P = maps("steps", 21, 50, k, k)
    both(hsc, ctx, I, P, 24, 9, 0.5)


@pytest.mark.parametrize("kind", ["smooth", "steps", "raw"])
@pytest.mark.parametrize("K,R,lam", [(40, 5, 1.0), (64, 3, 1.0), (40, 14, 0.25), (9, 6, 2.0),
                                     (24, 9, 0.5), (16, 7, 1e-3), (16, 7, 3e5)])
def test_cut_windows_and_lambdas(hsc, ctx, kind, K, R, lam):
    I, P = maps(kind, 26, 45, 4, K + R)
    both(hsc, ctx, I, P, K, R, lam)
