"""The tiled KNN reading the pixel-interleaved probabilities (hsc_classify and
hsc_classify_batch) for every class count: O and labels bit for bit as the full
search gives them on the I and P the call returns. Maps with tiles and border,
smaller than a tile, cut by the window, and of few levels (ties)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("H,W,K,R,lam,levels", [(45, 77, 40, 14, 1.0, 0), (33, 31, 16, 7, 0.5, 0),
                                                (9, 40, 24, 3, 1.0, 0), (52, 64, 24, 9, 0.3, 5),
                                                (6, 7, 12, 4, 2.0, 3)])
def test_classify_equals_full_search(hsc, ctx, k, H, W, K, R, lam, levels):
    import torch
    B, M = 17, k * (k - 1) // 2
    rng = np.random.default_rng(10 * k + H)
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    model = hsc.Model(k, f(rng.standard_normal((M, B))), f(0.2 * rng.standard_normal(M)),
                      f(-2 * np.ones(M)), f(np.zeros(M)))
    cubes = []
    for h, w in ((H, W), (H + 1, W + 3)):
        t = rng.random((h, w))
        if levels:
            t = np.round(t * levels) / levels
        cubes.append(f(t[None] * rng.random((B, 1, 1)) + (0 if levels else 0.05 * rng.random((B, h, w)))))
    ref = []
    for c in cubes:
        h, w = c.shape[1:]
        I, P = torch.empty((h, w), device="cuda"), torch.empty((k, h, w), device="cuda")
        O = torch.full((k, h, w), -1.0, device="cuda")
        lab = hsc.hsc_classify(ctx, c, model, K, R, lam, out_probs=O, one_band=I, probs=P)
        Of = torch.full_like(O, -2.0)
        labf = hsc.hsc_knn_filter(ctx, I, P, K, R, lam, out_probs=Of,
                                  search=hsc.HSC_KNN_SEARCH_FULL)
        ctx.sync()
        assert torch.equal(O, Of)
        assert torch.equal(lab, labf)
        ref.append((lab, O))
    Ob = [torch.full_like(o, -3.0) for _, o in ref]
    labs = hsc.hsc_classify_batch(ctx, cubes, model, K, R, lam, out_probs=Ob)
    ctx.sync()
    for (lab, O), lb, ob in zip(ref, labs, Ob):
        assert torch.equal(lab, lb)
        assert torch.equal(O, ob)
