"""Pixels the tiled walk leaves to the second KNN pass, by what they lack: a
larger buffer (17 - 32 undecided keys) or the unbounded walk (more, or a disk
beyond the offset table). Maps of noise from a spatial term that decides nearly
everything to one that decides nothing, whole frames (probabilities from the
planes and interleaved) and a batch: O and labels as the full search's, bit for
bit."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam", [0.7, 0.45, 0.3, 0.2, 0.05])
@pytest.mark.parametrize("H,W,K,R", [(33, 70, 16, 7), (40, 41, 40, 14), (9, 130, 24, 3)])
def test_left_pixels(hsc, ctx, lam, H, W, K, R):
    import torch
    rng = np.random.default_rng(H + K)
    k, B = 5, 24
    M = k * (k - 1) // 2
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    model = hsc.Model(k, f(rng.standard_normal((M, B))), f(np.zeros(M)), f(-np.ones(M)),
                      f(np.zeros(M)))
    cube = f(rng.random((B, H, W)))
    I, P, O = torch.empty((H, W), device="cuda"), *(torch.empty((k, H, W), device="cuda")
                                                     for _ in range(2))
    ctx.knn_diagnostics()
    lab = hsc.hsc_classify(ctx, cube, model, K, R, lam, out_probs=O, one_band=I, probs=P)
    left = ctx.knn_diagnostics()[1]
    assert lam > 0.1 or left > 0
    ref = torch.empty_like(O)
    rlab = hsc.hsc_knn_filter(ctx, I, P, K, R, lam, out_probs=ref, search=hsc.HSC_KNN_SEARCH_FULL)
    O2 = torch.empty_like(O)
    lab2 = hsc.hsc_knn_filter(ctx, I, P, K, R, lam, out_probs=O2)
    Ob = [torch.empty_like(O) for _ in range(2)]
    labb = hsc.hsc_classify_batch(ctx, [cube, cube], model, K, R, lam, out_probs=Ob)
    ctx.sync()
    for o, x in ((O, lab), (O2, lab2), (Ob[0], labb[0]), (Ob[1], labb[1])):
        assert torch.equal(o, ref)
        assert torch.equal(x, rlab)
