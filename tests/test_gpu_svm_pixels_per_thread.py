"""hsc_svm_probs where its pixels per thread change with the pixel count: the
sizes around each line, with and without 16-byte loads, for every class count.
A pixel's arithmetic does not depend on the grouping, so a frame's rows give
the same bits as the same rows in a frame of one pixel per thread (under
65536); both couplings."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("H,W", [(255, 257), (256, 256), (257, 256), (255, 385), (256, 384),
                                 (257, 385), (64, 3001)])
def test_same_bits_as_one_pixel_per_thread(hsc, ctx, k, H, W):
    import torch
    B, M = 19, k * (k - 1) // 2
    rng = np.random.default_rng(H * W + k)
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    model = hsc.Model(k, f(rng.standard_normal((M, B))), f(0.1 * rng.standard_normal(M)),
                      f(-np.ones(M)), f(np.zeros(M)))
    x = torch.rand((B, H, W), generator=torch.Generator("cuda").manual_seed(k), device="cuda")
    for flags in (0, hsc.HSC_SVM_COUPLE_F64):
        L = torch.full((H, W), -1, dtype=torch.int32, device="cuda")
        P = hsc.hsc_svm_probs(ctx, x, model, flags=flags, svm_labels=L)
        rows = 16384 // W
        for r in range(0, H, rows):
            r1 = min(H, r + rows)
            Ls = torch.full((r1 - r, W), -1, dtype=torch.int32, device="cuda")
            Ps = hsc.hsc_svm_probs(ctx, x[:, r:r1].contiguous(), model, flags=flags,
                                   svm_labels=Ls)
            assert torch.equal(P[:, r:r1], Ps), (flags, r)
            assert torch.equal(L[r:r1], Ls), (flags, r)
    ctx.sync()
