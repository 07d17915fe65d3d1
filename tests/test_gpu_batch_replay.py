"""The batch graph is replayed only for the launches it holds. Two batches of
more frames than SMs that agree in every sum over their frames (Gram and
projection items, KNN CTAs, scratch offsets) but not in the second group's
pixel count: a replay would keep the first one's room for pixels left to the
second KNN pass, and drop the last of them. lambda is so small that every
pixel is left to it."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_replay_needs_the_same_second_group(hsc, ctx):
    import torch
    B, H, W0, W1, k, K, R, lam = 16, 4, 17, 20, 4, 8, 4, 0.003
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    # the redo list (8 bytes per pixel) ends within the same 256 bytes for both
    n = next(n for n in range(sm + 1, sm + 33)
             if (8 * H * (W0 * n + W1 - W0) - 1) // 256 == (8 * H * W0 * n - 1) // 256)
    rng = np.random.default_rng(5)
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    M = k * (k - 1) // 2
    model = hsc.Model(k, f(rng.standard_normal((M, B))), f(np.zeros(M)), f(-np.ones(M)),
                      f(np.zeros(M)))
    with hsc.Context(0, stream=torch.cuda.current_stream()) as c:
        for last in (W0, W1):
            cubes = [f(rng.random((B, H, w))) for w in [W0] * (n - 1) + [last]]
            O = [torch.zeros((k,) + tuple(x.shape[1:]), device="cuda") for x in cubes]
            labels = hsc.hsc_classify_batch(c, cubes, model, K, R, lam,
                                            flags=hsc.HSC_BATCH_GRAPH, out_probs=O)
            c.sync()
            for i in (0, sm - 1, sm, n - 1):
                Oi = torch.zeros_like(O[i])
                li = hsc.hsc_classify(ctx, cubes[i], model, K, R, lam, out_probs=Oi)
                ctx.sync()
                assert torch.equal(labels[i], li), (last, i)
                assert torch.equal(O[i], Oi), (last, i)
