"""The two launch forms of the FP32-pipe covariance at the lines between them
(112 and 176 bands, more partitions than SMs or fewer), against 64-bit
arithmetic; the tolerance is test_gpu_gram_fp32.py's (one FP32 sum per entry
over at most 2048 pixels of a partition: 1e-5 of max|C|)."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 8, 105, 112, 113, 176, 177])
@pytest.mark.parametrize("H,W", [(47, 48), (397, 401)])
def test_forms(hsc, ctx, B, H, W):
    import torch
    g = torch.Generator("cuda").manual_seed(B + H)
    x = 0.5 + 0.1 * torch.randn((B, H, W), generator=g, device="cuda")
    mu, C = hsc.hsc_pca_covariance(ctx, x, flags=hsc.HSC_COV_FP32_PIPE)
    ctx.sync()
    y = x.reshape(B, -1).double()
    mu_ref = y.mean(1)
    y = y - mu_ref[:, None]
    C_ref = y @ y.t() / y.shape[1]
    assert float((mu - mu_ref).abs().max()) < 1e-6
    assert float((C - C_ref).abs().max()) < 1e-5 * float(C_ref.abs().max())
