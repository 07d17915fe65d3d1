"""Covariance on the FP32 pipe (129-256 bands with N % 32 != 0, more than 256
bands, HSC_COV_FP32_PIPE) around the edges of its tiles and chunks."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# bands: one tile, tiles cut at 8, the largest whose next chunk is loaded
# ahead, the first above, sums of more bands than threads; pixels: under a
# chunk of 32, across chunks, several partitions
@pytest.mark.parametrize("B,H,W", [(3, 5, 7), (129, 9, 7), (136, 33, 31), (255, 41, 43),
                                   (256, 40, 41), (257, 11, 13), (300, 20, 53), (577, 9, 10)])
def test_fp32_pipe_covariance(hsc, ctx, B, H, W):
    """Against 64-bit arithmetic; tolerance: one FP32 sum per entry over at most
    2048 pixels of a partition, 2048 * 2^-24 = 1.2e-4 of max|C| at worst, with
    roundings of random sign 45 * 2^-24 = 3e-6: 1e-5."""
    import torch
    cube = synth.make_frame(B + H, H, W, B, sigma=0.03).cube
    x = cube.reshape(B, -1).astype(np.float64)
    mu_ref = x.mean(1)
    d = x - mu_ref[:, None]
    C_ref = d @ d.T / x.shape[1]
    mu, C = hsc.hsc_pca_covariance(ctx, torch.as_tensor(np.ascontiguousarray(cube), device="cuda"),
                                   flags=hsc.HSC_COV_FP32_PIPE)
    ctx.sync()
    np.testing.assert_allclose(mu.cpu().numpy(), mu_ref, atol=1e-6)
    np.testing.assert_allclose(C.cpu().numpy(), C_ref, rtol=0, atol=1e-5 * np.abs(C_ref).max())
