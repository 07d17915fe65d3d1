"""Tensor-core Gram of frames the tensor map cannot describe (N % 4 != 0, or a
cube that does not start on a 16-byte boundary): 16-byte copies of the units
around each band row's pixels, shifted when they are converted."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def covariance(hsc, ctx, cube, offset):
    """Covariance of the cube placed ``offset`` floats past an aligned address,
    NaN in front of it and behind it."""
    import torch
    flat = torch.full((cube.size + 8,), float("nan"), dtype=torch.float32, device="cuda")
    view = flat[offset:offset + cube.size].view(cube.shape)
    view.copy_(torch.as_tensor(np.ascontiguousarray(cube), device="cuda"))
    mu, C = hsc.hsc_pca_covariance(ctx, view)
    ctx.sync()
    return mu.cpu().numpy(), C.cpu().numpy()


# sizes around the 64-pixel chunk, the 4-pixel unit, several chunks per CTA,
# one band row per group of copies and the largest band count
@pytest.mark.parametrize("B,H,W", [(1, 1, 4), (3, 2, 2), (8, 4, 16), (9, 4, 17), (31, 6, 10),
                                   (100, 33, 36), (128, 16, 68), (127, 200, 208)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_cube_same_bits(hsc, ctx, B, H, W, offset):
    """The same chunks reach the same accumulators in the same order, so an
    unaligned cube has the aligned one's covariance bit for bit."""
    cube = synth.make_frame(B + H, H, W, B, sigma=0.03).cube
    mu0, C0 = covariance(hsc, ctx, cube, 0)
    mu, C = covariance(hsc, ctx, cube, offset)
    np.testing.assert_array_equal(mu, mu0)
    np.testing.assert_array_equal(C, C0)


@pytest.mark.parametrize("B,H,W", [(2, 1, 2), (5, 1, 3), (16, 1, 65), (17, 1, 67), (33, 7, 9),
                                   (125, 41, 41), (128, 51, 61), (100, 203, 301)])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_ragged_frame(hsc, ctx, B, H, W, offset):
    """N % 4 != 0 against 64-bit arithmetic; tolerance: FP32 sums of 1024 and
    more pixels per partial and the FP16 hi/lo split, 1e-5 of max|C|."""
    cube = synth.make_frame(B + W, H, W, B, sigma=0.03).cube
    x = cube.reshape(B, -1).astype(np.float64)
    mu_ref = x.mean(1)
    d = x - mu_ref[:, None]
    C_ref = d @ d.T / x.shape[1]
    mu, C = covariance(hsc, ctx, cube, offset)
    np.testing.assert_allclose(mu, mu_ref, atol=1e-6)
    np.testing.assert_allclose(C, C_ref, rtol=0, atol=1e-5 * np.abs(C_ref).max())
