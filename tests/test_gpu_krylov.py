"""The Krylov eigensolver (default form, up to 256 bands) where its shapes
have edges: fewer bands than Krylov steps, band counts around a warp, around
the one-CTA form's 128 and the cluster's rows of 32, and spectra it leaves to
the full kernel. The bound is the eigensolver's own: ||C v - lambda v|| <=
2e-13 ||C|| on the GPU's FP64 covariance, lambda its largest eigenvalue."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cube_of(spectrum, seed, H=40, W=50):
    """x_p = 0.5 + 0.02 sum_j sqrt(l_j) z_jp q_j: sample covariance near the
    spectrum's, in random directions."""
    rng = np.random.default_rng(seed)
    B = len(spectrum)
    Q, _ = np.linalg.qr(rng.standard_normal((B, B)))
    z = rng.standard_normal((B, H * W))
    x = 0.5 + 0.02 * (Q * np.sqrt(spectrum)) @ z
    return x.reshape(B, H, W).astype(np.float32)


def check(hsc, ctx, cube):
    import torch
    B, H, W = cube.shape
    c = torch.as_tensor(cube, device="cuda")
    v = torch.zeros(B, dtype=torch.float64, device="cuda")
    lam = torch.zeros(1, dtype=torch.float64, device="cuda")
    I = hsc.hsc_pca_one_band(ctx, c, flags=0, eigvec=v, eigval=lam)
    _, C = hsc.hsc_pca_covariance(ctx, c)
    ctx.sync()
    v, lam, C, I = v.cpu().numpy(), float(lam.cpu()[0]), C.cpu().numpy(), I.cpu().numpy()
    cn = max(abs(lam), np.abs(np.diag(C)).max())
    assert abs(np.linalg.norm(v) - 1.0) < 1e-14
    assert v[np.abs(v).argmax()] > 0
    assert np.linalg.norm(C @ v - lam * v) <= 2e-13 * cn
    assert abs(lam - np.linalg.eigvalsh(C).max()) <= 1e-12 * cn
    ref = np.tensordot(v, cube.astype(np.float64) - cube.mean(axis=(1, 2), dtype=np.float64)[:, None, None], 1)
    assert np.abs(I - ref).max() < 2e-5 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("B", [1, 2, 3, 9, 10, 11, 31, 32, 33, 64, 127, 128, 129, 159, 160, 161,
                               224, 255, 256])
def test_band_counts(hsc, ctx, B):
    lam = np.full(B, 1e-3)
    lam[:4] = [1.0, 0.5, 0.2, 0.05][:min(4, B)]
    check(hsc, ctx, cube_of(lam, B))


@pytest.mark.parametrize("B", [48, 128, 160])
def test_spectra_left_to_the_full_kernel(hsc, ctx, B):
    """Eigenvalues evenly spaced down from 1: 10 steps do not separate the
    first; the guarded kernel finishes the frame, and the next frame is the
    Krylov form's again."""
    check(hsc, ctx, cube_of(np.linspace(1.0, 0.02, B), 3 * B, 80, 100))
    lam = np.full(B, 1e-3)
    lam[0] = 1.0
    check(hsc, ctx, cube_of(lam, B))


@pytest.mark.parametrize("B", [16, 200])
def test_constant_cube(hsc, ctx, B):
    """C = 0 is the full kernel's: a unit vector and a zero image."""
    import torch
    c = torch.full((B, 12, 16), 0.25, device="cuda")
    v = torch.zeros(B, dtype=torch.float64, device="cuda")
    I = hsc.hsc_pca_one_band(ctx, c, eigvec=v)
    ctx.sync()
    assert float(I.abs().max()) == 0.0
    assert abs(float(v.norm()) - 1.0) < 1e-14
