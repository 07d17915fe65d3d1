"""The Krylov eigensolver's restarts: which form finished a frame is read from
hsc_pca_diagnostics (sweeps 0, or 1 above 128 bands: the Krylov form alone; one
more and above: the full kernel behind it). The eigenpair's bounds are
test_gpu_krylov.check's."""

import numpy as np
import pytest

from test_gpu_krylov import check, cube_of

pytestmark = pytest.mark.gpu


def krylov_sweeps(B):
    return 0 if B <= 128 else 1


def exact_spectrum(lam, seed, H=40, W=50):
    """As cube_of, the sample covariance's eigenvalues lam themselves."""
    rng = np.random.default_rng(seed)
    B = len(lam)
    Q, _ = np.linalg.qr(rng.standard_normal((B, B)))
    z = rng.standard_normal((H * W, B))
    z, _ = np.linalg.qr(z - z.mean(axis=0))
    x = 0.5 + 0.02 * (Q * np.sqrt(lam)) @ z.T * np.sqrt(H * W)
    return x.reshape(B, H, W).astype(np.float32)


@pytest.mark.parametrize("B", [40, 128, 129, 200, 256])
@pytest.mark.parametrize("decay", ["exp5", "exp8", "exp12", "exp20", "sqrt"])
def test_decaying_spectra(hsc, ctx, B, decay):
    """Gaps of 5% and more at the top and no flat floor: restarts, not the
    full kernel."""
    j = np.arange(B)
    lam = 1.0 / np.sqrt(1.0 + j) if decay == "sqrt" else np.exp(-j / float(decay[3:]))
    check(hsc, ctx, cube_of(lam, 7 * B, 100, 120))
    assert ctx.pca_diagnostics()[0] == krylov_sweeps(B)


@pytest.mark.parametrize("seed,n", [(1194, 59), (1245, 60), (7, 47)])
def test_pivots_stay_positive(hsc, ctx, seed, n):
    """Four strong directions over a flat floor; at the first two the pivots of
    theta I - T at T's own eigenvalue were negative before the last one."""
    lam = np.full(125, 1e-3)
    lam[:4] = 1.0 / (1.0 + np.arange(4)) ** 2
    check(hsc, ctx, cube_of(lam, seed, n, n))
    assert ctx.pca_diagnostics()[0] == 0


@pytest.mark.parametrize("B", [48, 128, 160, 200])
def test_cluster_goes_to_the_full_kernel(hsc, ctx, B):
    """14 eigenvalues 1e-5 apart: FP32 steps cannot tell them apart, the full
    kernel takes the frame, and the next frame is the Krylov form's again."""
    lam = np.full(B, 1e-3)
    lam[:14] = 1.0 - 1e-5 * np.arange(14)
    check(hsc, ctx, exact_spectrum(lam, B))
    assert ctx.pca_diagnostics()[0] > krylov_sweeps(B)
    lam[1:] = 1e-3
    check(hsc, ctx, cube_of(lam, B))
    assert ctx.pca_diagnostics()[0] == krylov_sweeps(B)


@pytest.mark.parametrize("B,spread,m", [(48, 3e-5, 12), (128, 5e-5, 14)])
def test_components_of_a_frame_left(hsc, ctx, B, spread, m):
    """Two components of a frame that the Krylov form leaves: the lead is not
    its, both are the full kernel's (bound as check's)."""
    import torch
    lam = np.full(B, 1e-4)
    lam[:m] = 1.0 - spread * np.arange(m)
    c = torch.as_tensor(exact_spectrum(lam, B), device="cuda")
    hsc.hsc_pca_one_band(ctx, c)
    assert ctx.pca_diagnostics()[0] > 0
    V = torch.zeros((2, B), dtype=torch.float64, device="cuda")
    L = torch.zeros(2, dtype=torch.float64, device="cuda")
    hsc.hsc_pca_project(ctx, c, 2, eigvecs=V, eigvals=L)
    _, C = hsc.hsc_pca_covariance(ctx, c)
    ctx.sync()
    V, L, C = V.cpu().numpy(), L.cpu().numpy(), C.cpu().numpy()
    top = np.linalg.eigvalsh(C)[::-1]
    for j in range(2):
        assert np.linalg.norm(C @ V[j] - L[j] * V[j]) <= 2e-13 * top[0]
        assert abs(L[j] - top[j]) <= 1e-12 * top[0]
