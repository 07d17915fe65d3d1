"""Further components of frames whose basis the eigensolver could not refine
(the full Jacobi fallback): refined from the fallback's own columns. The bound
is the one of the other components (||C v - lambda v|| <= 2e-13 ||C||, lambda_j
the j-th largest eigenvalue)."""

import numpy as np
import pytest

from test_gpu_krylov_restart import exact_spectrum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [128, 160, 200, 272])
def test_components_after_the_fallback(hsc, ctx, B):
    import torch
    c = torch.as_tensor(exact_spectrum(np.linspace(1.0, 0.02, B), B), device="cuda")
    n = 4
    V = torch.zeros((n, B), dtype=torch.float64, device="cuda")
    L = torch.zeros(n, dtype=torch.float64, device="cuda")
    hsc.hsc_pca_project(ctx, c, n, eigvecs=V, eigvals=L)
    _, C = hsc.hsc_pca_covariance(ctx, c)
    ctx.sync()
    assert ctx.pca_diagnostics()[0] > 1  # the fallback's sweeps
    V, L, C = V.cpu().numpy(), L.cpu().numpy(), C.cpu().numpy()
    top = np.linalg.eigvalsh(C)[::-1]
    for j in range(n):
        assert abs(np.linalg.norm(V[j]) - 1.0) < 1e-14, j
        assert np.linalg.norm(C @ V[j] - L[j] * V[j]) <= 2e-13 * top[0], j
        assert abs(L[j] - top[j]) <= 1e-12 * top[0], j
