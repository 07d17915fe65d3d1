"""The pairwise coupling solve on pairwise probabilities known exactly: with
decision values of -1000, 0 and 1000 every r_ij is one of the two clips or
1/2, so the FP64 solution of the same system can be compared digit by digit.
HSC_SVM_COUPLE_F64 (FP32 factors, one double-float correction): its error
before the result is rounded to FP32 is below 1e-11 (condition number < 25),
so each p is within one rounding, 2^-24 relative, and 1e-11 of the FP64 one.
The FP32 solve: 25 x 2^-24 x a small factor."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reference(r, k):
    """(Q + e e^T) y = e, p = y / sum y in FP64; r: pixels x M (float32)."""
    n = r.shape[0]
    R = np.zeros((n, k, k))
    m = 0
    for i in range(k):
        for j in range(i + 1, k):
            R[:, i, j] = r[:, m]
            R[:, j, i] = 1.0 - r[:, m]
            m += 1
    A = 1.0 - np.swapaxes(R, 1, 2) * R
    for i in range(k):
        A[:, i, i] = 1.0 + (R[:, :, i] ** 2).sum(axis=1)
    y = np.linalg.solve(A, np.ones((n, k, 1)))[..., 0]
    return y / y.sum(axis=1, keepdims=True)


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8])
def test_exact_pairwise_probabilities(hsc, ctx, k):
    import torch
    M = k * (k - 1) // 2
    H, W = 13, 37
    rng = np.random.default_rng(k)
    x = rng.integers(-1, 2, (M, H, W)).astype(np.float32)
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    model = hsc.Model(k, f(1000 * np.eye(M)), f(np.zeros(M)), f(-np.ones(M)), f(np.zeros(M)))
    lo = np.float32(1e-7)
    r = np.choose(x.reshape(M, -1).T.astype(int) + 1, [lo, np.float32(0.5), np.float32(1) - lo])
    ref = reference(r.astype(np.float64), k)
    for flags, rel, tol in ((hsc.HSC_SVM_COUPLE_F64, 2.0 ** -24, 1e-11), (0, 1e-5, 1e-5)):
        P = hsc.hsc_svm_probs(ctx, f(x), model, flags=flags)
        ctx.sync()
        err = np.abs(P.cpu().numpy().reshape(k, -1).T.astype(np.float64) - ref)
        assert (err <= rel * np.abs(ref) + tol).all(), (flags, err.max())
