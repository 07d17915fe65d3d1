"""HSC_SVM_COUPLE_F64 for classes of small probability: each p against the
exact rational solution of the same system. The error of the refined solve
before its rounding to FP32 is below 2^-34 of p itself (two corrections of six
digits each, every term of a row as small as its class's y), so p is within
one rounding: 2^-24 |p| (1 + 2^-10). The pairwise probabilities are exact too:
with two classes p = (r, 1 - r), so the FP32 r comes back as p."""

from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def exact(r, k):
    """(Q + e e^T) y = e, p = y / sum y in rational arithmetic; r: M floats."""
    R = [[Fraction(0)] * k for _ in range(k)]
    m = 0
    for i in range(k):
        for j in range(i + 1, k):
            R[i][j] = Fraction(float(r[m]))
            R[j][i] = 1 - R[i][j]
            m += 1
    A = [[1 + sum(R[t][i] ** 2 for t in range(k)) if i == j else 1 - R[j][i] * R[i][j]
          for j in range(k)] + [Fraction(1)] for i in range(k)]
    for i in range(k):
        for t in range(i + 1, k):
            g = A[t][i] / A[i][i]
            A[t] = [a - g * b for a, b in zip(A[t], A[i])]
    y = [Fraction(0)] * k
    for i in reversed(range(k)):
        y[i] = (A[i][k] - sum(A[i][j] * y[j] for j in range(i + 1, k))) / A[i][i]
    s = sum(y)
    return [float(v / s) for v in y]


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("scores", ["normal", "ties", "any"])
def test_small_probabilities(hsc, ctx, k, scores):
    import torch
    M = k * (k - 1) // 2
    H, W = 4, 11
    rng = np.random.default_rng(100 * k + len(scores))
    # decision values of a consistent ranking (losing classes have p down to
    # 1e-8), of one with ties and clipped pairs, and of none
    s = rng.normal(0, 6.0, (k, H, W)) if scores == "normal" else 100.0 * rng.integers(0, 3, (k, H, W))
    pairs = [(i, j) for i in range(k) for j in range(i + 1, k)]
    x = (rng.normal(0, 4.0, (M, H, W)) if scores == "any"
         else np.array([s[i] - s[j] for i, j in pairs]))
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    x = f(x)

    def probs(kk, w):
        n = len(w)
        m = hsc.Model(kk, f(w), f(np.zeros(n)), f(-np.ones(n)), f(np.zeros(n)))
        P = hsc.hsc_svm_probs(ctx, x, m, flags=hsc.HSC_SVM_COUPLE_F64)
        ctx.sync()
        return P.cpu().numpy().reshape(kk, -1)

    eye = np.eye(M)
    r = np.array([probs(2, eye[m:m + 1])[0] for m in range(M)])
    P = probs(k, eye).astype(np.float64)
    ref = np.array([exact(r[:, p], k) for p in range(H * W)]).T
    err = np.abs(P - ref)
    assert (err <= 2.0 ** -24 * (1 + 2.0 ** -10) * ref).all(), (err / ref).max()
