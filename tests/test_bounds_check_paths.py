"""The debug build's index checks on the paths that run by default: each kernel
file carries them and compiles with them (CPU), and on the GPU the checked
library gives the normal one's outputs, with every check passing, for the tiled
KNN from both layouts of the probabilities (window whole and cut, border, left
pixels), the value sort, the Krylov solver in both sizes and with restarts, and
the work-item Gram's shifted copies (odd sizes, an unaligned cube, a batch)."""

import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_10631_gb300", "csrc")

RUN = r"""
import json, sys
sys.path.insert(0, %r)
import numpy as np, torch
import paper_2404_10631_gb300 as hsc
ctx = hsc.Context(0, stream=torch.cuda.current_stream())
f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")
out = []
def add(*ts):
    ctx.sync()
    for t in ts:
        v = t.double().cpu().numpy().ravel()
        out.append([v.size, float(v.sum()), float(np.abs(v).max())])
rng = np.random.default_rng(0)
for k, B, H, W, K, R, lam in ((4, 20, 37, 53, 40, 14, 1.0), (3, 7, 50, 64, 40, 5, 0.5),
                              (8, 33, 24, 41, 16, 7, 0.2), (5, 200, 31, 33, 24, 9, 1.0),
                              (2, 129, 20, 31, 8, 3, 0.0)):
    M = k * (k - 1) // 2
    m = hsc.Model(k, f(rng.standard_normal((M, B))), f(np.zeros(M)), f(-np.ones(M)),
                  f(np.zeros(M)))
    base = f(np.exp(-np.arange(B) / 8.0))[:, None, None]
    flat = 0.5 + 0.1 * base.sqrt() * torch.as_tensor(rng.standard_normal((B, H, W)),
                                                    dtype=torch.float32, device="cuda")
    for off in (0, 3):
        room = torch.empty(B * H * W + off, device="cuda")
        cube = room[off:].view(B, H, W)
        cube.copy_(flat)
        O, I, P = (torch.empty(s, device="cuda") for s in ((k, H, W), (H, W), (k, H, W)))
        lab = hsc.hsc_classify(ctx, cube, m, K, R, lam, out_probs=O, one_band=I, probs=P)
        add(lab, O, I, P)
        O2 = torch.empty_like(O)
        lab2 = hsc.hsc_knn_filter(ctx, I, P, K, R, lam, out_probs=O2)
        add(lab2, O2)
    if B <= 128 and lam > 0:
        Ob = [torch.empty_like(O) for _ in range(2)]
        lb = hsc.hsc_classify_batch(ctx, [cube, flat], m, K, R, lam, out_probs=Ob)
        add(*lb, *Ob)
print(json.dumps(out))
"""


@pytest.mark.parametrize("name", ["knn_generic.cuh", "knn_tile_kernel.cuh", "k_knn_value.cu",
                                  "k_krylov.cu", "k_gram_tc.cu", "k_knn.cu"])
def test_kernels_carry_checks(name):
    assert "HSC_IN_BOUNDS(" in open(os.path.join(CSRC, name)).read()


def test_checked_units_compile():
    from paper_2404_10631_gb300 import build
    units = ("k_knn_tile_p4", "k_knn_tile_planes", "k_knn_value", "k_krylov")
    out = build.build(bounds_check=True, sources_only=tuple(u + ".cu" for u in units))
    for u in units:
        assert os.path.exists(os.path.join(out, u + ".o"))


@pytest.mark.gpu
def test_default_paths_pass_their_checks(hsc):
    from paper_2404_10631_gb300 import build
    res = []
    for path in (build.build(bounds_check=True), build.LIB):
        r = subprocess.run([sys.executable, "-c", RUN % ROOT], env=dict(os.environ, HSC_LIBRARY=path),
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        res.append(json.loads(r.stdout.strip().splitlines()[-1]))
    assert res[0] == res[1]
