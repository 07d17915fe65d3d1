"""A call with much work in the second KNN pass leaves the SMs to other
streams: the next call's CTAs are not placed before the pass is known to have
none. A small frame classified on another stream meanwhile takes a small part
of one such call (it took as long as the call and longer when the next call's
CTAs waited in the SMs)."""

import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_frames_beside_a_hard_map(hsc, ctx):
    import torch
    rng = np.random.default_rng(4)
    f = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda")  # noqa: E731
    H = W = 1024
    I, P = torch.rand((H, W), device="cuda"), torch.softmax(torch.randn((4, H, W), device="cuda"), 0)
    cube = f(rng.random((64, 48, 48)))
    model = hsc.Model(4, f(rng.standard_normal((6, 64))), f(np.zeros(6)), f(-np.ones(6)),
                      f(np.zeros(6)))
    lab, small = torch.empty((H, W), dtype=torch.int32, device="cuda"), None
    torch.cuda.synchronize()
    with hsc.Context(0) as hard, hsc.Context(0) as live:
        def hard_call():
            hsc.hsc_knn_filter(hard, I, P, 40, 14, 0.1, labels=lab)
        small = hsc.hsc_classify(live, cube, model, 16, 7, 1.0)
        hard_call()
        live.sync()
        hard.sync()
        t = time.perf_counter()
        hard_call()
        hard.sync()
        one = time.perf_counter() - t
        for _ in range(8):
            hard_call()
        lat = []
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 6 * one:
            t = time.perf_counter()
            hsc.hsc_classify(live, cube, model, 16, 7, 1.0, labels=small)
            live.sync()
            lat.append(time.perf_counter() - t)
        hard.sync()
    assert sorted(lat)[len(lat) // 2] < 0.25 * one, (lat[:8], one)
