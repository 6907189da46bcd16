"""Infinite and NaN operands of the FP32 dense layer above 8 rows: the result is that of a chain of multiply-adds for every
place of the infinity among the parts' tiles, and takes no longer than finite operands."""

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _call(F, x, w, b):
    import torch
    y = torch.empty((x.shape[0], w.shape[0]), device="cuda")
    F.fusion_cnn_dense_noalloc(x, w, b, x.shape[0], w.shape[0], x.shape[1], False, y, torch.cuda.current_stream().cuda_stream)
    return y


@pytest.mark.parametrize("B,N,K", [(9, 40, 72), (64, 128, 4096), (70, 130, 8200)])
def test_patterns(B, N, K):
    F = require_gpu()
    import torch

    rng = np.random.default_rng(B)
    x = rng.uniform(-1.0, 1.0, (B, K)).astype(np.float32)
    w = rng.uniform(-1.0, 1.0, (N, K)).astype(np.float32)
    x[1, 3], x[2, K - 1], x[3, 5] = np.inf, -np.inf, np.nan
    x[4, 1], x[4, 9] = np.inf, -np.inf               # agree or not with the weights' signs
    x[5, 2] = 3.4e38                                 # finite beyond BF16's range
    x[6, 4], x[6, 6] = -3.4e38, 1e-30
    w[7, 8], w[8, 10] = np.inf, np.nan
    w[9, 11] = -3.395e38
    x[:, 11] *= np.float32(1e-3)
    w[10, 3] = 0.0                                   # infinity times zero
    x[8, 8] = 0.0
    with np.errstate(invalid="ignore", over="ignore"):
        ref = (x[:, None, :].astype(np.float64) * w[None].astype(np.float64)).sum(axis=2)
    got = _call(F, *(torch.from_numpy(a).cuda() for a in (x, w, np.zeros(N, np.float32)))).cpu().numpy()
    np.testing.assert_array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    np.testing.assert_array_equal(got[inf], ref[inf].astype(np.float32))
    fin = np.isfinite(ref)
    S = np.nan_to_num(np.abs(x.astype(np.float64)), posinf=0.0) @ np.nan_to_num(np.abs(w.astype(np.float64)), posinf=0.0).T
    # units of 2^-24 of the terms' magnitudes, as in test_gpu_dense_f32.py
    assert np.all(np.abs(got[fin] - ref[fin]) <= (-(-K // 64) + 64 + 8 + 64) * 2.0 ** -24 * S[fin])


@pytest.mark.parametrize("where", ["nan rows", "infinite weight"])
def test_takes_no_longer(where):
    F = require_gpu()
    import torch

    B, N, K = 64, 256, 221184
    x, w, b = torch.rand(B, K, device="cuda"), torch.rand(N, K, device="cuda") - 0.5, torch.zeros(N, device="cuda")

    def us():
        t = []
        for _ in range(9):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            _call(F, x, w, b)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1) * 1e3)
        return sorted(t)[4]

    finite = us()
    if where == "nan rows":
        x[::2] = float("nan")
    else:
        w[3, 7] = float("inf")
    assert us() <= 1.5 * finite
