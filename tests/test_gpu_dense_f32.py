"""The FP32 dense layer's kernels (weight streaming up to 16 poses, tiles above) through the no-allocation entry point.

Against float64 with the worst case of the sums: a chain of c = ceil(K / splits / 8) + 64 multiply-adds, then 8 chains,
the splits in eighths and the bias, each addition rounding to 2^-24 of at most S = sum |x w| + |bias|.  And every kernel
adds in the same order, so a row's bits do not depend on how many rows there are.
"""

import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

BATCHES = (1, 2, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65)


@pytest.mark.parametrize("N,K", [(1, 8), (33, 72), (64, 512), (70, 2040), (129, 8200), (31, 40008)])
def test_batches_against_float64_and_each_other(N, K):
    F = require_gpu()
    import torch

    rng = np.random.default_rng(N * 7 + K)
    x = rng.uniform(-1.0, 1.0, (max(BATCHES), K)).astype(np.float32)
    w = rng.uniform(-1.0, 1.0, (N, K)).astype(np.float32)
    b = rng.uniform(-1.0, 1.0, N).astype(np.float32)
    ref = x.astype(np.float64) @ w.astype(np.float64).T + b
    S = np.abs(x.astype(np.float64)) @ np.abs(w.astype(np.float64)).T + np.abs(b)
    splits = min(128, max(1, K // 2048))
    units = -(-K // splits) // 8 + 64 + 8 + -(-splits // 8) + 8 + 1
    xd, wd, bd = (torch.from_numpy(a).cuda() for a in (x, w, b))
    last = None
    for B in BATCHES:
        y = torch.full((B + 1, N), float("nan"), device="cuda")
        F.fusion_cnn_dense_noalloc(xd, wd, bd, B, N, K, False, y)
        got = y.cpu().numpy()
        assert np.all(np.isnan(got[B]))                              # nothing past the last row
        err = np.abs(got[:B] - ref[:B])
        assert np.all(err <= units * 2.0 ** -24 * S[:B]), (B, float((err / S[:B]).max()))
        if last is not None:
            np.testing.assert_array_equal(got[:len(last)], last)
        last = got[:B]
