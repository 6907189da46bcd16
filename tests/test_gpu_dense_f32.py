"""The FP32 dense layer's kernels: weight streaming up to 8 rows and the tensor-core split form above (the
no-allocation entry point), and the tiles that an FP32 model's larger batches take.

Against float64 with the worst case of the sums: a chain of c = ceil(K / splits / 8) + 64 multiply-adds, then 8 chains,
the splits in eighths and the bias, each addition rounding to 2^-24 of at most S = sum |x w| + |bias|; the tensor-core
form's chains are shorter (4 MMAs of 2 units, then one addition per 64 of K) and its dropped
products add 2 units.  The kernels a model takes add in the same order, so a pose's bits do not depend on the batch.
"""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

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
        if B <= 8:
            if last is not None:
                np.testing.assert_array_equal(got[:len(last)], last)
            last = got[:B]


@pytest.mark.parametrize("B", [4, 9, 70])
def test_infinities_and_nan_stay_in_their_row(B):
    """The split form has no infinities of its own: such outputs are those of a chain of multiply-adds."""
    F = require_gpu()
    import torch

    rng = np.random.default_rng(B)
    N, K = 40, 4104
    x = rng.uniform(-1.0, 1.0, (B, K)).astype(np.float32)
    w = rng.uniform(-1.0, 1.0, (N, K)).astype(np.float32)
    x[1, 5] = np.inf
    x[2, 4100] = np.nan
    x[3, 7] = 3.4e38                      # rounds to a BF16 infinity; its products are finite
    w[3, 9] = 0.0
    b = np.zeros(N, np.float32)
    y = torch.empty((B, N), device="cuda")
    F.fusion_cnn_dense_noalloc(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), torch.from_numpy(b).cuda(), B, N, K,
                               False, y)
    got = y.cpu().numpy()
    np.testing.assert_array_equal(got[1], np.where(w[:, 5] > 0, np.inf, -np.inf))
    assert np.all(np.isnan(got[2]))
    ref = x.astype(np.float64) @ w.astype(np.float64).T
    np.testing.assert_allclose(got[3], ref[3], rtol=1e-5)
    np.testing.assert_allclose(got[0], ref[0], rtol=0, atol=1e-2)


def test_model_batches_are_independent():
    """An FP32 model's dense layer at 1, 12, 20 and 40 poses (streaming, 32- and 64-pose tiles): the same bits per pose."""
    F = require_gpu()
    desc = configs.model("fusion-20grid-ragged")
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 7)), max_poses=40, max_atoms=256)
    three = poses.pack([poses.make_pose(s, (10, 20), (30, 60)) for s in (1, 2, 3)])
    one = np.concatenate([m.score(poses.subset(three, [p])) for p in range(3)])
    for n in (12, 20, 40):
        got = m.score(poses.subset(three, [i % 3 for i in range(n)]))
        np.testing.assert_array_equal(got, np.resize(one, n))
