"""Tensor-core convolutions of small batches on smaller tiles: calls of 1 to 9 poses (other tile heights are the shortest
schedule at each) must give every conv map and affinity bit for bit as the tiles planned for large batches do, which
setting the default slices per MMA explicitly keeps (a layer's own tile height then holds for every batch)."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("model", ["fusion-48grid-c64", "fusion-20grid-ragged", "fusion-paper-final"])
def test_small_batches_equal_the_planned_tiles(model, dtype):
    F = require_gpu()
    desc = configs.model(model, dtype=dtype)
    W = weights.init_weights(configs.model(model), 0)
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(9)))
    m = F.Model(desc, weights.to_blob(desc, W), max_poses=9, max_atoms=1200, keep_stages=True)
    m.conv_slices_per_mma(1)                       # one tile shape per layer, whatever the batch
    one = m.score(batch).copy()
    maps = [m.fetch(F.STAGE_CONV, (i << 16) | 0).copy() for i in range(len(desc["conv"]))]
    m.conv_slices_per_mma(-1)
    for n in (1, 2, 3, 4, 5, 7, 9):
        got = m.score(poses.subset(batch, list(range(n))))
        np.testing.assert_array_equal(got, one[:n])
        for i, ref in enumerate(maps):
            np.testing.assert_array_equal(m.fetch(F.STAGE_CONV, (i << 16) | 0), ref)


def test_other_channel_counts():
    """128- and 256-channel layers (heights down to one slice), stride 1 and 2, ragged sizes."""
    F = require_gpu()
    desc = configs.model("fusion-24grid-c32")
    cv = lambda ci, co, k, s=1, r=0: dict(c_in=ci, c_out=co, k=k, stride=s, residual=r)
    desc.update(grid_n=26, conv=[cv(19, 32, 3), cv(32, 128, 3), cv(128, 128, 3, 1, 1), cv(128, 256, 3, 2), cv(256, 64, 1)],
                cnn_dense=32, dtype="bf16")
    W = weights.init_weights(desc, 3)
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(6)))
    for dtype in ("bf16", "fp8"):
        d = dict(desc, dtype=dtype)
        m = F.Model(d, weights.to_blob(d, W), max_poses=6, max_atoms=1200)
        m.conv_slices_per_mma(1)
        one = m.score(batch).copy()
        m.conv_slices_per_mma(-1)
        for n in (1, 2, 3, 6):
            np.testing.assert_array_equal(m.score(poses.subset(batch, list(range(n)))), one[:n])
        m.close()
