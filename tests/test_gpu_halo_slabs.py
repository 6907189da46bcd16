"""Tensor-core convolutions whose single halo buffer is loaded in slabs of two planes against the whole-halo form, which one
slice per MMA takes (slabs need an even slice group): every conv map and affinity bit for bit, over kernel sizes 1 to 7,
one to many input chunks, and sizes that leave ragged tiles; and the batch's poses alone."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("n,first,second,k", [(17, 32, 32, 3), (26, 64, 64, 5), (33, 32, 64, 7), (24, 64, 32, 1),
                                              (40, 32, 32, 7), (18, 128, 64, 5)])
def test_slabs_equal_whole_halos(n, first, second, k, dtype):
    F = require_gpu()
    desc = configs.model("fusion-24grid-c32")
    cv = lambda ci, co, kk, r=0: dict(c_in=ci, c_out=co, k=kk, stride=1, residual=r)
    desc.update(grid_n=n, conv=[cv(19, first, 5), cv(first, second, k), cv(second, second, k, 1)], cnn_dense=32, dtype=dtype)
    W = weights.init_weights(desc, 11)
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(5)))
    m = F.Model(desc, weights.to_blob(desc, W), max_poses=5, max_atoms=1200, keep_stages=True)
    got = m.score(batch).copy()
    maps = [m.fetch(F.STAGE_CONV, (i << 16) | p).copy() for i in range(3) for p in (0, 4)]
    one = m.score(poses.subset(batch, [4]))
    np.testing.assert_array_equal(one, got[4:])
    m.conv_slices_per_mma(1)
    np.testing.assert_array_equal(m.score(batch), got)
    for at, (i, p) in enumerate((i, p) for i in range(3) for p in (0, 4)):
        np.testing.assert_array_equal(m.fetch(F.STAGE_CONV, (i << 16) | p), maps[at])
