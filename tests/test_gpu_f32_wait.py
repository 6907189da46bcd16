"""The FP32 convolutions' bounded waits: with a first tensor-core launch that loads nothing the call returns FUSION_ETIMEOUT in a
few seconds, leaves the output untouched, and later calls give the scores they gave before."""

import time

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


def test_waits_run_out_and_the_model_recovers():
    F = require_gpu()
    desc = configs.model("fusion-20grid-ragged")
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 3)), max_poses=4, max_atoms=256)
    batch = poses.pack([poses.make_pose(s, (10, 20), (40, 80)) for s in (1, 2, 3)])
    ref = m.score(batch).copy()
    assert all(t["slices_per_cta"] > 0 for t in m.last_conv_tiles())
    F.fusion_set_option(m.handle, F.FUSION_OPT_TEST_WAIT_TIMEOUT, 1)
    out = np.full(3, 7.0, dtype=np.float32)
    t0 = time.perf_counter()
    with pytest.raises(F.FusionError) as e:
        m.score(batch, out=out)
    assert e.value.code == F.FUSION_ETIMEOUT
    assert time.perf_counter() - t0 < 10.0
    assert np.all(out == 7.0)
    for _ in range(2):
        np.testing.assert_array_equal(m.score(batch), ref)
