"""The autotuner's choice holds for the batch size it was measured on: a layer whose tile configuration it replaced runs that
tile in calls of this size (an estimate chooses between tile heights only where nothing was measured), and the scores
stay the same there and at other sizes.  The graph branch's schedule is measured as calls of that size run it, and one that
was measured on a large batch does not take the place of the small calls' own."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


def _mixed(n):
    cv = lambda ci, co, k, s=1, r=0: dict(c_in=ci, c_out=co, k=k, stride=s, residual=r)
    d = configs.model("fusion-24grid-c32")
    d.update(grid_n=n, conv=[cv(19, 32, 3), cv(32, 128, 3), cv(128, 128, 3, 1, 1), cv(128, 256, 3, 2), cv(256, 64, 1)],
             cnn_dense=32)
    return d


@pytest.mark.parametrize("model,dtype,n", [("fusion-48grid-c64", "bf16", 1), ("fusion-paper-final", "bf16", 3),
                                           ("fusion-paper-final", "fp8", 8), ("fusion-20grid-ragged", "fp8", 9),
                                           (40, "fp8", 8), (26, "bf16", 2)])
def test_tuned_batch_size_takes_the_tuned_tile(model, dtype, n):
    F = require_gpu()
    desc = _mixed(model) if isinstance(model, int) else configs.model(model)
    W = weights.init_weights(desc, 0)
    desc["dtype"] = dtype
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(12)))
    tuned_on = poses.subset(batch, list(range(n)))
    m = F.Model(desc, weights.to_blob(desc, W), max_poses=12, max_atoms=1200)
    all_before, before = m.score(batch).copy(), m.score(tuned_on).copy()
    default = m.conv_tiles()
    m.autotune(tuned_on)
    np.testing.assert_array_equal(m.score(tuned_on), before)
    for i, (was, now, ran) in enumerate(zip(default, m.conv_tiles(), m.last_conv_tiles())):
        if now != was:
            assert (ran["slices_per_cta"], ran["slices_per_mma"]) == (now["slices_per_cta"], now["slices_per_mma"]), i
    ran = m.last_conv_tiles()
    np.testing.assert_array_equal(m.score(batch), all_before)
    m.score(tuned_on)
    assert m.last_conv_tiles() == ran


def _call_us(m, batch):
    m.score(batch)
    return float(np.median([(m.score(batch), m.timings()["total"])[1] for _ in range(15)])) * 1e3


@pytest.mark.parametrize("tuned_on", [1, 2, 12])
def test_small_calls_are_no_slower_after_tuning(tuned_on):
    """One and two paper-final poses, whose graph branch is the longer one: device time of a call before and after."""
    F = require_gpu()
    desc = configs.model("fusion-paper-final", dtype="bf16")
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(12)))
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 0)), max_poses=12, max_atoms=1200)
    sizes = [n for n in (1, 2) if n == tuned_on or tuned_on == 12]
    before = [_call_us(m, poses.subset(batch, list(range(n)))) for n in sizes]
    m.autotune(poses.subset(batch, list(range(tuned_on))))
    after = [_call_us(m, poses.subset(batch, list(range(n)))) for n in sizes]
    assert all(a <= 1.08 * b for a, b in zip(after, before)), (before, after)
