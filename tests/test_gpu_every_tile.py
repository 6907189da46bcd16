"""Every tile that a tensor-core convolution's plan may take, each made to run and seen to run: conv maps and scores bit for bit
those of the planned tile with one slice per MMA and whole halos, on ragged sizes, for every channel count at stride 1 and 2,
several kernel sizes, and halos in slabs."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


def _cv(ci, co, k, s=1, r=0):
    return dict(c_in=ci, c_out=co, k=k, stride=s, residual=r)


# layers, and the (channels, slices per CTA, slices per MMA) that must have run among their tiles
CASES = {
    "c32": ([_cv(19, 32, 7), _cv(32, 32, 5, 1, 1), _cv(32, 32, 5, 2)],
            {(32, 16, 8), (32, 8, 8), (32, 6, 6), (32, 4, 4), (32, 2, 2), (32, 8, 1), (32, 6, 1), (32, 4, 1), (32, 2, 1)}),
    "c64": ([_cv(19, 64, 5), _cv(64, 64, 7, 1, 1), _cv(64, 64, 3, 2)],
            {(64, 8, 4), (64, 6, 3), (64, 4, 4), (64, 2, 2), (64, 8, 1), (64, 6, 1), (64, 4, 1), (64, 2, 1)}),
    "c128": ([_cv(19, 32, 3), _cv(32, 128, 5), _cv(128, 128, 3, 2)],
             {(128, 4, 2), (128, 2, 2), (128, 1, 1), (128, 4, 1), (128, 2, 1)}),
    "c256": ([_cv(19, 64, 3, 2), _cv(64, 256, 3), _cv(256, 256, 3, 2)], {(256, 2, 1), (256, 1, 1)}),
}


@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_every_tile_runs_and_gives_the_same_bits(name, dtype):
    F = require_gpu()
    conv, expected = CASES[name]
    desc = configs.model("fusion-24grid-c32")
    desc.update(grid_n=26, conv=conv, cnn_dense=32, dtype=dtype, pool=1)
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 11)), max_poses=3, max_atoms=1200, keep_stages=True)
    batch = poses.subset(poses.make_batch(configs.WORKLOADS["batch64-lig20to50-pocket300to600"]), list(range(3)))
    at = [(i << 16) | p for i in range(len(conv)) for p in range(3)]
    m.conv_slices_per_mma(1)
    ref = m.score(batch).copy()
    maps = [m.fetch(F.STAGE_CONV, a).copy() for a in at]
    assert all(t["halo_slabs"] == 0 for t in m.last_conv_tiles())
    m.conv_slices_per_mma(-1)
    ran, slabs = set(), set()
    for tile in range(6):                            # five heights below the planned one at most
        F.fusion_set_option(m.handle, F.FUSION_OPT_TEST_CONV_TILE, tile)
        np.testing.assert_array_equal(m.score(batch), ref)
        for a, want in zip(at, maps):
            np.testing.assert_array_equal(m.fetch(F.STAGE_CONV, a), want)
        for t in m.last_conv_tiles():
            ran.add((t["channels_per_cta"], t["slices_per_cta"], t["slices_per_mma"]))
            slabs.add(t["halo_slabs"] > 0)
    assert expected <= ran, expected - ran
    assert True in slabs or name == "c256"
    F.fusion_set_option(m.handle, F.FUSION_OPT_TEST_CONV_TILE, -1)
    np.testing.assert_array_equal(m.score(batch), ref)
    with pytest.raises(F.FusionError) as e:
        F.fusion_set_option(m.handle, F.FUSION_OPT_TEST_CONV_TILE, 17)
    assert e.value.code == F.FUSION_EINVAL
