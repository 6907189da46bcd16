"""Device memory of FP32 models: the FP16 parts that the tensor-core convolutions read take a bounded buffer, which gives way
(fewer poses to a launch, then the CUDA cores) where the device is short of memory, and a model that fits
without them is never refused.  The poses to a launch do not change a score.

The sizes: a pose's largest conv input, as two FP16 parts, is as large as the FP32 map itself; everything else a model
holds per pose is counted here from its layers."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    import torch
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _create(F, desc, blob, max_poses, max_atoms=64, max_degree=16):
    """(model, device bytes it took)."""
    before = _free()
    m = F.Model(desc, blob, max_poses=max_poses, max_atoms=max_atoms, max_degree=max_degree)
    return m, before - _free()


def test_parts_are_bounded():
    """1,024 more poses cost their own maps (two activations, the grid, the pooled map and 64 atoms' share), not a second
    copy of the largest one."""
    F = require_gpu()
    desc = configs.model("fusion-24grid-c32")
    blob = weights.to_blob(desc, weights.init_weights(desc, 0))
    took = []
    for n in (1024, 2048):
        m, used = _create(F, desc, blob, n)
        took.append(used)
        m.close()
    act, grid, pooled = 24 ** 3 * 32 * 4, 24 ** 3 * 24 * 4, 12 ** 3 * 32 * 4
    atoms = 64 * (9 * 32 * 4 + 2 * 16 * 4 + 4 * (22 + 64))      # states and messages, edges, inputs and voxelize records
    per_pose = 2 * act + grid + pooled + atoms + 256 * 1024     # (cell list, splits of the dense layer: under 256 KB)
    assert took[1] - took[0] < 1024 * per_pose, (took, per_pose)
    assert per_pose < 2 * act + grid + pooled + act             # the bound would show a second copy


def test_more_poses_than_the_buffer_holds():
    """Up to 45 poses of 48^3 x 64 maps, whose buffer holds 18 (three poses, repeated, and 3^3 kernels): each pose's score
    is the one it has alone."""
    F = require_gpu()
    desc = configs.model("fusion-48grid-c64")
    desc["conv"] = [dict(c_in=19, c_out=64, k=3, stride=1, residual=0), dict(c_in=64, c_out=64, k=3, stride=1, residual=1),
                    dict(c_in=64, c_out=128, k=3, stride=2, residual=0)]
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 1)), max_poses=45, max_atoms=256)
    three = poses.pack([poses.make_pose(s, (10, 20), (30, 60)) for s in (1, 2, 3)])
    one = np.concatenate([m.score(poses.subset(three, [p])) for p in range(3)])
    for n in (18, 19, 45):
        got = m.score(poses.subset(three, [i % 3 for i in range(n)]))
        np.testing.assert_array_equal(got, np.resize(one, n))
    assert all(t["slices_per_cta"] > 0 for t in m.last_conv_tiles())


def test_created_without_room_for_the_parts():
    """With 10 MB less than the tensor-core form takes, the model is made on the CUDA cores and scores as well."""
    F = require_gpu()
    import torch
    desc = configs.model("fusion-48grid-c64")
    blob = weights.to_blob(desc, weights.init_weights(desc, 1))
    batch = poses.pack([poses.make_pose(5, (8, 12), (30, 45))])
    m, used = _create(F, desc, blob, 1)
    ref = m.score(batch).copy()
    assert all(t["slices_per_cta"] > 0 for t in m.last_conv_tiles())
    m.close()
    fill = torch.empty(_free() - used + 10 * MB, dtype=torch.uint8, device="cuda")
    try:
        m = F.Model(desc, blob, max_poses=1, max_atoms=64, max_degree=16)
        got = m.score(batch).copy()
        assert all(t["slices_per_cta"] == 0 for t in m.last_conv_tiles())
        m.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert abs(float(got[0]) - float(ref[0])) <= 1e-4
