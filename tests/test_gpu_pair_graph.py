"""The radius graph by every pair (poses of at most 2048 atoms): edges bit for bit against the oracle's float32 rule at the
edges of its tiles (32 candidates, 4 queries a warp, 8 shares a pose), in one launch (up to 16 poses) and in three, and
beside a batch whose largest pose sends it to the cell list."""

import numpy as np
import pytest

from gpu_common import require_gpu, split_csr
from oracle import fusion_oracle as O
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


def _pose(rng, n):
    side = max(6.0, (n / 0.08) ** (1 / 3))                     # protein-like density
    return rng.uniform(0, side, (n, 3)).astype(np.float32), rng.uniform(-1, 1, (n, 19)).astype(np.float32), min(n, 5)


@pytest.mark.parametrize("sizes", [(1, 2, 31, 32, 33, 63, 65, 255, 256, 257, 700), tuple([40, 9, 129] * 7), (2048,),
                                   (2049, 30)])
def test_edges(sizes):
    F = require_gpu()
    rng = np.random.default_rng(len(sizes))
    ps = [_pose(rng, n) for n in sizes]
    desc = configs.model("fusion-20grid-ragged")
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 7)), max_poses=len(ps), max_atoms=2560, keep_stages=True)
    m.score(poses.pack(ps))
    for p, (xyz, _, _) in enumerate(ps):
        g = O.radius_graph(xyz, desc["cut_cov"], desc["cut_nc"])
        for stage, name in ((F.STAGE_EDGES_COV, "cov"), (F.STAGE_EDGES_NC, "nc")):
            rp, col = split_csr(m.fetch(stage, p), len(xyz))
            np.testing.assert_array_equal(rp, g[name][0])
            np.testing.assert_array_equal(col, g[name][1])


@pytest.mark.parametrize("copies", [1, 20])
def test_capacity(copies):
    """A pose over its edge capacity fails the call in both forms; the model stays usable."""
    F = require_gpu()
    rng = np.random.default_rng(1)
    ok = _pose(rng, 60)
    dense = (rng.uniform(0, 3.0, (200, 3)).astype(np.float32), ok[1][:1].repeat(200, 0), 5)
    desc = configs.model("fusion-20grid-ragged")
    m = F.Model(desc, weights.to_blob(desc, weights.init_weights(desc, 7)), max_poses=2 * copies, max_atoms=256, max_degree=32)
    ref = m.score(poses.pack([ok] * copies))
    with pytest.raises(F.FusionError) as e:
        m.score(poses.pack([ok, dense] * copies))
    assert e.value.code == F.FUSION_ECAPACITY
    np.testing.assert_array_equal(m.score(poses.pack([ok] * copies)), ref)
