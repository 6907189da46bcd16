"""FP32 servers under an HBM budget: the buffer of the convolutions' FP16 parts gives way before a slot does, and every slot
of a server takes the same form, so a pose's score does not depend on its slot."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _scores(srv, three, n):
    tickets = [srv.submit(*three[i % 3]) for i in range(n)]
    srv.drain()
    return np.array([srv.poll(t)[0] for t in tickets], np.float32)


@pytest.mark.parametrize("share", [0.97, 0.9, 0.85])
def test_a_budget_below_a_slot_with_all_parts(share):
    """24^3 maps, batches of 256: the parts are over a fifth of a slot; a budget without room for them still has a slot,
    and its scores are those of a model with room for all."""
    F = require_gpu()
    desc = configs.model("fusion-24grid-c32")
    blob = weights.to_blob(desc, weights.init_weights(desc, 0))
    three = [poses.make_pose(s, (10, 20), (30, 60)) for s in (1, 2, 3)]
    m = F.Model(desc, blob, max_poses=3, max_atoms=128)
    one = m.score(poses.pack(three)).copy()
    m.close()
    srv = F.Server(desc, blob, max_batch=256, slots=1, max_atoms=128, batch_window_us=20000.0)
    per_slot = srv.stats()["slot_bytes"]
    np.testing.assert_array_equal(_scores(srv, three, 200), np.resize(one, 200))
    srv.close()
    srv = F.Server(desc, blob, max_batch=256, slots=1, max_atoms=128, batch_window_us=20000.0,
                   hbm_budget_bytes=int(share * per_slot))
    assert srv.stats()["slots"] == 1 and srv.stats()["slot_bytes"] <= share * per_slot
    np.testing.assert_array_equal(_scores(srv, three, 200), np.resize(one, 200))
    srv.close()


def test_a_budget_without_room_for_one_pose_of_parts():
    """Full-size maps, one pose: 10 MB less than a slot leaves the CUDA cores; two slots of that kind give one score."""
    F = require_gpu()
    desc = configs.model("fusion-48grid-c64")
    blob = weights.to_blob(desc, weights.init_weights(desc, 1))
    three = [poses.make_pose(s, (10, 20), (30, 60)) for s in (1, 2, 3)]
    srv = F.Server(desc, blob, max_batch=1, slots=1, max_atoms=128)
    per_slot = srv.stats()["slot_bytes"]
    ref = _scores(srv, three, 3)
    srv.close()
    srv = F.Server(desc, blob, max_batch=1, slots=1, max_atoms=128, hbm_budget_bytes=per_slot - 10 * MB)
    assert srv.stats()["slots"] == 1
    small = srv.stats()["slot_bytes"]
    got = _scores(srv, three, 3)
    srv.close()
    assert np.abs(got - ref).max() <= 1e-4
    srv = F.Server(desc, blob, max_batch=1, slots=2, max_atoms=128, hbm_budget_bytes=2 * small)
    assert srv.stats()["slots"] >= 1
    np.testing.assert_array_equal(_scores(srv, three, 12), np.resize(_scores(srv, three, 3), 12))
    srv.close()
