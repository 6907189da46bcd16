"""Infinities in the FP32 convolutions: an infinite feature or weight reaches the outputs that use it, as in a chain of
multiply-adds (an infinity of its sign, NaN where two disagree or one meets a zero, which ReLU stores as 0), and every
other output keeps its value.

Each layer's output is compared with a float64 convolution of the GPU's own input, the finite ones within the bound of
test_gpu_f32_conv_tc.py (the intervals' sums, the parts and the dropped product)."""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights
from test_gpu_f32_conv_tc import _conv, _cv, _desc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F_():
    return require_gpu()


def _check_layers(F, m, conv, W, n, p):
    """Returns how many outputs of each layer were infinite."""
    x = m.fetch(F.STAGE_GRID, p).reshape(n, n, n, 19).astype(np.float64)
    found = []
    for i, cv in enumerate(conv):
        y = m.fetch(F.STAGE_CONV, (i << 16) | p)
        s = round((y.size // cv["c_out"]) ** (1 / 3))
        y = y.reshape(s, s, s, cv["c_out"]).astype(np.float64)
        w, b = W[f"conv{i}.w"], W[f"conv{i}.b"]
        with np.errstate(invalid="ignore"):
            ref = _conv(x, w, b, cv["stride"])
            ref = np.where(np.isnan(ref), 0.0, np.maximum(ref, 0.0)) + (x if cv["residual"] else 0.0)
        np.testing.assert_array_equal(np.isinf(y), np.isinf(ref))
        assert not np.any(np.isnan(y))
        fin = np.isfinite(ref)
        ax, aw = np.where(np.isfinite(x), np.abs(x), 0.0), np.where(np.isfinite(w), np.abs(w), 0.0)
        S = _conv(ax, aw, None, cv["stride"])
        intervals = -(-cv["c_in"] // 16) * 8 * -(-cv["k"] ** 2 // max(1, 14 // cv["k"]))
        tol = 2.0 ** -24 * ((2 * 14 + intervals + 8) * S + 4 * np.where(fin, ref, 0.0) + 4 * np.abs(b))
        # (parts of a pose's smallest values: 2^-39 of its largest a term)
        tol = tol + 2.0 ** -39 * ax.max() * aw.sum(axis=(1, 2, 3, 4))
        assert np.all(np.abs(np.where(fin, y, 0.0) - np.where(fin, ref, 0.0)) <= tol), i
        found.append(int(np.isinf(y).sum()))
        x = y
    return found


@pytest.mark.parametrize("feature,k", [(5, 7), (5, 3), (17, 5), (18, 3)])
def test_an_infinite_feature(F_, feature, k):
    n, conv = 20, [_cv(19, 32, k), _cv(32, 32, 3, residual=1), _cv(32, 64, 3, 2)]
    desc = _desc(n, conv)
    W = weights.init_weights(desc, 3)
    for i in range(3):                       # eight channels whose infinities never disagree
        W[f"conv{i}.w"][:8] = np.abs(W[f"conv{i}.w"][:8])
    batch = poses.pack([poses.make_pose(s, (6, 8), (10, 20)) for s in (101, 102)])
    m = F_.Model(desc, weights.to_blob(desc, W), max_poses=2, max_atoms=64, keep_stages=True)
    ref = m.score(batch).copy()
    batch["feat"][int(batch["atom_off"][1]) - 1, feature] = np.inf
    got = m.score(batch)
    assert got[1] == ref[1]
    found = _check_layers(F_, m, conv, W, n, 0)
    # (the density's edge, where an infinity met a zero weight, is NaN: a 7^3 window always touches it)
    assert k == 7 or all(f > 0 for f in found), found


def test_an_infinite_weight(F_):
    n, conv = 16, [_cv(19, 32, 5), _cv(32, 64, 3), _cv(64, 32, 1)]
    desc = _desc(n, conv)
    W = weights.init_weights(desc, 3)
    W["conv1.w"][3, 2, 1, 1, 1] = np.inf
    W["conv1.w"][3, 4, 0, 1, 2] = 1e6        # beyond FP16 without the scale of the channel's finite weights
    batch = poses.pack([poses.make_pose(101, (6, 8), (10, 20))])
    m = F_.Model(desc, weights.to_blob(desc, W), max_poses=1, max_atoms=64, keep_stages=True)
    m.score(batch)
    found = _check_layers(F_, m, conv, W, n, 0)
    assert found[0] == 0 and found[1] > 0


@pytest.mark.parametrize("w_exp,x_exp", [(115, -110), (-110, 100)])
def test_scales_far_apart(F_, w_exp, x_exp):
    """Weights and densities at opposite ends of FP32's range, whose products are ordinary numbers: no step overflows."""
    n, conv = 14, [_cv(19, 64, 3), _cv(64, 32, 3, 2)]
    desc = _desc(n, conv)
    W = weights.init_weights(desc, 3)
    W["conv0.w"] = W["conv0.w"] * np.float32(2.0 ** w_exp)
    batch = poses.pack([poses.make_pose(101, (6, 8), (10, 20))])
    batch["feat"] = batch["feat"] * np.float32(2.0 ** x_exp)
    m = F_.Model(desc, weights.to_blob(desc, W), max_poses=1, max_atoms=64, keep_stages=True)
    m.score(batch)
    assert _check_layers(F_, m, conv, W, n, 0) == [0, 0]
