"""FP32 convolutions on the tensor cores (two-part FP16 operands) against a float64 convolution of the GPU's own input.

The tolerance is worst-case and per output, S = sum |x w| over its terms, in units of 2^-24 S: up to 14 MMAs of a kernel
offset each are added with truncation in an interval (2 units each), every interval's sum and the small products'
are added with rounding (1 unit each), and the operands' parts and the dropped product lose up to 8 units; layers
that no tile fits run on the CUDA cores, a chain of n multiply-adds (n units).
"""

import numpy as np
import pytest

from gpu_common import require_gpu
from synth import configs, poses, weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    return require_gpu()


def _cv(c_in, c_out, k, stride=1, residual=0):
    return dict(c_in=c_in, c_out=c_out, k=k, stride=stride, residual=residual)


# (grid side, layers): ragged sizes, odd stride-2 input (NDHWC parts), channel counts of several blocks, every kernel
# size, a first layer too wide or strided to fold, a residual layer, and a layer that falls back to the CUDA cores
LAYERS = {
    "odd-stride2": (13, [_cv(19, 64, 7), _cv(64, 128, 5, 2)]),
    "blocks": (20, [_cv(19, 32, 5), _cv(32, 32, 9, residual=1), _cv(32, 160, 3, 2), _cv(160, 256, 1)]),
    "first-strided": (17, [_cv(19, 96, 3, 2), _cv(96, 96, 3, residual=1), _cv(96, 64, 1, 2)]),
    "first-9": (10, [_cv(19, 32, 9), _cv(32, 64, 7, 2)]),
    "fallback": (8, [_cv(19, 32, 3), _cv(32, 128, 9), _cv(128, 32, 3)]),
}
CUDA_CORES = {("fallback", 1)}


def _desc(n, conv):
    d = configs.model("fusion-24grid-c32")
    d.update(grid_n=n, conv=conv, cnn_dense=32, pool=1)
    return d


def _batch():
    return poses.pack([poses.make_pose(s, a, b) for s, a, b in
                       [(101, (20, 30), (60, 120)), (102, (8, 12), (20, 40)), (104, (5, 5), (0, 0))]])


def _conv(x, W, b, stride):
    import torch
    t = torch.nn.functional.conv3d(torch.from_numpy(np.ascontiguousarray(x.transpose(3, 0, 1, 2)))[None],
                                   torch.from_numpy(W.astype(np.float64)),
                                   None if b is None else torch.from_numpy(b.astype(np.float64)), stride=stride,
                                   padding=W.shape[2] // 2)
    return t[0].numpy().transpose(1, 2, 3, 0)


@pytest.mark.parametrize("name", sorted(LAYERS))
def test_layers_against_float64(F, name):
    n, conv = LAYERS[name]
    desc = _desc(n, conv)
    W = weights.init_weights(desc, 3)
    batch = _batch()
    m = F.Model(desc, weights.to_blob(desc, W), max_poses=3, max_atoms=512, keep_stages=True)
    got = m.score(batch).copy()
    for p in range(3):
        x = m.fetch(F.STAGE_GRID, p).reshape(n, n, n, 19).astype(np.float64)
        for i, cv in enumerate(conv):
            y = m.fetch(F.STAGE_CONV, (i << 16) | p)
            s = round((y.size // cv["c_out"]) ** (1 / 3))
            y = y.reshape(s, s, s, cv["c_out"]).astype(np.float64)
            w = W[f"conv{i}.w"]
            ref = np.maximum(_conv(x, w, W[f"conv{i}.b"], cv["stride"]), 0.0) + (x if cv["residual"] else 0.0)
            S = _conv(np.abs(x), np.abs(w), None, cv["stride"])
            terms = cv["k"] ** 3 * cv["c_in"]
            intervals = -(-cv["c_in"] // 16) * 8 * -(-cv["k"] ** 2 // max(1, 14 // cv["k"]))
            units = terms if (name, i) in CUDA_CORES else 2 * 14 + intervals + 8
            err = np.abs(y - ref)
            tol = 2.0 ** -24 * (units * S + 4 * np.abs(ref) + 4 * np.abs(W[f"conv{i}.b"]))
            assert np.all(err <= tol), (i, p, float((err / (tol + 1e-300)).max()))
            x = y
    alone = [m.score(poses.subset(batch, [p]))[0] for p in range(3)]     # smaller tiles, the same sums
    np.testing.assert_array_equal(np.array(alone), got)


def test_tile_heights_and_other_poses_do_not_matter(F):
    """Batches from 1 to 24 poses take different tile heights; a pose with an infinite feature stays in its own maps."""
    desc = configs.model("fusion-20grid-ragged")
    W = weights.init_weights(desc, 7)
    batch = _batch()
    m = F.Model(desc, weights.to_blob(desc, W), max_poses=24, max_atoms=512)
    one = m.score(poses.subset(batch, [0]))[0]
    many = m.score(poses.subset(batch, [0, 1, 2] * 8))
    assert np.all(many[::3] == one)
    bad = poses.subset(batch, [0, 1, 0])
    bad["feat"][int(bad["atom_off"][1]), 12] = np.inf
    got = m.score(bad)
    assert got[0] == one and got[2] == one
