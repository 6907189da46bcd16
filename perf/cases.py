"""Performance cases of the pose-scoring library: what its users call, at the sizes they call it with.

Three kinds of case, each through the public binding (``paper_2104_04547_gb300.fusion``):

* ``score``: one ``Model.score`` call on a packed batch, host arrays or device buffers, plain launches or
  CUDA-graph replay;
* ``dense``: ``fusion_cnn_dense_noalloc``, the CNN dense layer for callers that cannot allocate;
* ``server``: a burst of single-pose requests to a continuous-batching server, drained and collected.

Poses are synthetic docked complexes of the shapes in ``synth/configs.py`` (a ligand in a pocket shell, 19
atom features); weights are the seeded random-init ones of ``synth/weights.py``.  A program creates its
model once and scores many batches with it, so states of one configuration share one model (or server).
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2104_04547_gb300 import fusion as F
from synth import configs, poses, weights

# (ligand lo, hi, pocket lo, hi) atoms per pose, from synth/configs.py WORKLOADS
SMALL_POSE = (24, 24, 200, 200)
BATCH_POSES = (20, 50, 300, 600)
UNEVEN_POSES = (15, 60, 250, 800)

MAX_ATOMS = 1200
MAX_DEGREE = 96          # mean edges per atom and type: the 5.22 A cutoff in an 800-atom pocket reaches 60
WEIGHT_SEED = 0


def _score(preset, dtype, n, shape, capacity, on_device, graphs=False, name=None):
    c = dict(kind="score", preset=preset, dtype=dtype, poses=n, lig_lo=shape[0], lig_hi=shape[1],
             pocket_lo=shape[2], pocket_hi=shape[3], capacity=capacity, on_device=on_device, graphs=graphs)
    if name:
        c["name"] = name
    return c


def _dense(B, N, K, relu, name=None):
    c = dict(kind="dense", B=B, N=N, K=K, relu=relu)
    if name:
        c["name"] = name
    return c


def _server(preset, dtype, n, shape, max_batch, slots, name=None):
    c = dict(kind="server", preset=preset, dtype=dtype, poses=n, lig_lo=shape[0], lig_hi=shape[1],
             pocket_lo=shape[2], pocket_hi=shape[3], max_batch=max_batch, slots=slots)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one pose of the single-pose model in FP32 (a check of one docked pose)
        _score("fusion-24grid-c32", "f32", 1, SMALL_POSE, 1, False, name="tiny_f32_1"),
        # one interactive request to a resident model of each size: latency, launches, a nearly empty chip
        _score("fusion-paper-final", "bf16", 1, BATCH_POSES, 64, False, name="paper_bf16_1"),
        _score("fusion-48grid-c64", "bf16", 1, BATCH_POSES, 64, False, name="full_bf16_1"),
        # the paper's smallest per-rank batch, and what a server's slot takes at moderate load
        _score("fusion-48grid-c64", "fp8", 12, BATCH_POSES, 64, False, name="full_fp8_12"),
        # the headline batch, resident on the device (bench.py's timed step)
        _score("fusion-48grid-c64", "bf16", 64, BATCH_POSES, 64, True, name="full_bf16_64"),
        # the largest: the 256-pose uneven batch of a screening job
        _score("fusion-48grid-c64", "fp8", 256, UNEVEN_POSES, 256, False, name="full_fp8_256"),
        # the paper's final architecture on the headline batch, replayed as a CUDA graph (batching.py)
        _score("fusion-paper-final", "bf16", 64, BATCH_POSES, 64, True, graphs=True, name="paper_bf16_64"),
        # the paper's per-rank batch of 56 poses, uneven, end to end from host arrays
        _score("fusion-paper-final", "fp8", 56, UNEVEN_POSES, 64, False, name="paper_fp8_56"),
        # full-precision scoring: a few poses re-scored in FP32 to check a lower-precision run
        _score("fusion-48grid-c64", "f32", 3, BATCH_POSES, 8, False, name="full_f32_3"),
        # a burst of single-pose requests to the continuous-batching server
        _server("fusion-paper-final", "bf16", 48, BATCH_POSES, 16, 2, name="server_bf16_48"),
        # the CNN dense layer without allocation: the full-size layer on the headline batch, and the
        # paper-final layer at a small batch (a latency-bound request loop)
        _dense(64, 256, 221184, True, name="dense_64x256x221184"),
        _dense(4, 128, 110592, True, name="dense_4x128x110592"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["score", "dense", "server"], [0.78, 0.14, 0.08])[0]
    if kind == "dense":
        K = 8 * _log_int(rng, 256, 27648)
        splits = max(1, min(128, K // 2048))
        N = _log_int(rng, 24, 300)
        B = _log_int(rng, 1, max(1, min(64, F.FUSION_NOALLOC_MAX_PARTIALS // (splits * N))))
        return _dense(B, N, K, rng.random() < 0.8)
    shape = rng.choice([SMALL_POSE, BATCH_POSES, BATCH_POSES, UNEVEN_POSES])
    if kind == "server":
        preset, most = rng.choice([("fusion-paper-final", 96), ("fusion-48grid-c64", 24)])
        return _server(preset, rng.choice(["bf16", "fp8"]), _log_int(rng, 4, most), shape,
                       rng.choice([8, 16, 32]), rng.choice([1, 2]))
    preset = rng.choices(["fusion-48grid-c64", "fusion-paper-final", "fusion-24grid-c32", "fusion-20grid-ragged",
                          "fusion-48grid-c64-mid", "fusion-paper-final-late", "fusion-24grid-c32-late"],
                         [0.3, 0.34, 0.08, 0.1, 0.06, 0.06, 0.06])[0]
    dtype = rng.choices(["bf16", "fp8", "f32"], [0.46, 0.34, 0.2])[0]
    big = preset.startswith("fusion-48grid")
    most = {"bf16": 96 if big else 256, "fp8": 200 if big else 256,
            "f32": 3 if big else 24 if preset.startswith("fusion-paper") else 64}[dtype]
    n = _log_int(rng, 1, most)
    return _score(preset, dtype, n, shape, max(n, rng.choice([1, 64])), rng.random() < 0.5, rng.random() < 0.25)


# ---- inputs and handles ----

def _poses(case, seed):
    """[(xyz, feat, n_lig)]: a few base complexes; every pose is one of them with its ligand rotated about its
    centroid and jittered by N(0, 0.5^2) A (as docked poses of one ligand are) and a part of its pocket."""
    rng = np.random.default_rng(seed)
    n = case["poses"]
    base = [poses.make_pose(int(rng.integers(1, 1 << 31)), (case["lig_lo"], case["lig_hi"]),
                            (case["pocket_hi"], case["pocket_hi"])) for _ in range(min(n, 5))]
    out = []
    for p in range(n):
        xyz, feat, n_lig = base[p % len(base)]
        q = rng.normal(size=4)
        w, x, y, z = q / np.sqrt((q * q).sum())
        R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                      [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                      [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])
        lig = xyz[:n_lig].astype(np.float64)
        c = lig.mean(axis=0)
        lig = (lig - c) @ R.T + c + 0.5 * rng.normal(size=lig.shape) * (p >= len(base))
        n_pocket = int(rng.integers(case["pocket_lo"], case["pocket_hi"] + 1))
        keep = n_lig + np.sort(rng.permutation(len(xyz) - n_lig)[:n_pocket])
        out.append((np.concatenate([lig.astype(np.float32), xyz[keep]]),
                    np.concatenate([feat[:n_lig], feat[keep]]), n_lig))
    return out


@functools.lru_cache(maxsize=2)
def _weights(preset):
    return weights.init_weights(configs.model(preset), WEIGHT_SEED)


@functools.lru_cache(maxsize=1)
def _model(preset, dtype, capacity, graphs):
    desc = configs.model(preset, dtype=dtype)
    m = F.Model(desc, weights.to_blob(desc, _weights(preset)), max_poses=capacity, max_atoms=MAX_ATOMS,
                max_degree=MAX_DEGREE)
    if graphs:
        m.use_cuda_graphs()
    return m


@functools.lru_cache(maxsize=1)
def _server_of(preset, dtype, max_batch, slots):
    desc = configs.model(preset, dtype=dtype)
    return F.Server(desc, weights.to_blob(desc, _weights(preset)), max_batch=max_batch, slots=slots,
                    max_atoms=MAX_ATOMS, max_degree=MAX_DEGREE)


def _dense_inputs(case, seed, device="cuda"):
    g = torch.Generator(device=device).manual_seed(seed)
    B, N, K = case["B"], case["N"], case["K"]
    x = torch.rand((B, K), generator=g, device=device).mul_(2).sub_(1).clamp_(min=0)   # post-ReLU activations
    bound = math.sqrt(6.0 / K)
    w = torch.rand((N, K), generator=g, device=device).mul_(2 * bound).sub_(bound)
    b = torch.rand((N,), generator=g, device=device).mul_(2).sub_(1).mul_(1 / math.sqrt(K))
    return x, w, b


def prepare(case, seed):
    if case["kind"] == "dense":
        x, w, b = _dense_inputs(case, seed)
        y = torch.empty((case["B"], case["N"]), device="cuda")
        return dict(case=case, x=x, w=w, b=b, y=y)
    ps = _poses(case, seed)
    if case["kind"] == "server":
        return dict(case=case, server=_server_of(case["preset"], case["dtype"], case["max_batch"], case["slots"]),
                    poses=ps)
    batch = poses.pack(ps)
    m = _model(case["preset"], case["dtype"], case["capacity"], case["graphs"])
    if case["on_device"]:
        batch = {k: torch.from_numpy(v).cuda() for k, v in batch.items()}
        out = torch.empty(case["poses"], device="cuda")
        torch.cuda.synchronize()
    else:
        out = np.empty(case["poses"], dtype=np.float32)
    return dict(case=case, model=m, batch=batch, out=out)


def run(state):
    case = state["case"]
    if case["kind"] == "dense":
        F.fusion_cnn_dense_noalloc(state["x"], state["w"], state["b"], case["B"], case["N"], case["K"],
                                   case["relu"], state["y"])
        return state["y"]
    if case["kind"] == "server":
        s = state["server"]
        tickets = [s.submit(xyz, feat, n_lig) for xyz, feat, n_lig in state["poses"]]
        s.drain()
        return np.array([s.poll(t)[0] for t in tickets], dtype=np.float32)
    return state["model"].score(state["batch"], n_poses=case["poses"], out=state["out"],
                                on_device=case["on_device"])


# ---- what a pass cannot do without ----

def _edges_per_atom(cut, n_atoms):
    """Typical directed edges per atom at a cutoff: the pocket shell's density over a ball, half of it outside."""
    return 0.55 * n_atoms / 6500.0 * 4.19 * cut ** 3


def _pose_work(desc, atoms):
    """(conv flops, dense flops, graph + head flops) of one pose with that many atoms, real channels."""
    n, conv = desc["grid_n"], 0.0
    for cv in desc["conv"]:
        n = (n + 2 * (cv["k"] // 2) - cv["k"]) // cv["stride"] + 1
        conv += 2.0 * n ** 3 * cv["k"] ** 3 * cv["c_in"] * cv["c_out"]
    c, side = weights.cnn_out_shape(desc)
    dense = 2.0 * c * side ** 3 * desc["cnn_dense"] + 2.0 * desc["cnn_dense"] * desc.get("cnn_dense2", 0)
    graph, wid = 0.0, weights.stage_widths(desc)
    for s, st in enumerate(desc["sg_stages"]):
        H, types = wid[s], weights.edge_types(st["edges"])
        deg = _edges_per_atom(desc["cut_nc"] if "nc" in types else desc["cut_cov"], atoms)
        graph += st["steps"] * atoms * (2.0 * H * H * (6 + len(types)) + H * deg)
    graph += 2.0 * desc["sg_gather_width"] * 3 * wid[-1] * 40
    return conv, dense, graph


def work(case):
    if case["kind"] == "dense":
        B, N, K = case["B"], case["N"], case["K"]
        return {"bytes": 4.0 * (B * K + N * K + N + B * N), "flops": 2.0 * B * N * K}
    desc = configs.model(case["preset"])
    atoms = (case["lig_lo"] + case["lig_hi"] + case["pocket_lo"] + case["pocket_hi"]) / 2.0
    n = case["poses"]
    conv, dense, graph = _pose_work(desc, atoms)
    conv_b = {"f32": 4, "bf16": 2, "fp8": 1}[case["dtype"]]
    other_b = 4 if case["dtype"] == "f32" else 2
    wb = 0.0
    for name, shape, _kind, _fan in weights.layout(desc):
        size = float(np.prod(shape))
        wb += size * (conv_b if name.startswith("conv") else other_b if name.startswith("cnn_dense.w") else 4)
    return {"bytes": wb + n * (atoms * (12 + 76) + 8 + 4), "flops": n * (conv + dense + graph)}


# ---- the same results in 64 bits ----

def _grid64(desc, xyz, feat, n_lig, dev):
    """Density grid [n][n][n][19]: voxel-integrated Gaussians over the +-k voxel cube; the grid origin and the
    containing voxel are defined in float32."""
    n, h, sigma, k = desc["grid_n"], np.float32(desc["grid_h"]), desc["sigma"], desc["support"]
    s = np.zeros(3, dtype=np.float32)
    for a in range(n_lig):
        s = s + xyz[a]
    origin = s / np.float32(n_lig) - np.float32(np.float32(n) * h) * np.float32(0.5)
    ci = np.floor((xyz - origin) / h).astype(np.int64)
    d = torch.from_numpy(xyz.astype(np.float64) - origin.astype(np.float64)).to(dev)
    cell = torch.from_numpy(ci).to(dev)
    idx = torch.arange(n, device=dev)
    lo = idx[None, None, :] * float(h) - d[:, :, None]
    s2 = sigma * math.sqrt(2.0)
    w = 0.5 * (torch.erf((lo + float(h)) / s2) - torch.erf(lo / s2))
    w = w * ((idx[None, None, :] - cell[:, :, None]).abs() <= k)
    f = torch.from_numpy(feat.astype(np.float64)).to(dev)
    wx, wy, wz = w[:, 0], w[:, 1], w[:, 2]
    a = (wz[:, :, None] * wy[:, None, :]).reshape(len(xyz), n * n)
    b = (wx[:, :, None] * f[:, None, :]).reshape(len(xyz), n * f.shape[1])
    return (a.T @ b).reshape(n, n, n, -1)


def _conv64(x, w, b, stride, residual):
    k = w.shape[2]
    p = k // 2
    n = x.shape[0]
    m = (n + 2 * p - k) // stride + 1
    xp = torch.nn.functional.pad(x, (0, 0, p, p, p, p, p, p))
    e = stride * (m - 1) + 1
    y = b.expand(m ** 3, -1).clone()
    for z in range(k):
        for r in range(k):
            for c in range(k):
                s = xp[z:z + e:stride, r:r + e:stride, c:c + e:stride].reshape(m ** 3, -1)
                y.addmm_(s, w[:, :, z, r, c].T)
    y = y.clamp_(min=0).reshape(m, m, m, -1)
    return x + y if residual else y


def _selu(x):
    return torch.nn.functional.selu(x)


def _affinity64(desc, W, xyz, feat, n_lig, dev):
    x = _grid64(desc, xyz, feat, n_lig, dev)
    for i, cv in enumerate(desc["conv"]):
        x = _conv64(x, W[f"conv{i}.w"], W[f"conv{i}.b"], cv["stride"], cv["residual"])
    x = x.permute(3, 0, 1, 2)
    if desc["pool"] and desc["pool"] > 1:
        x = torch.nn.functional.max_pool3d(x[None], desc["pool"])[0]
    cnn = torch.relu(W["cnn_dense.w"] @ x.reshape(-1) + W["cnn_dense.b"])
    if desc.get("cnn_dense2"):
        cnn = torch.relu(W["cnn_dense2.w"] @ cnn + W["cnn_dense2.b"])
    # edges: the float32 rule
    d = xyz[:, None, :] - xyz[None, :, :]
    s = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    cc, cn = np.float32(desc["cut_cov"]), np.float32(desc["cut_nc"])
    off = ~np.eye(len(xyz), dtype=bool)
    cov = (s < cc * cc) & off
    adj = {"cov": cov, "nc": ~cov & (s < cn * cn) & off}
    adj = {e: torch.from_numpy(a.astype(np.float64)).to(dev) for e, a in adj.items()}
    wid = weights.stage_widths(desc)
    h0 = torch.zeros(len(xyz), wid[0], dtype=torch.float64, device=dev)
    h0[:, :feat.shape[1]] = torch.from_numpy(feat.astype(np.float64)).to(dev)
    h = x_in = h0
    for si, st in enumerate(desc["sg_stages"]):
        x_in, H = h, wid[si]
        wih, whh = W[f"sg{si}.gru.w_ih"], W[f"sg{si}.gru.w_hh"]
        bih, bhh = W[f"sg{si}.gru.b_ih"], W[f"sg{si}.gru.b_hh"]
        for _ in range(st["steps"]):
            m = sum(adj[e] @ (h @ W[f"sg{si}.{e}.w"].T + W[f"sg{si}.{e}.b"]) for e in weights.edge_types(st["edges"]))
            gi, gh = m @ wih.T + bih, h @ whh.T + bhh
            r = torch.sigmoid(gi[:, :H] + gh[:, :H])
            z = torch.sigmoid(gi[:, H:2 * H] + gh[:, H:2 * H])
            t = torch.tanh(gi[:, 2 * H:] + r * gh[:, 2 * H:])
            h = (1 - z) * t + z * h
        if desc["sg_gate"] and si + 1 < len(desc["sg_stages"]):
            hh = torch.cat([h, h0], 1)
            h = torch.sigmoid(hh @ W[f"sg{si}.gate.wi"].T + W[f"sg{si}.gate.bi"]) * \
                (h @ W[f"sg{si}.gate.wj"].T + W[f"sg{si}.gate.bj"])
    hl, xl = h[:n_lig], x_in[:n_lig]
    if desc["sg_gather"] == "gated":
        sg = torch.sigmoid(torch.cat([hl, xl], 1) @ W["gather.wg"].T + W["gather.bg"]) * \
            (hl @ W["gather.wo"].T + W["gather.bo"])
    else:
        sg = hl @ W["gather.w"].T + W["gather.b"]
    sg = sg.sum(0)

    def dense(name, v):
        return W[f"{name}.w"] @ v + W[f"{name}.b"]

    if desc["fusion"] == "late":
        out = []
        for br, v in (("cnn_out", cnn), ("sg_out", sg)):
            for l in range(len(desc[br])):
                v = dense(f"{br}{l}", v)
                if l + 1 < len(desc[br]):
                    v = torch.relu(v)
            out.append(float(v[0]))
        return 0.5 * (out[0] + out[1])
    v = [cnn, sg]
    if desc["fusion"] == "mid":
        for br, u in (("cnn_out", cnn), ("sg_out", sg)):
            for l in range(len(desc[br])):
                u = _selu(dense(f"{br}{l}", u))
            v.append(u)
    v = torch.cat(v)
    for l in range(len(desc["head"])):
        u = dense(f"head{l}", v)
        if l + 1 < len(desc["head"]):
            u = _selu(u)
            if desc["head_residual"] and u.shape == v.shape:
                u = v + u
        v = u
    return float(v[0])


def exact(case, seed):
    if case["kind"] == "dense":
        x, w, b = _dense_inputs(case, seed)
        y = b.double().expand(case["B"], -1).clone()
        for k in range(0, case["K"], 1 << 16):
            y += x[:, k:k + (1 << 16)].double() @ w[:, k:k + (1 << 16)].double().T
        return torch.relu(y) if case["relu"] else y
    if work(case)["flops"] > 1e13:        # 64-bit convolutions of larger batches take over 20 seconds
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    desc = configs.model(case["preset"])
    W = {k: torch.from_numpy(v).to(dev).double() for k, v in _weights(case["preset"]).items()}
    return np.array([_affinity64(desc, W, *p, dev) for p in _poses(case, seed)], dtype=np.float64)
