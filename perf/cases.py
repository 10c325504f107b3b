"""What a user of this package has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``kind`` says which entry points it calls:

* ``pair``      build the target's tree and register the source, device buffers
                (``Tree.build`` + ``Tree.register``) or, with ``host``, the
                one call from pinned host buffers (``hgmm_register_pair_host``)
* ``build``     build a tree and export every level (the saved model)
* ``register``  register a new source to a tree the program keeps
* ``odometry``  a few sweeps of a drive through ``odometry.Odometry``
* ``batch``     many uneven pairs in one launch (``hgmm_batch_register``)
* ``descent``   the descent / M-step variants (``Tree.register_descent``)
* ``flat``      the single-level GMM: from a tree, then a registration
* ``forward``   the pose-proposal network's forward pass
* ``train``     optimisation steps of that network and its updated parameters
* ``propose``   the initial pose of one pair from its two trees

``exact`` restates each of them in plain float64 torch / numpy.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_1807_02587_gb300 import binding as B
from paper_1807_02587_gb300 import synth
from paper_1807_02587_gb300.odometry import Odometry

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WEIGHTS = os.path.join(ROOT, "paper_1807_02587_gb300", "weights", "proposal_mlp.npz")
EM_ITERS, N_MIN, LAM_C, EPS_REL = 8, 8.0, 0.01, 1e-3
MODES = {"local": B.HGMM_DESCENT_ML_LOCAL, "global": B.HGMM_DESCENT_ML_GLOBAL,
         "multipath": B.HGMM_DESCENT_MULTIPATH}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # object-scale pair: the smallest registration in use, all latency
        {"name": "corner pair", "kind": "pair", "scene": "corner", "n": 10000, "depth": 3, "iters": 30,
         "lam_c": -1.0, "host": False},
        # consecutive LiDAR sweeps from host buffers: the call a driver makes per frame
        {"name": "lidar pair from host", "kind": "pair", "scene": "lidar", "n": 120000, "depth": 4, "iters": 30,
         "lam_c": -1.0, "host": True},
        # two depth-camera frames already on the device
        {"name": "depth-camera pair", "kind": "pair", "scene": "depth", "n": 307200, "depth": 4, "iters": 30,
         "lam_c": -1.0, "host": False},
        # a mapping program's large cloud modelled and saved
        {"name": "large build", "kind": "build", "scene": "primitive", "n": 16_777_216, "depth": 4},
        # a large scan (unordered) localised against a kept model
        {"name": "large register", "kind": "register", "scene": "primitive", "n": 16_777_216, "n_tgt": 4_000_000,
         "depth": 4, "iters": 10, "lam_c": -1.0},
        # streaming: builds and three-start registrations overlapped on two streams
        {"name": "odometry", "kind": "odometry", "frames": 4, "n": 120000, "depth": 4, "iters": 30},
        # the batched form at its documented size
        {"name": "batch of 256", "kind": "batch", "pairs": 256, "n_lo": 2000, "n_hi": 200000, "iters": 30},
        # every likely path descended instead of the best one
        {"name": "multipath descent", "kind": "descent", "scene": "lidar", "n": 120000, "depth": 4, "iters": 30,
         "mode": "multipath", "tau": 0.1, "eq7": False},
        # the flat model at the scale of the depth-4 leaves
        {"name": "flat lidar", "kind": "flat", "scene": "lidar", "n": 120000, "depth": 4, "iters": 30},
        # proposals for a large batch of pairs
        {"name": "network forward", "kind": "forward", "batch": 8192},
        # mini-batches of the documented training run, then the parameters
        {"name": "network training", "kind": "train", "rows": 16384, "batch": 1024, "steps": 4, "gather": True},
        # one proposal: the smallest call, launches and latency only
        {"name": "propose one pair", "kind": "propose", "n": 50000, "depth": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "build", "register", "odometry", "batch", "descent", "flat",
                       "forward", "train", "propose"])
    scene = rng.choice(["corner", "lidar", "depth", "primitive"])
    lam_c = rng.choice([-1.0, -1.0, 0.0])
    if kind == "pair":
        return {"kind": kind, "scene": scene, "n": _log_int(rng, 1000, 300000), "depth": rng.randint(2, 5),
                "iters": rng.randint(5, 40), "lam_c": lam_c, "host": rng.random() < 0.4}
    if kind == "build":
        return {"kind": kind, "scene": "primitive", "n": _log_int(rng, 1000, 16_000_000), "depth": rng.randint(2, 5)}
    if kind == "register":
        return {"kind": kind, "scene": "primitive", "n": _log_int(rng, 1000, 16_000_000),
                "n_tgt": _log_int(rng, 20000, 2_000_000), "depth": rng.randint(2, 5), "iters": rng.randint(3, 10),
                "lam_c": lam_c}
    if kind == "odometry":
        return {"kind": kind, "frames": rng.randint(2, 5), "n": _log_int(rng, 10000, 100000),
                "depth": rng.randint(3, 4), "iters": rng.randint(10, 30)}
    if kind == "batch":
        return {"kind": kind, "pairs": rng.randint(2, 48), "n_lo": 2000, "n_hi": _log_int(rng, 4000, 120000),
                "iters": rng.randint(10, 30)}
    if kind == "descent":
        return {"kind": kind, "scene": scene, "n": _log_int(rng, 2000, 120000), "depth": rng.randint(2, 4),
                "iters": rng.randint(5, 20), "mode": rng.choice(["local", "global", "multipath"]),
                "tau": rng.choice([0.02, 0.05, 0.1, 0.25]), "eq7": rng.random() < 0.4}
    if kind == "flat":
        return {"kind": kind, "scene": scene, "n": _log_int(rng, 2000, 90000), "depth": rng.randint(2, 4),
                "iters": rng.randint(3, 20)}
    if kind == "forward":
        return {"kind": kind, "batch": _log_int(rng, 1, 8192)}
    if kind == "train":
        return {"kind": kind, "rows": 8192, "batch": _log_int(rng, 100, 4096), "steps": rng.randint(1, 4),
                "gather": rng.random() < 0.7}
    return {"kind": kind, "n": _log_int(rng, 5000, 100000), "depth": rng.randint(2, 4)}


# ------------------------------------------------------------------ the inputs
def _f4(P):
    """(N, 3) on the device -> contiguous (N, 4) float32 with a zero pad."""
    P = torch.as_tensor(P)
    out = torch.zeros((P.shape[0], 4), dtype=torch.float32, device="cuda")
    out[:, :3] = P.to(device="cuda", dtype=torch.float32)
    return out


def _thin(rng, P, n):
    """At most n of the points, in their own (scan) order."""
    if P.shape[0] <= n:
        return P
    return P[np.sort(rng.choice(P.shape[0], size=n, replace=False))]


def _sample_scene(scene, n, gen):
    """n area-weighted samples of a plane/box/sphere scene, in random order, with 5 mm noise."""
    rects, spheres = scene
    areas = [float(np.linalg.norm(np.cross(u, v))) for _, u, v in rects] + [4 * math.pi * r * r for _, r in spheres]
    cdf = torch.tensor(np.cumsum(areas) / np.sum(areas), dtype=torch.float32, device="cuda")
    k = torch.searchsorted(cdf, torch.rand(n, generator=gen, device="cuda")).clamp_(max=len(areas) - 1)
    tab = np.zeros((len(areas), 3, 3))
    for i, (o, u, v) in enumerate(rects):
        tab[i] = [o, u, v]
    for i, (c, r) in enumerate(spheres):
        tab[len(rects) + i] = [c, [r, 0, 0], [0, 0, 0]]
    tab = torch.tensor(tab, dtype=torch.float32, device="cuda")
    ab = torch.rand((n, 2), generator=gen, device="cuda")
    P = tab[k, 0] + ab[:, :1] * tab[k, 1] + ab[:, 1:] * tab[k, 2]
    if spheres:
        ball = k >= len(rects)
        d = torch.randn((n, 3), generator=gen, device="cuda")
        d /= d.norm(dim=1, keepdim=True)
        P = torch.where(ball[:, None], tab[k, 0] + tab[k, 1, :1] * d, P)
    return P + 0.005 * torch.randn((n, 3), generator=gen, device="cuda")


def _moved(P, T):
    T = torch.tensor(T, dtype=torch.float32, device="cuda")
    return P @ T[:3, :3].T + T[:3, 3]


def _primitive_clouds(seed, n_tgt, n_src, max_deg, max_t):
    rng = synth.make_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    scene = synth.primitive_scene(rng)
    T = synth.rigid(synth.random_rotation(rng, max_deg), rng.uniform(-max_t, max_t, 3))
    return _f4(_moved(_sample_scene(scene, n_tgt, gen), T)), _f4(_sample_scene(scene, n_src, gen))


def _clouds(case, seed):
    """(target, source) of a case as (N, 4) float32 device tensors."""
    n, scene = case["n"], case.get("scene")
    if scene == "primitive":
        return _primitive_clouds(seed, case.get("n_tgt", n), n, 3.0, 0.03)
    rng = synth.make_rng(seed + 1)
    if scene == "corner":
        p = synth.corner_pair(seed, n=n, max_deg=3.0, max_t=0.02)
    elif scene == "lidar":
        p = synth.lidar_pair(seed)
    else:
        p = synth.depth_pair(seed)
    return _f4(_thin(rng, p["tgt"], n)), _f4(_thin(rng, p["src"], n))


def _sweeps(case, seed):
    rng = synth.make_rng(seed + 1)
    return [_f4(_thin(rng, f, case["n"])) for f in synth.lidar_sequence(seed, frames=case["frames"])["frames"]]


def _so3_clouds(case, seed):
    """Two samples of a scene, the target turned by any rotation."""
    rng = synth.make_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    scene = synth.primitive_scene(rng)
    T = synth.rigid(synth.uniform_rotation(rng), rng.uniform(-0.1, 0.1, 3))
    return _f4(_moved(_sample_scene(scene, case["n"], gen), T)), _f4(_sample_scene(scene, case["n"], gen))


def _batch_inputs(case, seed):
    """All clouds in one buffer, the ranges and depths of the pairs (poses within 10 degrees)."""
    rng = synth.make_rng(seed)
    sizes = np.exp(rng.uniform(np.log(case["n_lo"]), np.log(case["n_hi"]), size=case["pairs"])).astype(np.int64)
    depths = rng.integers(3, 5, size=case["pairs"]).astype(np.int32)
    seeds = rng.integers(0, 2**31 - 1, size=case["pairs"])
    clouds, t_rng, s_rng, at = [], [], [], 0
    for k, n in enumerate(sizes):
        t, s = _primitive_clouds(int(seeds[k]), int(n), int(n), 10.0, 0.1)
        clouds += [t, s]
        t_rng.append([at, at + n])
        s_rng.append([at + n, at + 2 * n])
        at += 2 * int(n)
    return torch.cat(clouds), np.array(t_rng), np.array(s_rng), depths, int(sizes.max())


def _network_rows(rows, seed):
    """Feature rows like those of real trees: 2 x 64 nodes of (weight, mean, covariance), a quarter
    of the slots empty; and pose labels near the four sign flips of a canonical frame."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    x = torch.empty((rows, 128, 10), device="cuda")
    x[..., 0] = -torch.log(torch.rand((rows, 128), generator=gen, device="cuda") + 1e-6)
    x[..., 1:4] = 0.9 * torch.randn((rows, 128, 3), generator=gen, device="cuda")
    x[..., 4:] = 0.1 * torch.randn((rows, 128, 6), generator=gen, device="cuda")
    for a in (4, 7, 9):
        x[..., a] = 0.6 * torch.rand((rows, 128), generator=gen, device="cuda")
    x *= (torch.rand((rows, 128, 1), generator=gen, device="cuda") > 0.25)
    flips = torch.tensor([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=torch.float32, device="cuda")
    f = flips[torch.randint(4, (rows,), generator=gen, device="cuda")]
    w = 0.05 * torch.randn((rows, 3), generator=gen, device="cuda")
    K = torch.zeros((rows, 3, 3), device="cuda")
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -w[:, 2], w[:, 1], -w[:, 0]
    R = torch.linalg.matrix_exp(K - K.transpose(1, 2)) * f[:, None, :]
    lab = torch.cat([R.reshape(rows, 9), 0.05 * torch.randn((rows, 3), generator=gen, device="cuda")], dim=1)
    return x.reshape(rows, 1280).to(torch.bfloat16).contiguous(), lab.float().contiguous()


def _weights():
    with np.load(WEIGHTS) as f:
        return f["params"].astype(np.float32)


def _network(max_batch):
    net = B.Mlp(max_batch)
    B.hgmm_mlp_set_params(net.handle, _weights())
    return net


def _train_inputs(case, seed):
    x, lab = _network_rows(case["rows"], seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 1)
    idx = [torch.randperm(case["rows"], generator=gen, device="cuda")[:case["batch"]].to(torch.int32).contiguous()
           for _ in range(case["steps"])]
    return x, lab, idx


LEARNING_RATE = 1e-4


# ------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "pair":
        tgt, src = _clouds(case, seed)
        n = max(tgt.shape[0], src.shape[0])
        st["tree"] = B.Tree(n, case["depth"])
        if case["host"]:
            tgt, src = tgt.cpu().pin_memory(), src.cpu().pin_memory()
            st["prm"] = B.params()
        else:
            st["hist"] = torch.zeros((case["iters"], 16), dtype=torch.float64, device="cuda")
            st["obj"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        st["tgt"], st["src"] = tgt, src
    elif kind == "build":
        st["tgt"], _ = _primitive_clouds(seed, case["n"], 8, 3.0, 0.03)
        st["tree"] = B.Tree(case["n"], case["depth"])
    elif kind == "register":
        tgt, st["src"] = _clouds(case, seed)
        st["tree"] = B.Tree(max(case["n"], case["n_tgt"]), case["depth"])
        st["tree"].build(tgt, case["depth"])
        st["hist"] = torch.zeros((case["iters"], 16), dtype=torch.float64, device="cuda")
        st["obj"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "odometry":
        st["frames"] = _sweeps(case, seed)
        st["odo"] = Odometry(case["n"], case["depth"], case["iters"])
    elif kind == "batch":
        st["points"], t_rng, s_rng, depths, most = _batch_inputs(case, seed)
        n = case["pairs"]
        st["batch"] = B.Batch(most, 4, n)
        B.hgmm_batch_set_shape(st["batch"].handle, 8)
        B.hgmm_batch_plan_ranges(st["batch"].handle, t_rng, s_rng, depths)
        st["T"] = torch.zeros((n, 16), dtype=torch.float64, device="cuda")
        st["obj"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        st["status"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    elif kind == "descent":
        tgt, st["src"] = _clouds(case, seed)
        st["tree"] = B.Tree(max(tgt.shape[0], st["src"].shape[0]), case["depth"])
        st["tree"].build(tgt, case["depth"])
        st["hist"] = torch.zeros((case["iters"], 16), dtype=torch.float64, device="cuda")
        st["obj"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "flat":
        tgt, st["src"] = _clouds(case, seed)
        n = max(tgt.shape[0], st["src"].shape[0])
        st["tree"] = B.Tree(n, case["depth"])
        st["tree"].build(tgt, case["depth"])
        st["flat"] = B.Flat(n, B.hgmm_node_count(case["depth"]))
        st["hist"] = torch.zeros((case["iters"], 16), dtype=torch.float64, device="cuda")
        st["obj"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "forward":
        st["x"], _ = _network_rows(case["batch"], seed)
        st["net"] = _network(case["batch"])
        st["y"] = torch.zeros((case["batch"], 9), dtype=torch.float32, device="cuda")
    elif kind == "train":
        st["x"], st["lab"], st["idx"] = _train_inputs(case, seed)
        st["net"] = _network(case["batch"])
        st["loss"] = torch.zeros(case["steps"], dtype=torch.float32, device="cuda")
    elif kind == "propose":
        tgt, src = _so3_clouds(case, seed)
        st["tgt"], st["src"] = B.Tree(case["n"], case["depth"]), B.Tree(case["n"], case["depth"])
        st["tgt"].build(tgt, case["depth"])
        st["src"].build(src, case["depth"])
        st["net"] = _network(1)
        st["T"] = torch.zeros((4, 4), dtype=torch.float64, device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "pair":
        if case["host"]:
            return B.hgmm_register_pair_host(st["tree"].handle, st["tgt"], st["src"], case["depth"], st["prm"],
                                             iters=case["iters"])
        st["tree"].build(st["tgt"], case["depth"])
    if kind in ("pair", "register"):
        T = st["tree"].register(st["src"], iters=case["iters"], lam_c=case["lam_c"], T_hist=st["hist"])
        B.hgmm_register_objective(st["tree"].handle, st["obj"])
        return {"T": T, "T_hist": st["hist"], "objective": st["obj"]}
    if kind == "build":
        st["tree"].build(st["tgt"], case["depth"])
        return [st["tree"].export(l) for l in range(case["depth"])]
    if kind == "odometry":
        T = st["odo"].run(st["frames"])
        st["odo"].sync()
        return T
    if kind == "batch":
        B.hgmm_batch_register(st["batch"].handle, st["points"], st["T"], iters=case["iters"],
                              pair_status=st["status"])
        B.hgmm_batch_objective(st["batch"].handle, st["obj"])
        return {"T": st["T"], "objective": st["obj"], "status": st["status"]}
    if kind == "descent":
        T = st["tree"].register_descent(st["src"], MODES[case["mode"]], tau=case["tau"], iters=case["iters"],
                                        T_hist=st["hist"], full_eq7=case["eq7"])
        B.hgmm_register_objective(st["tree"].handle, st["obj"])
        return {"T": T, "T_hist": st["hist"], "objective": st["obj"]}
    if kind == "flat":
        st["flat"].from_tree(st["tree"])
        T = st["flat"].register(st["src"], iters=case["iters"], T_hist=st["hist"])
        B.hgmm_flat_objective(st["flat"].handle, st["obj"])
        return {"T": T, "T_hist": st["hist"], "objective": st["obj"]}
    if kind == "forward":
        return B.hgmm_mlp_forward(st["net"].handle, st["x"], st["y"])
    if kind == "train":
        h, b = st["net"].handle, case["batch"]
        for k in range(case["steps"]):
            if case["gather"]:
                B.hgmm_mlp_train_step(h, st["x"], st["lab"], b, index=st["idx"][k], lr=LEARNING_RATE,
                                      loss=st["loss"][k:])
            else:
                B.hgmm_mlp_train_step(h, st["x"], st["lab"], b, lr=LEARNING_RATE, loss=st["loss"][k:])
        return {"loss": st["loss"], "params": B.hgmm_mlp_get_params(h)}
    return B.hgmm_propose(st["tgt"].handle, st["src"].handle, st["net"].handle, st["T"])


# ------------------------------------------------------------------------ work
def _nodes(depth):
    return sum(8 ** (l + 1) for l in range(depth))


def _build_work(n, depth):
    """Points read once, the node table written; 355 flops per point, EM iteration and level."""
    return 16 * n + 128 * _nodes(depth), 355.0 * n * EM_ITERS * depth


def _register_work(n, depth, iters):
    """Source read once, the node table read once; 30 + 168 flops per visited level, per point and round."""
    return 16 * n + 96 * _nodes(depth), float(n) * iters * (30 + 168 * depth)


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    depth, iters = case.get("depth", 4), case.get("iters", 0)
    if kind in ("pair", "odometry"):
        b, f = _build_work(n, depth)
        rb, rf = _register_work(n, depth, iters)
        k = case["frames"] - 1 if kind == "odometry" else 1
        starts = 3 if kind == "odometry" else 1
        return {"bytes": k * (b + rb), "flops": k * (f + starts * rf)}
    if kind == "build":
        b, f = _build_work(n, depth)
        return {"bytes": b, "flops": f}
    if kind == "register":
        b, f = _register_work(n, depth, iters)
        return {"bytes": b, "flops": f}
    if kind == "batch":
        mean = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        b, f = _build_work(mean, 4)
        rb, rf = _register_work(mean, 4, iters)
        return {"bytes": case["pairs"] * (b + rb), "flops": case["pairs"] * (f + rf)}
    if kind == "descent":
        b, f = _register_work(n, depth, iters)
        return {"bytes": b, "flops": f}
    if kind == "flat":
        J = min(0.45 * 8 ** depth, n / 50.0)
        return {"bytes": 16 * n + 96 * J, "flops": 49.0 * n * J * iters}
    params = 396041
    if kind == "forward":
        return {"bytes": case["batch"] * (2560 + 36) + 2 * params, "flops": 2.0 * case["batch"] * params}
    if kind == "train":
        return {"bytes": case["steps"] * (case["batch"] * (2560 + 48) + 24 * params) + 4 * params,
                "flops": 6.0 * case["batch"] * params * case["steps"]}
    return {"bytes": 2 * 72 * 232 + 2 * params + 128, "flops": 2.0 * params}


# ------------------------------------------------- the same in plain 64 bits
def _eig(S):
    """Eigenvalues descending, eigenvectors in columns, the largest entry of each positive."""
    w, V = np.linalg.eigh(S)
    w, V = w[..., ::-1].copy(), V[..., ::-1].copy()
    k = np.argmax(np.abs(V), axis=-2)
    s = np.take_along_axis(V, k[..., None, :], axis=-2)[..., 0, :]
    return w, V * np.where(s < 0, -1.0, 1.0)[..., None, :]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _inverse(S):
    """Inverse and log-determinant of symmetric positive 3x3 stacks (cofactors); singular ones give zeros."""
    a, b, c, d, e, f = S[:, 0, 0], S[:, 0, 1], S[:, 0, 2], S[:, 1, 1], S[:, 1, 2], S[:, 2, 2]
    A, Bc, C = d * f - e * e, c * e - b * f, b * e - c * d
    det = a * A + b * Bc + c * C
    ok = det > 0
    i = torch.where(ok, 1.0 / torch.where(ok, det, torch.ones_like(det)), torch.zeros_like(det))
    rows = torch.stack([A, Bc, C, Bc, a * f - c * c, b * c - a * e, C, b * c - a * e, a * d - b * b], 1) * i[:, None]
    return rows.view(-1, 3, 3), torch.where(ok, torch.log(torch.where(ok, det, torch.ones_like(det))), torch.zeros_like(det))


def _scores(Z, node, lv):
    """log(pi N(z | node)) of every point and its candidate nodes (N, K); -inf for dead ones."""
    if "inv" not in lv:
        inv, ld = _inverse(lv["S"])
        const = torch.log(lv["pi"].clamp(min=1e-300)) - 0.5 * ld - 1.5 * math.log(2 * math.pi)
        lv["inv"], lv["const"] = inv, torch.where(lv["live"], const, torch.full_like(const, -math.inf))
    d = Z[:, None, :] - lv["mu"][node]
    q = torch.einsum("nki,nkij,nkj->nk", d, lv["inv"][node], d)
    return lv["const"][node] - 0.5 * q


def _posterior(s):
    m = s.max(dim=1, keepdim=True).values
    none = ~torch.isfinite(m)
    p = torch.exp(s - torch.where(none, torch.zeros_like(m), m))
    t = p.sum(dim=1, keepdim=True)
    return torch.where(none, torch.zeros_like(p), p / torch.where(none, torch.ones_like(t), t)), ~none[:, 0]


def _tree64(P, depth):
    Z = P[:, :3].double()
    n = Z.shape[0]
    mu = Z.mean(dim=0)
    S = (Z - mu).T @ (Z - mu) / n
    extent = float((Z.max(dim=0).values - Z.min(dim=0).values).norm())
    eps = (float(np.float32(EPS_REL)) * extent) ** 2
    eye = torch.eye(3, dtype=torch.float64, device="cuda")
    eight = torch.arange(8, device="cuda")
    parent = torch.zeros(n, dtype=torch.int64, device="cuda")
    p_mu, p_S, p_cnt = mu[None], S[None], torch.tensor([n], device="cuda")
    p_live = torch.tensor([True], device="cuda")
    root_lam, root_V = _eig(S.cpu().numpy())
    p_lam, p_V = root_lam[None], root_V[None]
    signs = np.array([[1.0 if (k >> a) & 1 else -1.0 for a in range(3)] for k in range(8)])
    levels = []
    for _ in range(depth):
        alive = (p_live & (p_cnt > 0)).repeat_interleave(8)
        off = np.einsum("pij,kj,pj->pki", p_V, signs, 0.5 * np.sqrt(np.maximum(p_lam, 0.0)))
        lv = {"live": alive.clone(), "pi": torch.where(alive, 0.125, 0.0).double()}
        lv["mu"] = p_mu.repeat_interleave(8, 0) + _dev(off.reshape(-1, 3)) * alive[:, None]
        lv["S"] = (p_S.repeat_interleave(8, 0) / 4 + eps * eye) * alive[:, None, None]
        m = alive.shape[0]
        node = parent[:, None] * 8 + eight
        flat = node.reshape(-1)
        for _ in range(EM_ITERS):
            g, _ = _posterior(_scores(Z, node, lv))
            S0 = torch.zeros(m, dtype=torch.float64, device="cuda").index_add_(0, flat, g.reshape(-1))
            d = Z[:, None, :] - lv["mu"][node]
            gd = (g[..., None] * d).reshape(-1, 3)
            S1 = torch.zeros((m, 3), dtype=torch.float64, device="cuda").index_add_(0, flat, gd)
            S2 = torch.zeros((m, 9), dtype=torch.float64, device="cuda").index_add_(
                0, flat, (gd[:, :, None] * d.reshape(-1, 3)[:, None, :]).reshape(-1, 9)).view(m, 3, 3)
            live = lv["live"] & (S0 >= N_MIN) & (S0 > 0)
            r = 1.0 / torch.where(live, S0, torch.ones_like(S0))
            dm = S1 * r[:, None]
            cov = S2 * r[:, None, None] - dm[:, :, None] * dm[:, None, :] + eps * eye
            lv = {"live": live, "pi": torch.where(live, S0 / p_cnt.repeat_interleave(8).clamp(min=1), 0.0),
                  "mu": torch.where(live[:, None], lv["mu"] + dm, lv["mu"]),
                  "S": torch.where(live[:, None, None], cov, lv["S"])}
        s = _scores(Z, node, lv)
        best = torch.where(torch.isfinite(s.max(dim=1).values), s.argmax(dim=1), torch.zeros_like(parent))
        parent = parent * 8 + best
        lv["count"] = torch.bincount(parent, minlength=m)
        lam, V = np.ones((m, 3)), np.tile(np.eye(3), (m, 1, 1))
        k = lv["live"].cpu().numpy()
        if k.any():
            lam[k], V[k] = _eig(lv["S"].cpu().numpy()[k])
        lv["lam"], lv["V"] = lam, V
        cx = np.where(k, lam[:, 2] / lam.sum(axis=1), 1.0)
        lv["cx"] = _dev(cx)
        lv["P"] = _dev(np.einsum("mik,mk,mjk->mij", V, 1.0 / np.maximum(lam, eps), V))
        levels.append(lv)
        p_mu, p_S, p_cnt, p_live, p_lam, p_V = lv["mu"], lv["S"], lv["count"], lv["live"], lam, V
    return {"levels": levels, "eps": eps, "mu": mu, "S": S, "lam": root_lam, "V": root_V}


def _descend64(tree, Zp, mode, tau, lam_c):
    """(point, level offset + node, gamma) of every stopping node."""
    L = len(tree["levels"])
    eight = torch.arange(8, device="cuda")
    pt = torch.arange(Zp.shape[0], device="cuda")
    par = torch.full_like(pt, 0)
    gp = torch.ones(Zp.shape[0], dtype=torch.float64, device="cuda")
    out, off, prev = [], 0, 0
    for l, lv in enumerate(tree["levels"]):
        node = (par[:, None] * 8 if l else torch.zeros_like(par)[:, None]) + eight
        s = _scores(Zp[pt], node, lv)
        post, any_live = _posterior(s)
        if l:
            out.append((pt[~any_live], prev + par[~any_live], gp[~any_live]))
        pt, node, gp, post, s = pt[any_live], node[any_live], gp[any_live], post[any_live], s[any_live]
        if mode == "multipath":
            g = post * gp[:, None]
            r, c = torch.nonzero(lv["live"][node] & (g >= tau), as_tuple=True)
            pt, par, gp = pt[r], node[r, c], g[r, c]
        else:
            c = s.argmax(dim=1)
            r = torch.arange(pt.shape[0], device="cuda")
            gp = post[r, c] * (gp if mode == "global" else 1.0)
            par = node[r, c]
        stop = lv["cx"][par] <= lam_c if l < L - 1 else torch.ones_like(par, dtype=torch.bool)
        out.append((pt[stop], off + par[stop], gp[stop]))
        pt, par, gp = pt[~stop], par[~stop], gp[~stop]
        prev, off = off, off + lv["pi"].shape[0]
    return tuple(torch.cat([o[k] for o in out]) for k in range(3))


def _skew(m):
    z = torch.zeros_like(m[:, 0])
    return torch.stack([z, -m[:, 2], m[:, 1], m[:, 2], z, -m[:, 0], -m[:, 1], m[:, 0], z], 1).view(-1, 3, 3)


def _normal64(w, m, P, d):
    """sum w B P B^T, sum w B P d and sum w d^T P d with B = [[m]x; I]."""
    K = _skew(m)
    KP = K @ P * w[:, None, None]
    Pw = P * w[:, None, None]
    H = torch.zeros((6, 6), dtype=torch.float64, device="cuda")
    H[:3, :3] = torch.einsum("kij,klj->il", KP, K)
    H[:3, 3:] = KP.sum(dim=0)
    H[3:, :3] = H[:3, 3:].T
    H[3:, 3:] = Pw.sum(dim=0)
    Pd = (Pw @ d[:, :, None])[:, :, 0]
    g = torch.cat([(K @ Pd[:, :, None])[:, :, 0].sum(dim=0), Pd.sum(dim=0)])
    return H.cpu().numpy(), g.cpu().numpy(), float((d * Pd).sum())


def _step64(H, g, T):
    x = np.linalg.solve(H, g)
    th = np.linalg.norm(x[:3])
    K = np.array([[0, -x[2], x[1]], [x[2], 0, -x[0]], [-x[1], x[0], 0]])
    R = np.eye(3) + K if th < 1e-300 else np.eye(3) + np.sin(th) / th * K + (1 - np.cos(th)) / th**2 * (K @ K)
    dT = np.eye(4)
    dT[:3, :3], dT[:3, 3] = R, x[3:]
    return dT @ T


def _move64(Z, T):
    return Z @ _dev(T[:3, :3]).T + _dev(T[:3, 3])


def _register64(tree, src, iters, lam_c=-1.0, mode="local", tau=0.0, eq7=False, T0=None):
    Z = src[:, :3].double()
    T = np.eye(4) if T0 is None else np.array(T0, float)
    lam_c = float(np.float32(LAM_C if lam_c < 0 else lam_c))
    mu = torch.cat([lv["mu"] for lv in tree["levels"]])
    P = torch.cat([lv["P"] for lv in tree["levels"]])
    hist, obj, n = [], 0.0, Z.shape[0]
    for _ in range(iters):
        Zp = _move64(Z, T)
        i, r, g = _descend64(tree, Zp, mode, tau, lam_c)
        if eq7:
            H, b, obj = _normal64(g / n, Zp[i], P[r], mu[r] - Zp[i])
        else:
            M0 = torch.zeros(mu.shape[0], dtype=torch.float64, device="cuda").index_add_(0, r, g)
            M1 = torch.zeros_like(mu).index_add_(0, r, g[:, None] * (Zp[i] - mu[r]))
            k = M0 > 0
            o = M1[k] / M0[k][:, None]
            H, b, obj = _normal64(M0[k] / n, mu[k] + o, P[k], -o)
        T = _step64(H, b, T)
        hist.append(T.reshape(16))
    return T, np.array(hist), obj


def _flat64(tree, src, iters):
    glob, comp = None, []
    L = len(tree["levels"])
    for l, lv in enumerate(tree["levels"]):
        glob = lv["pi"] * (1.0 if l == 0 else glob.repeat_interleave(8))
        leaf = lv["live"].clone()
        if l + 1 < L:
            leaf &= ~tree["levels"][l + 1]["live"].view(-1, 8).any(dim=1)
        comp.append((glob[leaf], lv["mu"][leaf], lv["S"][leaf], lv["P"][leaf]))
    pi, mu, S, P = (torch.cat([c[k] for c in comp]) for k in range(4))
    pi = pi / pi.sum()
    inv, ld = _inverse(S)
    const = torch.log(pi) - 0.5 * ld
    # the quadratic form as one product: [xx, xy, xz, yy, yz, zz, x, y, z, 1] about a common centre
    c0 = mu.mean(dim=0)
    m = mu - c0
    im = (inv @ m[:, :, None])[:, :, 0]
    W = torch.stack([inv[:, 0, 0], 2 * inv[:, 0, 1], 2 * inv[:, 0, 2], inv[:, 1, 1], 2 * inv[:, 1, 2], inv[:, 2, 2],
                     -2 * im[:, 0], -2 * im[:, 1], -2 * im[:, 2], (m * im).sum(dim=1)], 1)
    Z = src[:, :3].double()
    n, T, hist, obj = Z.shape[0], np.eye(4), [], 0.0
    for _ in range(iters):
        Zp = _move64(Z, T) - c0
        M0 = torch.zeros(pi.shape[0], dtype=torch.float64, device="cuda")
        M1 = torch.zeros((pi.shape[0], 3), dtype=torch.float64, device="cuda")
        for z in Zp.split(16384):
            x, y, w = z[:, 0], z[:, 1], z[:, 2]
            F = torch.stack([x * x, x * y, x * w, y * y, y * w, w * w, x, y, w, torch.ones_like(x)], 1)
            g = torch.softmax(const - 0.5 * (F @ W.T), dim=1)
            M0 += g.sum(dim=0)
            M1 += g.T @ z
        k = M0 > 0
        o = M1[k] / M0[k][:, None] - m[k]
        H, b, obj = _normal64(M0[k] / n, mu[k] + o, P[k], -o)
        T = _step64(H, b, T)
        hist.append(T.reshape(16))
    return T, np.array(hist), obj


def _unpack64(p):
    out, k = [], 0
    for shape in synth.MLP_SHAPES:
        c = int(np.prod(shape))
        out.append(p[k:k + c].view(shape))
        k += c
    return out


def _forward64(p, x):
    W1, b1, W2, b2, W3, b3 = _unpack64(p)
    h = torch.relu(x.double() @ W1.T + b1)
    return torch.relu(h @ W2.T + b2) @ W3.T + b3


def _columns64(y):
    b1 = y[:, 0:3] / y[:, 0:3].norm(dim=1, keepdim=True)
    u = y[:, 3:6] - (b1 * y[:, 3:6]).sum(dim=1, keepdim=True) * b1
    b2 = u / u.norm(dim=1, keepdim=True)
    return torch.stack([b1, b2, torch.linalg.cross(b1, b2)], dim=2)


def _train64(case, seed):
    x, lab, idx = _train_inputs(case, seed)
    p = _dev(_weights()).double()
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for k in range(case["steps"]):
        rows = idx[k].long() if case["gather"] else slice(0, case["batch"])
        q = p.clone().requires_grad_(True)
        y, l = _forward64(q, x[rows]), lab[rows].double()
        e = ((_columns64(y) - l[:, :9].view(-1, 3, 3))**2).sum(dim=(1, 2)) + ((y[:, 6:9] - l[:, 9:])**2).sum(dim=1)
        e.mean().backward()
        losses.append(float(e.mean()))
        m = 0.9 * m + 0.1 * q.grad
        v = 0.999 * v + 0.001 * q.grad**2
        p = p - LEARNING_RATE * (m / (1 - 0.9**(k + 1))) / ((v / (1 - 0.999**(k + 1))).sqrt() + 1e-8)
    return {"loss": np.array(losses), "params": p.cpu().numpy()}


def _features64(tree):
    """640 features of a tree in its canonical frame, and that frame (c, s, V)."""
    V = tree["V"].copy()
    flip = np.linalg.det(V) < 0
    if flip:
        V[:, 2] = -V[:, 2]
    c, s = tree["mu"].cpu().numpy(), math.sqrt(np.maximum(tree["lam"], 0).sum())
    l0, l1 = ({k: lv[k].cpu().numpy() for k in ("pi", "mu", "S", "live")} for lv in tree["levels"][:2])
    F = np.zeros((64, 10))

    def entry(w, mu, S):
        C = V.T @ S @ V
        return np.concatenate([[64 * w], V.T @ (mu - c) / s, 16 * C[np.triu_indices(3)] / s**2])

    for k in range(8):
        if not l0["live"][k]:
            continue
        at = 8 * (k ^ (4 if flip else 0))
        kids = sorted((j for j in range(8 * k, 8 * k + 8) if l1["live"][j]), key=lambda j: (-l1["pi"][j], j))
        if not kids:
            F[at] = entry(l0["pi"][k], l0["mu"][k], l0["S"][k])
        for r, j in enumerate(kids):
            F[at + r] = entry(l0["pi"][k] * l1["pi"][j], l1["mu"][j], l1["S"][j])
    return F.reshape(-1), (c, s, V)


def _propose64(tgt, src):
    (Ft, (ct, st, Vt)), (Fs, (cs, _, Vs)) = (_features64(_tree64(c, 2)) for c in (tgt, src))
    y = _forward64(_dev(_weights()).double(), _dev(np.concatenate([Fs, Ft])[None]))
    T = np.eye(4)
    T[:3, :3] = Vt @ _columns64(y)[0].cpu().numpy() @ Vs.T
    T[:3, 3] = ct + st * (Vt @ y[0, 6:9].cpu().numpy()) - T[:3, :3] @ cs
    return T


def _odometry64(case, seed):
    frames = _sweeps(case, seed)
    T = [np.eye(4)]
    for k in range(1, len(frames)):
        tree = _tree64(frames[k - 1], case["depth"])
        best = None
        for deg in (0.0, 3.0, -3.0):
            R = np.eye(4)
            R[:3, :3] = synth.axis_angle_matrix([0, 0, 1], np.radians(deg))
            got = _register64(tree, frames[k], case["iters"], T0=R @ T[-1])
            if best is None or got[2] < best[2]:
                best = got
        T.append(best[0])
    return np.array(T)


EXACT_POINTS = 400_000


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pair", "register", "descent", "flat"):
        if max(case["n"], case.get("n_tgt", 0)) > EXACT_POINTS:
            return None
        tgt, src = _clouds(case, seed)
        tree = _tree64(tgt, case["depth"])
        if kind == "flat":
            T, hist, obj = _flat64(tree, src, case["iters"])
        else:
            T, hist, obj = _register64(tree, src, case["iters"], lam_c=case.get("lam_c", -1.0),
                                       mode=case.get("mode", "local"), tau=float(np.float32(case.get("tau", 0.0))),
                                       eq7=case.get("eq7", False))
        if case.get("host"):
            return T
        return {"T": T, "T_hist": hist, "objective": np.array([obj])}
    if kind == "build":
        if case["n"] > EXACT_POINTS:
            return None
        tgt, _ = _primitive_clouds(seed, case["n"], 8, 3.0, 0.03)
        out = []
        for lv in _tree64(tgt, case["depth"])["levels"]:
            out.append({"pi": torch.where(lv["live"], lv["pi"], 0.0).cpu().numpy(), "mu": lv["mu"].cpu().numpy(),
                        "Sigma": lv["S"].cpu().numpy(), "live": None, "count": None,
                        "complexity": lv["cx"].cpu().numpy(), "lam": lv["lam"]})
        return out
    if kind == "odometry":
        return _odometry64(case, seed)
    if kind == "batch":
        points, t_rng, s_rng, depths, _ = _batch_inputs(case, seed)
        if points.shape[0] > 8 * EXACT_POINTS or case["pairs"] > 64:
            return None
        got = [_register64(_tree64(points[t[0]:t[1]], int(d)), points[s[0]:s[1]], case["iters"])
               for t, s, d in zip(t_rng, s_rng, depths)]
        return {"T": np.array([g[0].reshape(16) for g in got]), "objective": np.array([g[2] for g in got]),
                "status": None}
    if kind == "forward":
        return _forward64(_dev(_weights()).double(), _network_rows(case["batch"], seed)[0])
    if kind == "train":
        return _train64(case, seed)
    return _propose64(*_so3_clouds(case, seed))
