"""The work that a user of this library has it do, as cases that can be timed.

Each case is one kind of call at one size, through the Python layer:

  relocalise  Relocaliser.relocalise_batch on device frames: a lost camera (one
              frame), or a batch of queries;
  cascade     Cascade.relocalise_batch, three levels;
  serve       Server: requests from several cameras of two resolutions, submitted
              as host frames and waited for;
  score       Scene.score_poses: given poses ranked against a live depth frame;
  icp         Scene.icp_poses: given poses refined against a live depth frame;
  train       a forest adapted to a room from posed frames, all leaves clustered,
              its modes read back;
  track       the online loop from empty leaves: posed frames adapted one by one
              with a budget of leaves re-clustered per frame, then a lost frame
              relocalised.

Inputs are rendered on the GPU from the seed: an axis-aligned box room tiled
with 8 cm cells of random colour, a training trajectory round the room, query
poses near it, 2 mm depth noise.  Forest and relocaliser sizes are those of the
library's workloads and presets.
"""
import math

import numpy as np
import torch

import paper_1810_12163_gb300 as rg

ROOMS = ((4.0, 3.0, 2.5), (6.0, 5.0, 3.0), (10.0, 8.0, 3.0))
CELL = 0.08    # metres, side of a texture cell
SIGMA = 0.002  # metres, depth noise

# the relocaliser of the library's 640x480 workload: halving to one pose
PAPER = dict(rg.presets.DEFAULT, eta=500, halve_to_one=1)
PRESETS = {"default": rg.presets.DEFAULT, "paper": PAPER, "fast": rg.presets.FAST,
           "intermediate": rg.presets.INTERMEDIATE, "slow": rg.presets.SLOW}
# the three-level cascade: input subsampling and parameters of each level
LEVELS = ((4, dict(PAPER, n_hyp=64, n_trees_used=1, k_out=1, eta=100, halve_to_one=0)),
          (2, dict(PAPER, n_hyp=256, k_out=1, eta=250, halve_to_one=0)),
          (1, dict(PAPER, halve_to_one=0)))
THRESHOLDS = (0.071, 0.085)


def _forest(trees=5, depth=15, kappa=1024, m_max=50, min_size=20, tau_c=0.05, fp16=True, frames=160):
    return dict(trees=trees, depth=depth, kappa=kappa, m_max=m_max, min_size=min_size, tau_c=tau_c, fp16=fp16,
                frames=frames)


def _size(width, height, room=0, missing=0.0):
    return dict(width=width, height=height, room=room, missing=missing)


SMALL = _forest(trees=1, depth=10, kappa=256, m_max=10, min_size=5, frames=20)
FAST_FOREST = _forest(depth=13, kappa=2048, min_size=5, tau_c=0.2, frames=60)


def _reloc(preset, batch, n_hyp=0, eta=0, k_top=10, trees_used=0, icp=False, redraw=False, loose=False):
    """0: the preset's value (trees_used: every tree); loose: checks that most triples pass, as the library's small
    workload has them."""
    return dict(preset=preset, batch=batch, n_hyp=n_hyp, eta=eta, k_top=k_top, trees_used=trees_used, icp=icp,
                redraw=redraw, loose=loose)


def listed():
    return [
        # a low-resolution camera that lost track: the smallest call, latency
        dict(name="frame 160x120", kind="relocalise", **_size(160, 120), **SMALL,
             **_reloc("default", 1, n_hyp=64, eta=100, loose=True)),
        # one 640x480 frame, as a tracker asks when it is lost: latency
        dict(name="frame 640x480", kind="relocalise", **_size(640, 480), **_forest(), **_reloc("paper", 1)),
        # a batch of queries, the throughput workload
        dict(name="batch 64x640x480", kind="relocalise", **_size(640, 480), **_forest(), **_reloc("paper", 64)),
        # the Fast preset (no refinement, Euclidean energies) on a ragged size with holes in the depth
        dict(name="fast 6x333x250", kind="relocalise", **_size(333, 250, missing=0.1), **FAST_FOREST,
             **_reloc("fast", 6, redraw=True)),
        # every stored mode of a leaf used, four times the hypotheses, FP32 modes
        dict(name="all modes 4x640x480", kind="relocalise", **_size(640, 480), **_forest(fp16=False),
             **_reloc("paper", 4, n_hyp=4096, k_top=50)),
        # ICP of the chosen poses before ranking
        dict(name="with icp 8x640x480", kind="relocalise", **_size(640, 480), **_forest(),
             **_reloc("default", 8, icp=True)),
        # the cascade on a full server batch
        dict(name="cascade 16x640x480", kind="cascade", **_size(640, 480), **_forest(), batch=16),
        # requests of eight cameras, two resolutions, through the serving loop
        dict(name="serve 24", kind="serve", **_size(640, 480), **_forest(), batch=24, max_batch=16),
        # candidate poses of a pose graph scored against a live frame
        dict(name="score 128 poses", kind="score", **_size(640, 480), poses=128),
        # the last candidates of a RANSAC of one's own refined by ICP
        dict(name="icp 16 poses", kind="icp", **_size(640, 480), poses=16),
        # a forest adapted to a room and clustered whole
        dict(name="train 24 frames", kind="train", **_size(640, 480, room=1),
             **_forest(depth=11, m_max=10, frames=24)),
        # a room mapped online, then a lost frame
        dict(name="track 16 frames", kind="track", **_size(640, 480), **_forest(depth=12, min_size=5, frames=16),
             **_reloc("default", 1), budget=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _frame_size(rng, most=640):
    w = _log(rng, 96, most)
    return _size(w, max(64, int(w * rng.uniform(0.55, 0.8))), room=rng.randrange(3),
                 missing=rng.choice([0.0, 0.0, round(rng.uniform(0.02, 0.4), 3)]))


def draw(rng):
    kind = rng.choice(["relocalise"] * 6 + ["cascade", "cascade", "serve", "score", "icp", "train", "track"])
    size = _frame_size(rng)
    pixels = size["width"] * size["height"]
    if kind in ("score", "icp"):
        return dict(kind=kind, **size, poses=_log(rng, 1, 128 if kind == "score" else 48))
    if kind == "train":
        return dict(kind=kind, **size, **_forest(trees=rng.randint(1, 5), depth=rng.randint(7, 11),
                                                 kappa=_log(rng, 100, 1024), m_max=rng.randint(4, 12),
                                                 min_size=rng.randint(2, 12), tau_c=round(rng.uniform(0.05, 0.2), 3),
                                                 fp16=rng.random() < 0.7, frames=rng.randint(4, 24)))
    # frames to train on, and leaves that hold 25 to 80 of their grid pixels each: fewer leave no modes
    frames = rng.randint(30, 80)
    depth = int(round(math.log2(frames * pixels / 16 / rng.uniform(25, 80))))
    forest = _forest(trees=rng.randint(1, 5), depth=min(15, max(8, depth)), kappa=_log(rng, 256, 1024),
                     m_max=rng.randint(8, 50), min_size=rng.randint(3, 6), tau_c=round(rng.uniform(0.08, 0.2), 3),
                     fp16=rng.random() < 0.7, frames=frames)
    if kind == "cascade":
        return dict(kind=kind, **size, **forest, batch=_log(rng, 1, max(1, min(64, 24 * 307200 // pixels))))
    if kind == "serve":
        return dict(kind=kind, **size, **forest, batch=_log(rng, 2, 32), max_batch=rng.randint(2, 16))
    if kind == "track":
        forest.update(frames=min(frames, 32), depth=max(7, min(13, depth - 1)))
        return dict(kind=kind, **size, **forest, **_reloc("default", 1, n_hyp=_log(rng, 128, 1024), loose=True),
                    budget=_log(rng, 256, 4096))
    wide = rng.random() < 0.2  # most or all stored modes used
    batch = _log(rng, 1, max(1, min(64, (2 if wide else 32) * 307200 // pixels)))
    preset = rng.choice(["default", "paper", "paper", "fast", "intermediate", "slow"])
    trees = rng.randint(1, forest["trees"])
    # few generation iterations or few modes: only the loose checks find triples
    few = preset in ("fast", "intermediate", "slow") or trees < 3
    return dict(kind=kind, **size, **forest, **_reloc(
        preset, batch, n_hyp=_log(rng, 192, 2048), eta=_log(rng, 48, 512),
        k_top=rng.randint(16, 50) if wide else rng.randint(5, 11), trees_used=trees, icp=rng.random() < 0.15,
        redraw=rng.random() < 0.2, loose=few or rng.random() < 0.5))


# ---- inputs ---------------------------------------------------------------
def _K(width, height):
    s = width / 640.0
    return rg.Intrinsics(585.0 * s, 585.0 * s, 320.0 * s, 240.0 * s, width, height)


class _Room:
    """A textured box room rendered on the GPU."""

    def __init__(self, size, seed):
        self.size = size
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        X, Y, Z = size
        self.cells = [(math.ceil(a / CELL) + 1, math.ceil(b / CELL) + 1) for a, b in
                      ((Y, Z), (Y, Z), (X, Z), (X, Z), (X, Y), (X, Y))]  # x = 0, x = X, y = 0, ...
        n = [a * b for a, b in self.cells]
        self.base = torch.tensor(np.concatenate([[0], np.cumsum(n)[:-1]]), device="cuda")
        self.width = torch.tensor([b for _, b in self.cells], device="cuda")
        self.rows = torch.tensor([a for a, _ in self.cells], device="cuda")
        self.texture = torch.randint(0, 256, (sum(n), 3), dtype=torch.uint8, device="cuda", generator=self.gen)

    def render(self, K, poses, missing=0.0):
        """(depth [n][H][W] float32 metres, colour [n][H][W][3] uint8) at camera->world poses [n][4][4]."""
        depths, colours = [], []
        for k in range(0, len(poses), 32):
            P = torch.tensor(np.asarray(poses[k:k + 32]), device="cuda", dtype=torch.float32)
            u = torch.arange(K.width, device="cuda", dtype=torch.float32)
            v = torch.arange(K.height, device="cuda", dtype=torch.float32)
            c = torch.stack([((u - K.cx) / K.fx)[None, :].expand(K.height, -1),
                             ((v - K.cy) / K.fy)[:, None].expand(-1, K.width),
                             torch.ones(K.height, K.width, device="cuda")], -1)
            d = torch.einsum("nrc,hwc->nhwr", P[:, :3, :3], c)
            o = P[:, None, None, :3, 3]
            hi = torch.tensor(self.size, device="cuda", dtype=torch.float32)
            t = torch.where(d > 0, (hi - o) / d, torch.where(d < 0, -o / d, torch.inf))
            z, axis = t.min(-1)
            p = o + z[..., None] * d
            side = d.gather(-1, axis[..., None])[..., 0] > 0
            face = axis * 2 + side
            other = torch.tensor([[1, 2], [0, 2], [0, 1]], device="cuda")[axis]
            cell = (p.gather(-1, other) / CELL).long().clamp_(min=0)
            row, col = cell[..., 0].minimum(self.rows[face] - 1), cell[..., 1].minimum(self.width[face] - 1)
            colours.append(self.texture[self.base[face] + row * self.width[face] + col])
            z = z + SIGMA * torch.randn(z.shape, device="cuda", generator=self.gen)
            if missing > 0:
                z = torch.where(torch.rand(z.shape, device="cuda", generator=self.gen) < missing, 0.0, z)
            depths.append(z.clamp_(min=0))
        return torch.cat(depths), torch.cat(colours)


def _look(position, yaw, pitch):
    """Camera->world pose looking along (yaw, pitch), world z up, camera x right, y down, z forward."""
    f = np.array([math.cos(pitch) * math.cos(yaw), math.cos(pitch) * math.sin(yaw), math.sin(pitch)])
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    T = np.eye(4)
    T[:3, :3] = np.stack([r, np.cross(f, r), f], axis=1)
    T[:3, 3] = position
    return T


def _trajectory(size, n, rng):
    """Once round the room on an ellipse, looking outwards, pitch swaying."""
    out = []
    for i in range(n):
        a = 2 * math.pi * i / n
        c = np.array([size[0] / 2 + 0.3 * size[0] * math.cos(a), size[1] / 2 + 0.3 * size[1] * math.sin(a),
                      min(1.5, 0.6 * size[2])])
        out.append(_look(c + rng.uniform(-0.02, 0.02, 3), a + math.radians(rng.uniform(-2, 2)),
                         math.radians(10.0 * math.sin(3 * a) + rng.uniform(-2, 2))))
    return out


def _turn(axis, angle):
    a = np.asarray(axis) / np.linalg.norm(axis)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    return np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * (K @ K)


def _near(poses, size, rng, trans, degrees):
    """Each pose moved by at most `trans` and turned by at most `degrees`, inside the room."""
    out = []
    for P in poses:
        T = P.copy()
        v = rng.normal(size=3)
        v *= trans * rng.uniform() ** (1 / 3) / np.linalg.norm(v)
        T[:3, 3] = np.clip(T[:3, 3] + v, 0.5, np.asarray(size) - 0.5)
        T[:3, :3] = _turn(rng.normal(size=3), math.radians(degrees) * rng.uniform()) @ T[:3, :3]
        out.append(T)
    return out


def _queries(case, n, rng):
    size = ROOMS[case["room"]]
    along = _trajectory(size, 360, rng)
    return _near([along[int(rng.integers(360))] for _ in range(n)], size, rng, 0.3, 20.0)


class _State:
    """What a program keeps between calls; gives the library's handles back when dropped."""

    def __init__(self, case, seed, arena):
        self.case = case
        self.rng = np.random.default_rng(seed)
        self.room = _Room(ROOMS[case["room"]], seed)
        self.K = _K(case["width"], case["height"])
        self.ctx = rg.Context(0, arena_bytes=arena)
        self.handles = []

    def keep(self, handle):
        self.handles.append(handle)
        return handle

    def __del__(self):
        for h in reversed(getattr(self, "handles", [])):
            h.close()
        if hasattr(self, "ctx"):
            self.ctx.close()


def _relocaliser_params(case):
    p = dict(PRESETS[case["preset"]], k_top=case["k_top"], icp=int(case["icp"]), redraw=int(case["redraw"]),
             n_trees_used=case["trees_used"] or case["trees"])
    p["n_hyp"] = case["n_hyp"] or p["n_hyp"]
    p["eta"] = case["eta"] or p["eta"]
    if case["loose"]:
        p.update(colour_thresh=120, max_trans_err=0.15, min_sq_dist=0.04)
    return p


def _frame_bytes(case, p, n):
    """Device memory of a relocaliser of n frames (an upper estimate)."""
    pixels = case["width"] * case["height"]
    modes = p["n_trees_used"] * min(p["k_top"], case["m_max"]) + 1
    drawn = 8 * p["eta"] + 16
    parts = drawn / max(1, min(32, 40960 // (36 * modes))) + 1
    return int(n * (pixels * (2 * p["n_trees_used"] + 40) + drawn * (modes * 36 + 64 * 20 + 64) +
                    p["n_hyp"] * (120 + 4 * parts) + (1 << 20)))


def _forest_bytes(case):
    return (case["trees"] << case["depth"]) * (case["kappa"] * 16 + case["m_max"] * 120 + 128) + (64 << 20)


def _random_forest(s):
    c = s.case
    return s.keep(rg.Forest.random(s.ctx, dict(
        n_trees=c["trees"], depth=c["depth"], kappa=c["kappa"], m_max=c["m_max"], min_cluster_size=c["min_size"],
        tau_c=c["tau_c"], mode_precision=int(c["fp16"])), int(s.rng.integers(1 << 40))))


def _trained(s):
    """The case's forest, adapted to the room from posed frames, every leaf clustered."""
    c, f = s.case, _random_forest(s)
    poses = _trajectory(s.room.size, c["frames"], s.rng)
    for k in range(0, len(poses), 32):
        depth, rgb = s.room.render(s.K, poses[k:k + 32], c["missing"])
        for d, r, T in zip(depth, rgb, poses[k:k + 32]):
            f.adapt(d, r, s.K, T)
    f.update_modes(-1)
    return f


def prepare(case, seed):
    kind, n = case["kind"], case.get("batch", 1)
    if kind in ("score", "icp"):
        s = _State(case, seed, 256 << 20)
        s.scene = s.keep(rg.Scene(s.ctx, np.zeros(3), s.room.size))
        truth = _queries(case, 1, s.rng)
        s.depth = s.room.render(s.K, truth, case["missing"])[0][0]
        wide = kind == "score"
        s.poses = np.stack(_near(truth * case["poses"], s.room.size, s.rng, 0.5 if wide else 0.06, 20.0 if wide else 3.0))
        return s
    if kind == "train":
        s = _State(case, seed, _forest_bytes(case) + (256 << 20))
        s.forest = _random_forest(s)
        s.poses = _trajectory(s.room.size, case["frames"], s.rng)
        s.depth, s.rgb = s.room.render(s.K, s.poses, case["missing"])
        return s
    room_for = [p for _, p in LEVELS] if kind in ("cascade", "serve") else [_relocaliser_params(case)]
    slots = 2 * case["max_batch"] if kind == "serve" else n
    room_for = [dict(p, n_trees_used=min(p["n_trees_used"], case["trees"])) for p in room_for]
    s = _State(case, seed, int(1.1 * (_forest_bytes(case) + sum(_frame_bytes(case, p, slots) for p in room_for))) +
               (256 << 20))
    if kind == "track":
        s.forest = _random_forest(s)
        s.forest.set_streaming(True)
    else:
        s.forest = _trained(s)
    s.scene = s.keep(rg.Scene(s.ctx, np.zeros(3), s.room.size))
    s.seeds = [int(x) for x in s.rng.integers(1 << 40, size=n)]
    W, H = case["width"], case["height"]
    if kind == "cascade":
        levels = [s.keep(rg.Relocaliser(s.forest, s.scene, p, (W + f - 1) // f, (H + f - 1) // f, n))
                  for (f, _), p in zip(LEVELS, room_for)]
        s.reloc = s.keep(rg.Cascade(levels, THRESHOLDS, [f for f, _ in LEVELS]))
    elif kind == "serve":
        s.server = s.keep(rg.Server(s.ctx, max_batch=case["max_batch"]))
        s.model = s.server.add_cascade_model(s.forest, s.scene, room_for, [f for f, _ in LEVELS], THRESHOLDS, W, H)
        poses = _queries(case, n, s.rng)
        half = _K(W // 2, H // 2)  # every other camera has half the resolution
        s.requests = []
        for i, T in enumerate(poses):
            K = s.K if i % 2 == 0 else half
            depth, rgb = s.room.render(K, [T], case["missing"])
            s.requests.append((depth[0].cpu().numpy(), rgb[0].cpu().numpy(), K, s.seeds[i]))
        return s
    else:
        s.reloc = s.keep(rg.Relocaliser(s.forest, s.scene, room_for[0], W, H, n))
    if kind == "track":
        s.poses = _trajectory(s.room.size, case["frames"], s.rng)
        s.tracked = s.room.render(s.K, s.poses, case["missing"])
        lost = _near([s.poses[case["frames"] // 2]], s.room.size, s.rng, 0.2, 10.0)
    else:
        lost = _queries(case, n, s.rng)
    s.depth, s.rgb = s.room.render(s.K, lost, case["missing"])
    return s


# ---- the calls --------------------------------------------------------------
def _gather(results):
    """The results of a call's frames, field by field; chosen poses and their figures are zero from n_chosen on.
    Energies, scores and inlier fractions are 32-bit values."""
    out = {k: np.array([r[k] for r in results]) for k in
           ("pose", "level", "n_hypotheses", "n_chosen", "n_pixels", "status", "best", "icp_mask")}
    for k in ("energy", "energy_per_pixel", "score"):
        out[k] = np.array([r[k] for r in results], np.float32)
    for k, shape, dtype in (("chosen_pose", (16, 4, 4), np.float64), ("chosen_energy", (16,), np.float32),
                            ("chosen_score", (16,), np.float32), ("chosen_slot", (16,), np.int32),
                            ("chosen_icp_frac", (16,), np.float32)):
        out[k] = np.zeros((len(results),) + shape, dtype)
        for row, r in zip(out[k], results):
            if len(r[k]):
                row[:len(r[k])] = r[k]
    return out


def run(state):
    kind = state.case["kind"]
    if kind == "score":
        return state.scene.score_poses(state.depth, state.K, state.poses)
    if kind == "icp":
        return state.scene.icp_poses(state.depth, state.K, state.poses)
    if kind == "serve":
        tickets = [state.server.submit(state.model, *r) for r in state.requests]
        return _gather([state.server.wait(t) for t in tickets])
    if kind == "train":
        f = state.forest
        f.reset_leaves()
        for d, r, T in zip(state.depth, state.rgb, state.poses):
            f.adapt(d, r, state.K, T)
        f.update_modes(-1)
        e = f.export()
        return {k: e[k] for k in ("res_count", "nmodes", "mode_pos", "mode_rgb", "mode_U", "mode_size")}
    if kind == "track":
        state.forest.reset_leaves()
        for d, r, T in zip(*state.tracked, state.poses):
            state.forest.adapt(d, r, state.K, T)
            state.forest.update_modes(state.case["budget"])
    return _gather(state.reloc.relocalise_batch(state.depth, state.rgb, state.K, state.seeds))


# ---- what a pass cannot do without ------------------------------------------
# flops of one unit of each step, as the method states it
NODE, RAY, ICP_PIXEL, MODE, GENERATION = 8, 20, 50, 18, 12


def _relocalise_flops(p, trees, depth, m_max, pixels):
    """One frame: every pixel down every tree, the hypotheses' first accepted triples, the energies of the cull,
    one refinement pass per preemptive round, the chosen poses' depth images."""
    modes = trees * min(p["k_top"], m_max) / 2
    total = pixels * trees * depth * NODE + p["n_hyp"] * p["max_iter"] * GENERATION
    total += p["n_hyp"] / 10 * p["eta"] * modes * MODE
    n, drawn = p["n_cull"], p["eta"]
    while n > (1 if p["halve_to_one"] else p["k_out"]):
        drawn += p["eta"]
        total += n * drawn * modes * MODE * (3 if p["pose_update"] else 1)
        n = (n + 1) // 2
    return total + p["k_out"] * pixels * RAY * p["rank"]


def _relocalise_work(case, p, n, pixels):
    trees = min(p["n_trees_used"], case["trees"])
    nodes = trees * (2 << case["depth"]) * 8
    return (n * (pixels * 7 + 2800) + nodes,
            n * _relocalise_flops(p, trees, case["depth"], case["m_max"], pixels))


def work(case):
    kind, n = case["kind"], case.get("batch", 1)
    pixels = case["width"] * case["height"]
    if kind == "score":
        return {"bytes": pixels * 4 + case["poses"] * 136, "flops": case["poses"] * pixels * RAY}
    if kind == "icp":  # strides 4, 2, 1 for 6, 3, 2 iterations
        return {"bytes": pixels * 4 + case["poses"] * 264,
                "flops": case["poses"] * pixels * (6 / 16 + 3 / 4 + 2) * ICP_PIXEL}
    if kind in ("train", "track"):
        frames, grid = case["frames"], (pixels + 15) // 16
        leaves = case["trees"] << case["depth"]
        done = leaves if kind == "train" else case["budget"] * frames
        seen = frames if kind == "train" else frames / 2
        points = min(case["kappa"], seen * grid * case["trees"] / leaves)  # in a mean leaf
        byte = frames * grid * 7 + done * (points * 16 + case["m_max"] * 43)
        flops = frames * grid * case["trees"] * case["depth"] * NODE + done * points * points * 20
        if kind == "track":
            b, f = _relocalise_work(case, _relocaliser_params(case), 1, pixels)
            byte, flops = byte + b, flops + f
        return {"bytes": byte, "flops": flops}
    if kind == "relocalise":
        b, f = _relocalise_work(case, _relocaliser_params(case), n, pixels)
        return {"bytes": b, "flops": f}
    # cascade, serve: nine in ten frames end at the first level, one in ten at the second
    full = n if kind == "cascade" else (n + 1) // 2 + n // 2 / 4
    byte, flops = n * 2800 + full * pixels * 7, 0
    for (s, p), share in zip(LEVELS, (1.0, 0.1, 0.03)):
        flops += share * full * _relocalise_flops(p, min(p["n_trees_used"], case["trees"]), case["depth"],
                                                  case["m_max"], pixels / (s * s))
    return {"bytes": byte, "flops": flops}


# ---- the same results in 64 bits ----------------------------------------------
def _rays(K):
    u = (torch.arange(K.width, device="cuda", dtype=torch.float64) - K.cx) / K.fx
    v = (torch.arange(K.height, device="cuda", dtype=torch.float64) - K.cy) / K.fy
    return torch.stack([u[None, :].expand(K.height, -1), v[:, None].expand(-1, K.width),
                        torch.ones(K.height, K.width, device="cuda", dtype=torch.float64)], -1)


def _exit(d, o, hi):
    """(depth, axis) of the face where rays d from o inside [0, hi] leave the box."""
    t = torch.where(d > 0, (hi - o) / d, torch.where(d < 0, -o / d, torch.inf))
    return t.min(-1)


def _exact_icp(depth, rays, hi, T):
    """Point-to-plane Gauss-Newton with projective association and a relative ridge, coarse to fine."""
    H = torch.tensor(T, device="cuda")
    frac, ok = 0.0, True
    for stride, iters, dist in zip((4, 2, 1), (6, 3, 2), (0.1, 0.05, 0.025)):
        z, c = depth[::stride, ::stride].reshape(-1), rays[::stride, ::stride].reshape(-1, 3)
        c, z = c[z > 0], z[z > 0]
        for _ in range(iters):
            d = c @ H[:3, :3].T
            s, axis = _exit(d, H[:3, 3], hi)
            gap = z - s
            near = gap.abs() * d.norm(dim=-1) <= dist
            frac = float(near.double().mean())
            x = c[near] * z[near, None]
            m = H[:3, :3][axis[near]]  # the face normal in the camera frame
            J = torch.cat([m, torch.linalg.cross(x, m)], -1)
            r = gap[near] * d[near].gather(-1, axis[near][:, None])[:, 0]
            A = J.T @ J
            A = A + 1e-4 * A.trace() / 6 * torch.eye(6, device="cuda", dtype=torch.float64)
            xi = torch.linalg.solve(A, -(J.T @ r)).cpu().numpy()
            X = np.zeros((4, 4))
            X[:3, :3] = [[0, -xi[5], xi[4]], [xi[5], 0, -xi[3]], [-xi[4], xi[3], 0]]
            X[:3, 3] = xi[:3]
            H = H @ torch.linalg.matrix_exp(torch.tensor(X, device="cuda"))
    return (H.cpu().numpy() if frac >= 0.5 else T), frac


def exact(case, seed):
    """The scores and the refined poses are formulas of the inputs; what the other calls return hangs on choices
    (leaves, triples, inliers) that no short program repeats."""
    if case["kind"] not in ("score", "icp"):
        return None
    s = prepare(case, seed)
    rays, depth = _rays(s.K), s.depth.double()
    hi = torch.tensor(s.room.size, device="cuda", dtype=torch.float64)
    if case["kind"] == "icp":
        poses, frac = zip(*[_exact_icp(depth, rays, hi, T) for T in s.poses])
        return np.stack(poses), None, np.array(frac)
    scores = []
    for T in s.poses:
        P = torch.tensor(T, device="cuda")
        z, _ = _exit(rays @ P[:3, :3].T, P[:3, 3], hi)
        valid = depth > 0
        scores.append(float((depth - z).abs()[valid].mean()))
    return np.array(scores), np.ones(len(scores))
