"""Kernels whose launch shape follows the number of frames or poses in a call
(generation teams, LM clusters, ICP clusters): a frame's or pose's result is
the same bits in a call of one and in calls on every side of the rules, and
the call of one matches the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from synth import rooms, workloads
from tests import helpers as H

pytestmark = pytest.mark.gpu

FIELDS = ("pose", "energy", "score", "n_hypotheses", "n_chosen", "n_pixels", "best", "chosen_pose", "chosen_energy",
          "chosen_score", "chosen_slot", "chosen_icp_frac", "icp_mask")


@pytest.fixture(scope="module")
def rg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    rg.lib()
    return rg


@pytest.fixture(scope="module")
def model(rg):
    """A forest whose pixels have up to 5 x 40 modes, and 40 query frames."""
    w = workloads.small_case(n_trees=5, depth=6, n_train=10)
    w = dataclasses.replace(w, forest=dict(w.forest, m_max=40, kappa=300, min_cluster_size=2, tau_c=0.1))
    ctx = rg.Context(0, arena_bytes=3 << 30)
    f = H.gpu_model(ctx, w)
    scene = rg.Scene(ctx, w.room().lo, w.room().hi)
    nodes = H.oracle_forest_nodes(w)
    res = oracle.Reservoirs(nodes, w.forest["kappa"], w.forest_seed)
    for d, c, T in w.training_frames():
        res.add_frame(d, c, w.K, T)
    modes = oracle.Modes(res.n_leaves, w.forest["m_max"])
    fp = w.forest
    oracle.update_modes(res, modes, fp["sigma"], fp["tau_c"], fp["min_cluster_size"], cov_eps=fp["cov_eps"],
                        fp16_offsets=bool(fp["mode_precision"]))
    return w, f, scene, nodes, modes, w.queries(40)


# rows of 50 modes (LM clusters with sets of hypotheses), 10 (one set), 200 (LM parts); 40 exceeds every rule's bound
PARAMS = {
    "50 modes": dict(k_top=10),
    "50 modes, redraw, icp": dict(k_top=10, redraw=1, **workloads.ICP_ON),
    "10 modes": dict(k_top=10, n_trees_used=1),
    "200 modes": dict(k_top=40),
    "200 modes, Euclidean": dict(k_top=40, use_cov=0),
    "few slots": dict(k_top=10, n_hyp=20, n_cull=20),
}


@pytest.mark.parametrize("name", list(PARAMS))
def test_results_do_not_depend_on_the_frames_in_the_call(rg, model, name):
    w, f, scene, nodes, modes, queries = model
    p = dict(w.ransac, n_trees_used=5, n_cull=64, n_hyp=200, max_iter=500)
    p.update(PARAMS[name])
    rel = rg.Relocaliser(f, scene, p, w.width, w.height, len(queries))
    depth = np.stack([q[0] for q in queries])
    rgb = np.stack([q[1] for q in queries])
    seeds = [q[3] for q in queries]
    alone = rel.relocalise_batch(depth[:1], rgb[:1], w.K, seeds[:1])[0]
    assert alone["n_hypotheses"] > 1
    lv = oracle.forest_leaves(nodes, queries[0][0], queries[0][1], w.K.fx, n_trees=p["n_trees_used"])
    run = H.OracleRun(p, queries[0][0], queries[0][1], w.K, lv, modes, w.room().lo, w.room().hi, seeds[0],
                      1 << w.forest["depth"])
    H.compare_results(rg, alone, rel.debug(0), run, dict(oracle.PARAM_DEFAULTS, **p), name)
    for n in (2, 4, 5, 8, 9, 10, 16, 17, 20, 33, 39, 40):
        got = rel.relocalise_batch(depth[:n], rgb[:n], w.K, seeds[:n])
        for k in FIELDS:
            np.testing.assert_array_equal(got[0][k], alone[k], err_msg=f"{name}: {k} of frame 0 among {n}")
        if n == 2:
            second = got[1]
        for k in FIELDS:
            np.testing.assert_array_equal(got[1][k], second[k], err_msg=f"{name}: {k} of frame 1 among {n}")
    rel.close()


@pytest.mark.parametrize("size", [(101, 67), (160, 120), (7, 5)])
def test_icp_does_not_depend_on_the_poses_in_the_call(rg, size):
    room = rooms.Room((4.0, 3.0, 2.5), 5)
    K = rooms.Intrinsics(0.9 * size[0], 0.9 * size[0], size[0] / 2, size[1] / 2, *size)
    truth = rooms.query_poses(room, 1, seed=77)[0]
    d, _ = rooms.render(room, K, truth, noise_seed=3)
    d = rooms.mask_depth(d, 0.15, 4)
    rng = np.random.default_rng(8)
    poses = np.repeat(truth[None], 160, 0)
    poses[:, :3, 3] += rng.uniform(-0.04, 0.04, (160, 3))
    poses[5, :3, 3] = [9.0, 1.0, 1.0]  # outside the box
    ctx = rg.Context(0, arena_bytes=64 << 20)
    scene = rg.Scene(ctx, room.lo, room.hi)
    # 160 poses: a block each; 58 to 152: clusters of four; fewer: of eight
    whole = scene.icp_poses(d, K, poses)
    for n in (1, 20, 57, 58, 100, 152, 153):
        part = scene.icp_poses(d, K, poses[:n])
        for a, b in zip(part, whole):
            np.testing.assert_array_equal(a, b[:n], err_msg=f"{n} poses")
    for i in range(3):
        P, ok, frac = oracle.icp_refine(poses[i], d, K, room.lo, room.hi)
        H.check_icp_one(whole[1][i], whole[2][i], whole[0][i], ok, frac, P, 0.5, f"pose {i}")
    scene.close()
    ctx.close()


@pytest.mark.parametrize("inside,outside", [(1, 0), (3, 0), (4, 0), (17, 0), (3, 1), (15, 1), (16, 17), (1, 32)])
def test_scores_do_not_depend_on_the_poses_beside(rg, inside, outside):
    """Groups of four poses are reduced together while all of a chunk are
    inside the box: a pose's score has the same bits alone, and the inside
    poses' match the FP64 oracle (FP32 rays: 1e-4 relative)."""
    w = workloads.small_case(n_trees=1, depth=3, n_train=1)
    room, rng = w.room(), np.random.default_rng(inside * 64 + outside)
    depth, _ = rooms.render(room, w.K, rooms.look_pose([2.0, 1.4, 1.3], 2.0, -0.1), noise_seed=2)
    depth = rooms.mask_depth(depth, 0.25, seed=9)
    lo, hi = np.asarray(room.lo, np.float64), np.asarray(room.hi, np.float64)
    poses = []
    for k in range(inside + outside):
        at = lo + (hi - lo) * rng.uniform(0.2, 0.8, 3)
        if k >= inside:
            at[k % 3] = lo[k % 3] - rng.uniform(0.1, 1.0)
        poses.append(rooms.look_pose(at, rng.uniform(-3, 3), rng.uniform(-0.3, 0.3)))
    poses = np.stack(poses)[rng.permutation(inside + outside)]
    ctx = rg.Context(0, arena_bytes=1 << 26)
    scene = rg.Scene(ctx, lo, hi)
    s, f = scene.score_poses(depth, w.K, poses)
    for i, P in enumerate(poses):
        s1, f1 = scene.score_poses(depth, w.K, poses[i:i + 1])
        assert s[i] == s1[0] and f[i] == f1[0], i
        o_s, _, _ = oracle.depth_score(P, depth, w.K, room.lo, room.hi)
        if np.all(P[:3, 3] > lo) and np.all(P[:3, 3] < hi):
            assert abs(s[i] - o_s) <= 1e-4 * o_s, (i, s[i], o_s)
    scene.close()
    ctx.close()
