"""Reservoirs and modes (Sec. 3.2.2) at the sizes where the adaptation and
clustering kernels split their work differently: leaves of a few points to
full ones, capacities that are odd or above a block's threads, leaves that
overflow within one frame, every leaf in one tree; against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from synth import rooms, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    rg.lib()
    return rg


CASES = {
    # depth 1: two leaves a tree; 1200 points of 96x72 frames every pixel fill them in the first frame
    "two leaves, capacity 1": dict(trees=1, depth=1, kappa=1, m_max=1, size=(64, 48), step=2, frames=2, min_size=1),
    "few leaves, odd capacity": dict(trees=2, depth=2, kappa=77, m_max=8, size=(96, 72), step=2, frames=3, min_size=3),
    "a block's threads": dict(trees=1, depth=1, kappa=512, m_max=16, size=(96, 72), step=2, frames=3, min_size=4),
    "one more": dict(trees=1, depth=1, kappa=513, m_max=16, size=(96, 72), step=2, frames=3, min_size=4),
    "two rows a thread": dict(trees=1, depth=1, kappa=1025, m_max=64, size=(101, 67), step=1, frames=2, min_size=2),
    "largest capacity": dict(trees=1, depth=1, kappa=4096, m_max=64, size=(160, 120), step=1, frames=1, min_size=5),
    "leaves of every size": dict(trees=3, depth=7, kappa=200, m_max=10, size=(160, 120), step=2, frames=6, min_size=1),
    "more pixels than a table's": dict(trees=2, depth=2, kappa=50, m_max=4, size=(480, 360), step=1, frames=2,
                                       min_size=2),
    "repeated frames": dict(trees=2, depth=3, kappa=300, m_max=12, size=(96, 72), step=3, frames=4, min_size=3,
                            repeat=True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_reservoirs_and_modes_match_the_oracle(rg, name):
    c = CASES[name]
    fp = dict(workloads.FOREST_DEFAULT, n_trees=c["trees"], depth=c["depth"], kappa=c["kappa"], m_max=c["m_max"],
              min_cluster_size=c["min_size"], tau_c=0.15, grid_step=c["step"])
    seed = 21
    ctx = rg.Context(0, arena_bytes=1 << 28)
    g = rg.Forest.random(ctx, fp, seed)
    o = oracle.forest_random(fp["n_trees"], fp["depth"], fp["p_depth"], (fp["delta_lo"], fp["delta_hi"]),
                             (fp["tau_depth_lo"], fp["tau_depth_hi"]), (fp["tau_rgb_lo"], fp["tau_rgb_hi"]),
                             bool(fp["tau_zero"]), seed)
    res = oracle.Reservoirs(o, fp["kappa"], seed)
    room = rooms.Room((4.0, 3.0, 2.5), 5)
    K = dataclasses.replace(rooms.intrinsics_for(640, 480), width=c["size"][0], height=c["size"][1], fx=120.0, fy=120.0,
                            cx=c["size"][0] / 2, cy=c["size"][1] / 2)
    for i, T in enumerate(rooms.training_trajectory(room, c["frames"])):
        if c.get("repeat"):  # equal points, so equal densities: ties go to the lower index
            i, T = 0, rooms.training_trajectory(room, c["frames"])[0]
        d, rgb = rooms.render(room, K, T, noise_seed=40 + i)
        d = rooms.mask_depth(d, 0.1, 60 + i)
        g.adapt(d, rgb, K, T)
        res.add_frame(d, rgb, K, T, fp["grid_step"], 0)
    g.update_modes(-1)
    modes = oracle.Modes(res.n_leaves, fp["m_max"])
    oracle.update_modes(res, modes, fp["sigma"], fp["tau_c"], fp["min_cluster_size"], cov_eps=fp["cov_eps"],
                        fp16_offsets=True)
    e = g.export(reservoirs=True)
    np.testing.assert_array_equal(e["res_count"], res.count)
    held = np.arange(fp["kappa"])[None, :] < res.count[:, None]
    np.testing.assert_array_equal(e["res_pos"][held], res.pos.reshape(-1, fp["kappa"], 3)[held])
    np.testing.assert_array_equal(e["res_rgb"][held], res.rgb.reshape(-1, fp["kappa"], 3)[held])
    np.testing.assert_array_equal(e["nmodes"], modes.nmodes)
    np.testing.assert_array_equal(e["mode_size"], modes.size.reshape(e["mode_size"].shape))
    np.testing.assert_array_equal(e["mode_rgb"], modes.rgb.reshape(e["mode_rgb"].shape))
    # FP64 sums in the same order, rounded once to the stored precision
    np.testing.assert_allclose(e["mode_pos"], modes.pos.reshape(e["mode_pos"].shape), rtol=2e-7, atol=1e-9)
    np.testing.assert_allclose(e["mode_U"], modes.U.reshape(e["mode_U"].shape), rtol=2e-7, atol=1e-9)
    assert modes.nmodes.max() > 0
    g.close()
    ctx.close()


@pytest.mark.parametrize("offset", [0.0, 1e-7, -3e-6, 1e-38])
def test_means_of_values_of_any_range(rg, offset):
    """A plane seen head-on: one column of points lies at x = offset, so the
    sums of a cluster's x are exact or, where their bits span more than 53,
    rounded in index order."""
    fp = dict(workloads.FOREST_DEFAULT, n_trees=1, depth=1, kappa=700, m_max=8, min_cluster_size=3, tau_c=0.15,
              grid_step=2)
    ctx = rg.Context(0, arena_bytes=1 << 28)
    g = rg.Forest.random(ctx, fp, 3)
    o = oracle.forest_random(1, 1, fp["p_depth"], (fp["delta_lo"], fp["delta_hi"]),
                             (fp["tau_depth_lo"], fp["tau_depth_hi"]), (fp["tau_rgb_lo"], fp["tau_rgb_hi"]),
                             bool(fp["tau_zero"]), 3)
    res = oracle.Reservoirs(o, fp["kappa"], 3)
    K = dataclasses.replace(rooms.intrinsics_for(640, 480), width=96, height=72, fx=120.0, fy=120.0, cx=48.0, cy=36.0)
    rng = np.random.default_rng(4)
    d = (2.0 + 0.05 * rng.random((72, 96))).astype(np.float32)
    rgb = rng.integers(0, 256, (72, 96, 3), dtype=np.uint8)
    T = np.eye(4)
    T[0, 3] = offset
    g.adapt(d, rgb, K, T)
    res.add_frame(d, rgb, K, T, fp["grid_step"], 0)
    g.update_modes(-1)
    modes = oracle.Modes(res.n_leaves, fp["m_max"])
    oracle.update_modes(res, modes, fp["sigma"], fp["tau_c"], fp["min_cluster_size"], cov_eps=fp["cov_eps"],
                        fp16_offsets=True)
    e = g.export(reservoirs=True)
    np.testing.assert_array_equal(e["res_count"], res.count)
    np.testing.assert_array_equal(e["nmodes"], modes.nmodes)
    np.testing.assert_array_equal(e["mode_size"], modes.size.reshape(e["mode_size"].shape))
    np.testing.assert_allclose(e["mode_pos"], modes.pos.reshape(e["mode_pos"].shape), rtol=2e-7, atol=1e-9)
    np.testing.assert_allclose(e["mode_U"], modes.U.reshape(e["mode_U"].shape), rtol=2e-7, atol=1e-9)
    assert modes.size.max() > 50
    g.close()
    ctx.close()


@pytest.mark.parametrize("m_max,precision,chunk", [(1, 0, 1), (7, 1, 5), (50, 1, 11), (64, 0, 16), (33, 1, 40)])
def test_streaming_store_catches_up(rg, m_max, precision, chunk):
    """After every round-robin update the front store of a streaming forest
    holds what the single store of another holds."""
    fp = dict(workloads.FOREST_DEFAULT, n_trees=2, depth=3, kappa=120, m_max=m_max, min_cluster_size=2, tau_c=0.15,
              grid_step=3, mode_precision=precision)
    ctx = rg.Context(0, arena_bytes=1 << 28)
    forests = [rg.Forest.random(ctx, fp, 8) for _ in range(2)]
    forests[1].set_streaming(True)
    room = rooms.Room((4.0, 3.0, 2.5), 5)
    K = dataclasses.replace(rooms.intrinsics_for(640, 480), width=96, height=72, fx=120.0, fy=120.0, cx=48.0, cy=36.0)
    for i, T in enumerate(rooms.training_trajectory(room, 5)):
        d, rgb = rooms.render(room, K, T, noise_seed=40 + i)
        stores = []
        for f in forests:
            f.adapt(d, rgb, K, T)
            f.update_modes(chunk)
            stores.append(f.export())
        a, b = stores
        np.testing.assert_array_equal(a["nmodes"], b["nmodes"])
        held = np.arange(m_max)[None, :] < a["nmodes"][:, None]  # the others are not set before a leaf's first update
        for k in ("mode_pos", "mode_rgb", "mode_U", "mode_size"):
            np.testing.assert_array_equal(a[k][held], b[k][held], err_msg=k)
    assert held.any()
    for f in forests:
        f.close()
    ctx.close()
