"""Clustering (Sec. 3.2.2) of leaves that hold points which are not finite, from
infinite or huge depths: a distance to such a point has no order, nor have the
densities it enters.  Modes against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from synth import rooms, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth,rows", [(np.inf, slice(10, 12)), (3e38, slice(10, 30)), (1e25, slice(10, 30)),
                                        (np.nan, slice(10, 30))])
@pytest.mark.parametrize("min_size,fp16", [(1, False), (3, True)])
def test_modes_match_the_oracle(depth, rows, min_size, fp16):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    fp = dict(workloads.FOREST_DEFAULT, n_trees=2, depth=3, kappa=700, m_max=12, min_cluster_size=min_size, tau_c=0.1,
              grid_step=2, mode_precision=int(fp16))
    room = rooms.Room((4.0, 3.0, 2.5), 5)
    K = dataclasses.replace(rooms.intrinsics_for(640, 480), width=96, height=72, fx=120.0, fy=120.0, cx=48.0, cy=36.0)
    ctx = rg.Context(0, arena_bytes=1 << 28)
    g = rg.Forest.random(ctx, fp, 8)
    o = oracle.forest_random(2, 3, fp["p_depth"], (fp["delta_lo"], fp["delta_hi"]),
                             (fp["tau_depth_lo"], fp["tau_depth_hi"]), (fp["tau_rgb_lo"], fp["tau_rgb_hi"]),
                             bool(fp["tau_zero"]), 8)
    res = oracle.Reservoirs(o, fp["kappa"], 8)
    for i, T in enumerate(rooms.training_trajectory(room, 3)):
        d, rgb = rooms.render(room, K, T, noise_seed=40 + i)
        if i == 1:
            d[rows, 20:60] = depth
        g.adapt(d, rgb, K, T)
        res.add_frame(d, rgb, K, T, 2, 0)
    g.update_modes(-1)
    modes = oracle.Modes(res.n_leaves, fp["m_max"])
    oracle.update_modes(res, modes, fp["sigma"], fp["tau_c"], min_size, cov_eps=fp["cov_eps"], fp16_offsets=fp16)
    e = g.export(reservoirs=True)
    np.testing.assert_array_equal(e["res_count"], res.count)
    held = np.arange(fp["kappa"])[None, :] < res.count[:, None]
    pos = res.pos.reshape(-1, fp["kappa"], 3)
    np.testing.assert_array_equal(e["res_pos"][held], pos[held])
    assert np.isfinite(pos[held]).all() == bool(np.isnan(depth) or depth == 1e25)
    np.testing.assert_array_equal(e["nmodes"], modes.nmodes)
    np.testing.assert_array_equal(e["mode_size"], modes.size.reshape(e["mode_size"].shape))
    np.testing.assert_array_equal(e["mode_rgb"], modes.rgb.reshape(e["mode_rgb"].shape))
    # FP64 sums rounded once to the stored precision
    np.testing.assert_allclose(e["mode_pos"], modes.pos.reshape(e["mode_pos"].shape), rtol=2e-7, atol=1e-9)
    np.testing.assert_allclose(e["mode_U"], modes.U.reshape(e["mode_U"].shape), rtol=2e-7, atol=1e-9)
    assert modes.nmodes.max() > 0
    g.close()
    ctx.close()
