"""Clustering (Sec. 3.2.2) where no density bound decides: points so close
together that every term of a density is exactly 1, so that all densities are
exactly equal and the lower index is the denser one.  Every point then takes
the last stage of the parent search, FP64 densities summed in index order.
The leaf's modes against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from synth import rooms, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size,missing", [((9, 7), 0.3), ((13, 10), 0.5), ((40, 31), 0.5), ((96, 72), 0.5)])
def test_the_lower_index_is_the_denser_point(size, missing):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    # points 2e-12 m apart: exp(-d^2 / 2 sigma^2) = 1 in FP64; tau_c reaches the eight neighbours
    fp = dict(workloads.FOREST_DEFAULT, n_trees=1, depth=1, kappa=4096, m_max=64, min_cluster_size=1, p_depth=1.0,
              tau_c=3e-12, grid_step=1, mode_precision=0)
    K = dataclasses.replace(rooms.intrinsics_for(640, 480), width=size[0], height=size[1], fx=1e12, fy=1e12,
                            cx=size[0] / 2, cy=size[1] / 2)
    rng = np.random.default_rng(size[0])
    d = rooms.mask_depth(np.full((size[1], size[0]), 2.0, np.float32), missing, 5)
    rgb = rng.integers(0, 256, (size[1], size[0], 3), dtype=np.uint8)
    ctx = rg.Context(0, arena_bytes=1 << 28)
    g = rg.Forest.random(ctx, fp, 3)
    o = oracle.forest_random(1, 1, 1.0, (fp["delta_lo"], fp["delta_hi"]), (fp["tau_depth_lo"], fp["tau_depth_hi"]),
                             (fp["tau_rgb_lo"], fp["tau_rgb_hi"]), bool(fp["tau_zero"]), 3)
    res = oracle.Reservoirs(o, fp["kappa"], 3)
    g.adapt(d, rgb, K, np.eye(4))
    res.add_frame(d, rgb, K, np.eye(4), 1, 0)
    g.update_modes(-1)
    modes = oracle.Modes(res.n_leaves, fp["m_max"])
    oracle.update_modes(res, modes, fp["sigma"], fp["tau_c"], fp["min_cluster_size"], cov_eps=fp["cov_eps"],
                        fp16_offsets=False)
    e = g.export(reservoirs=True)
    np.testing.assert_array_equal(e["res_count"], res.count)
    assert res.count.max() == int((d > 0).sum())  # one leaf holds every point
    np.testing.assert_array_equal(e["nmodes"], modes.nmodes)
    np.testing.assert_array_equal(e["mode_size"], modes.size.reshape(e["mode_size"].shape))
    np.testing.assert_array_equal(e["mode_rgb"], modes.rgb.reshape(e["mode_rgb"].shape))
    assert modes.nmodes.max() > 1
    g.close()
    ctx.close()
