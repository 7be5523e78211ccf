"""ICP by a cluster of blocks per pose (few poses in a call), whose warps
evaluate pixels or add up terms and meet at a barrier per chunk of pixels,
against a block per pose (160 poses in a call): the same bits, whatever the
levels, strides and images, down to fewer pixels than one chunk has."""
import numpy as np
import pytest

from synth import rooms

pytestmark = pytest.mark.gpu

LEVELS = {
    "one level, one iteration": dict(icp_levels=1, icp_stride=(1, 1, 1), icp_iters=(1, 1, 1), icp_dist=(0.1, 0.1, 0.1)),
    "odd strides": dict(icp_levels=3, icp_stride=(7, 3, 2), icp_iters=(2, 1, 5), icp_dist=(0.2, 0.1, 0.04)),
    "whole images": dict(icp_levels=2, icp_stride=(16, 1, 1), icp_iters=(3, 4, 1), icp_dist=(0.1, 0.03, 0.1)),
}


@pytest.mark.parametrize("levels", list(LEVELS))
@pytest.mark.parametrize("size", [(1, 1), (16, 16), (33, 31), (64, 48), (161, 119)])
def test_teams_match_single_blocks(size, levels):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    room = rooms.Room((4.0, 3.0, 2.5), 5)
    f = 0.9 * max(size)
    K = rooms.Intrinsics(f, f, size[0] / 2, size[1] / 2, *size)
    truth = rooms.query_poses(room, 1, seed=31)[0]
    d, _ = rooms.render(room, K, truth, noise_seed=3)
    d = rooms.mask_depth(d, 0.1, 4)
    rng = np.random.default_rng(9)
    poses = np.repeat(truth[None], 160, 0)
    poses[:, :3, 3] += rng.uniform(-0.03, 0.03, (160, 3))
    poses[2, :3, 3] = [9.0, 1.0, 1.0]  # outside the box
    ctx = rg.Context(0, arena_bytes=64 << 20)
    scene = rg.Scene(ctx, room.lo, room.hi)
    icp = LEVELS[levels]
    whole = scene.icp_poses(d, K, poses, **icp)
    for n in (3, 57, 100):  # clusters of eight, of eight, of four
        for a, b in zip(scene.icp_poses(d, K, poses[:n], **icp), whole):
            np.testing.assert_array_equal(a, b[:n], err_msg=f"{n} poses")
    if min(size) > 30:
        assert whole[1].any()
    scene.close()
    ctx.close()
