"""Hypothesis generation where its path or its launch shape changes: teams of
warps per slot, more modes per pixel than the colour masks cover, frames whose
bitmap does not fit shared memory; winning iterations against the oracle."""
import numpy as np
import pytest

import oracle
from synth import rooms
from tests.test_gpu_launch_shapes import model, rg  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def oracle_iterations(p, d, c, w, K, nodes, modes, seed):
    lv = oracle.forest_leaves(nodes, d, c, K.fx, n_trees=p["n_trees_used"])
    r = oracle.relocalise(p, d, c, K, lv, modes, w.room().lo, w.room().hi, seed, 1 << w.forest["depth"], debug=True)
    return r["debug"]["hyp_iter"]


@pytest.mark.parametrize("redraw", [0, 1])
@pytest.mark.parametrize("n_hyp", [1, 6, 40])
def test_a_team_stops_at_its_mates_success(rg, model, n_hyp, redraw):  # noqa: F811
    """A slot of a small call is walked by up to 16 warps of a block, each of
    which stops where another has succeeded: the lowest success is the
    oracle's, whichever warp finds it, in tight and loose checks (late and
    early successes)."""
    w, f, scene, nodes, modes, queries = model
    found = []
    for thresh, err in ((30, 0.05), (120, 0.15)):
        p = dict(w.ransac, n_trees_used=5, k_top=10, n_hyp=n_hyp, n_cull=min(n_hyp, 24), max_iter=6000, redraw=redraw,
                 colour_thresh=thresh, max_trans_err=err)
        rel = rg.Relocaliser(f, scene, p, w.width, w.height, 1)
        for d, c, _, seed in queries[:6]:
            rel.relocalise(d, c, w.K, seed)
            got = rel.debug(0)["hyp_iter"]
            np.testing.assert_array_equal(got, oracle_iterations(p, d, c, w, w.K, nodes, modes, seed))
            found += [it for it in got if it >= 0]
        rel.close()
    assert max(found) > 64  # beyond the first warp's first group


@pytest.mark.parametrize("warps", [2, 4, 8, 16])
def test_block_size_does_not_change_a_small_call(rg, model, warps):  # noqa: F811
    """Blocks tuned on batches: in a call of few slots they grow to its teams,
    and in one of many slots hold this many slots."""
    w, f, scene, nodes, modes, queries = model
    for n_hyp, k_top in ((3, 10), (200, 10), (200, 40), (4096, 10)):  # colour masks and pixel records
        p = dict(w.ransac, n_trees_used=5, k_top=k_top, n_hyp=n_hyp, n_cull=min(n_hyp, 24), max_iter=700)
        rel = rg.Relocaliser(f, scene, p, w.width, w.height, 1)
        rel.set_tuning(dict(rel.tuning, hypgen_warps=warps))
        d, c, _, seed = queries[1]
        rel.relocalise(d, c, w.K, seed)
        np.testing.assert_array_equal(rel.debug(0)["hyp_iter"],
                                      oracle_iterations(p, d, c, w, w.K, nodes, modes, seed))
        rel.close()


@pytest.mark.parametrize("missing", [0.0, 0.6])
@pytest.mark.parametrize("n_hyp", [5, 300])
def test_records_with_redraws(rg, model, n_hyp, missing):  # noqa: F811
    """More modes per pixel than the masks cover, unusable pixels redrawn
    within an iteration; alone and beside other frames."""
    w, f, scene, nodes, modes, queries = model
    p = dict(w.ransac, n_trees_used=5, k_top=40, n_hyp=n_hyp, n_cull=min(n_hyp, 24), max_iter=700, redraw=1)
    rel = rg.Relocaliser(f, scene, p, w.width, w.height, 8)
    depth = np.stack([rooms.mask_depth(q[0], missing, 9 + i) for i, q in enumerate(queries[:8])])
    rgb = np.stack([q[1] for q in queries[:8]])
    seeds = [q[3] for q in queries[:8]]
    want = [oracle_iterations(p, depth[i], rgb[i], w, w.K, nodes, modes, seeds[i]) for i in range(8)]
    rel.relocalise_batch(depth, rgb, w.K, seeds)
    for i in range(8):
        np.testing.assert_array_equal(rel.debug(i)["hyp_iter"], want[i], err_msg=f"frame {i} of 8")
    rel.relocalise(depth[3], rgb[3], w.K, seeds[3])
    np.testing.assert_array_equal(rel.debug(0)["hyp_iter"], want[3])
    assert max(x.max() for x in want) >= 0
    rel.close()


@pytest.mark.parametrize("k_top", [10, 40])
@pytest.mark.parametrize("n_hyp,redraw", [(3, 0), (3, 1), (400, 0)])
def test_frames_whose_bitmap_does_not_fit(rg, model, n_hyp, redraw, k_top):  # noqa: F811
    """Above 524,288 pixels generation reads the colour masks, or the records,
    without the bitmap: teams of up to 16 warps, alone and beside others."""
    w, f, scene, nodes, modes, _ = model
    room = w.room()
    K = rooms.intrinsics_for(1024, 600)
    p = dict(w.ransac, n_trees_used=5, k_top=k_top, n_hyp=n_hyp, n_cull=min(n_hyp, 24),
             max_iter=6000 if n_hyp < 10 else 700, redraw=redraw)
    frames = [rooms.render(room, K, T, noise_seed=70 + i) for i, T in enumerate(rooms.query_poses(room, 3, seed=11))]
    depth = np.stack([rooms.mask_depth(d, 0.2, 5 + i) for i, (d, _) in enumerate(frames)])
    rgb = np.stack([c for _, c in frames])
    want = [oracle_iterations(p, depth[i], rgb[i], w, K, nodes, modes, 500 + i) for i in range(3)]
    rel = rg.Relocaliser(f, scene, p, 1024, 600, 3)
    rel.relocalise(depth[0], rgb[0], K, 500)
    np.testing.assert_array_equal(rel.debug(0)["hyp_iter"], want[0])
    rel.relocalise_batch(depth, rgb, K, [500, 501, 502])
    for i in range(3):
        np.testing.assert_array_equal(rel.debug(i)["hyp_iter"], want[i], err_msg=f"frame {i} of 3")
    assert max(x.max() for x in want) >= 0
    rel.close()
