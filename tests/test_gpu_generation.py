"""Hypothesis generation where its path or its launch shape changes: teams of
warps per slot, more modes per pixel than the colour masks cover, frames whose
bitmap does not fit shared memory; winning iterations against the oracle."""
import numpy as np
import pytest

import oracle
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
