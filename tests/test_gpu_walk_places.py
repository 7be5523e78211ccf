"""The forest walk of a call whose pixels have more modes than the colour masks
cover, by where its packed frames fit: nowhere (up to three trees), the leaf
maps' array (four or five, also where a sub-batch's part of it starts off an
8-byte boundary); at the focal length of the call's nodes and at another one.
Every stage against the oracle, and batches against single frames."""
import dataclasses

import numpy as np
import pytest

import oracle
from tests import helpers as H
from tests.test_gpu_launch_shapes import FIELDS, model, rg  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(96, 72), (95, 71), (1, 1)])
@pytest.mark.parametrize("trees", [2, 3, 4, 5])
def test_walk_matches_the_oracle(rg, model, trees, size):  # noqa: F811
    w, f, scene, nodes, modes, queries = model
    p = dict(w.ransac, n_trees_used=trees, k_top=40, n_hyp=64, max_iter=500)
    frames = [(np.ascontiguousarray(d[:size[1], :size[0]]), np.ascontiguousarray(c[:size[1], :size[0]]), seed)
              for d, c, _, seed in queries[:25]]
    depth, rgb = np.stack([x[0] for x in frames]), np.stack([x[1] for x in frames])
    rel = rg.Relocaliser(f, scene, p, size[0], size[1], 25)  # three sub-batches of 9, 8 and 8 frames
    for zoom in (1.0, 1.3):  # the second call replays the first one's graph
        K = dataclasses.replace(w.K, width=size[0], height=size[1], fx=w.K.fx * zoom)
        alone = []
        for i in (0, 9):
            d, c, seed = frames[i]
            alone.append(rel.relocalise(d, c, K, seed))
            lv = oracle.forest_leaves(nodes, d, c, K.fx, n_trees=trees)
            run = H.OracleRun(p, d, c, K, lv, modes, w.room().lo, w.room().hi, seed, 1 << w.forest["depth"])
            H.compare_results(rg, alone[-1], rel.debug(0), run, dict(oracle.PARAM_DEFAULTS, **p),
                              f"{trees} trees, {size}, fx x {zoom}, frame {i}")
        got = rel.relocalise_batch(depth, rgb, K, [x[2] for x in frames])
        for i, a in zip((0, 9), alone):
            for k in FIELDS:
                np.testing.assert_array_equal(got[i][k], a[k], err_msg=f"{k} of frame {i}")
    rel.close()
