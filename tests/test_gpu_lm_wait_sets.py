"""LM waits that run out in every cluster shape: one CTA per SM with sets of
hypotheses (few frames, 50 modes per pixel) and two per SM (many frames),
rounds of many hypotheses and rounds whose passes read the table directly.
The call times out, the next one with the default bound gives the same bits
as before, and its first frame is the oracle's."""
import numpy as np
import pytest

import oracle
from tests import helpers as H
from tests.test_gpu_launch_shapes import FIELDS, model, rg  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 12, 40])
@pytest.mark.parametrize("n_cull", [64, 8])
def test_lm_waits_run_out_then_recover(rg, model, n, n_cull):  # noqa: F811
    import torch
    w, f, scene, nodes, modes, queries = model
    p = dict(w.ransac, n_trees_used=5, k_top=10, n_cull=n_cull, n_hyp=200, max_iter=500)
    rel = rg.Relocaliser(f, scene, p, w.width, w.height, n)
    depth = np.stack([q[0] for q in queries[:n]])
    rgb = np.stack([q[1] for q in queries[:n]])
    seeds = [q[3] for q in queries[:n]]
    before = rel.relocalise_batch(depth, rgb, w.K, seeds)
    assert before[0]["n_hypotheses"] > 8  # more than the passes that read the table directly take
    rel.set_wait_limit(0)  # every tile wait gives up at once
    with pytest.raises(rg.RelocError) as e:
        rel.relocalise_batch(depth, rgb, w.K, seeds)
    assert e.value.status == 5  # RL_ERR_TIMEOUT
    torch.cuda.synchronize()  # the context is still usable
    for probes in (1, 2, 8):  # copies and stages late for some of the waits, for all or for none
        rel.set_wait_limit(probes)
        try:
            got = rel.relocalise_batch(depth, rgb, w.K, seeds)
        except rg.RelocError as e:
            assert e.status == 5
            continue
        for a, b in zip(got, before):
            np.testing.assert_array_equal(a["chosen_pose"], b["chosen_pose"], err_msg=f"{probes} probes")
    rel.set_wait_limit(-1)
    for graphs in (False, True):
        rel.set_graphs(graphs)
        after = rel.relocalise_batch(depth, rgb, w.K, seeds)
        for a, b in zip(after, before):
            for k in FIELDS:
                np.testing.assert_array_equal(a[k], b[k], err_msg=f"{k}, graphs={graphs}")
    d, c, _, seed = queries[0]
    lv = oracle.forest_leaves(nodes, d, c, w.K.fx, n_trees=5)
    run = H.OracleRun(p, d, c, w.K, lv, modes, w.room().lo, w.room().hi, seed, 1 << w.forest["depth"])
    H.compare_results(rg, after[0], rel.debug(0), run, dict(oracle.PARAM_DEFAULTS, **p), f"{n} frames")
    rel.close()
