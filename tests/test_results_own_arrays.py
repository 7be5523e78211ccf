"""Results as dictionaries (host code): each frame's arrays are its own."""
import numpy as np
import pytest

import paper_1810_12163_gb300 as rg


@pytest.mark.parametrize("n_chosen", [16, 5, 1, 0])
def test_each_frame_owns_its_arrays(n_chosen):
    rng = np.random.default_rng(n_chosen)
    out = (rg.Result * 3)()
    for i, r in enumerate(out):
        r.n_chosen, r.best, r.energy, r.level = n_chosen, i, 0.5 * i, i
        r.pose[:] = list(rng.random(16))
        for c in range(16):
            r.chosen_pose[c][:] = list(rng.random(16))
            r.chosen_energy[c], r.chosen_score[c], r.chosen_slot[c] = rng.random(), rng.random(), 7 * i + c
            r.chosen_icp_frac[c] = rng.random()
    want = []
    for r in out:
        want.append(dict(
            pose=np.array(r.pose).reshape(4, 4),
            chosen_pose=np.array([np.array(r.chosen_pose[c]).reshape(4, 4) for c in range(n_chosen)]),
            chosen_energy=np.array(r.chosen_energy[:n_chosen]), chosen_score=np.array(r.chosen_score[:n_chosen]),
            chosen_slot=np.array(r.chosen_slot[:n_chosen]),
            chosen_icp_frac=np.array(r.chosen_icp_frac[:max(n_chosen, 1)])))
    got = rg.result_dicts(out, 3)
    for i, (g, w) in enumerate(zip(got, want)):
        assert (g["n_chosen"], g["best"], g["energy"], g["level"]) == (n_chosen, i, 0.5 * i, i)
        for k, v in w.items():
            for other in (got[j] for j in range(3) if j != i):  # nothing of another frame is kept with it
                assert g[k].base is None or g[k].base is not other[k].base, k
            assert g[k].base is None or g[k].base.nbytes <= 8 * (16 + 16 * 16 + 3 * 16), k
            assert g[k].dtype == v.dtype and g[k].shape == v.shape, k
            np.testing.assert_array_equal(g[k], v, err_msg=k)
    got[0]["pose"][:] = -1.0
    np.testing.assert_array_equal(got[1]["pose"], want[1]["pose"])
    np.testing.assert_array_equal(np.array(out[0].pose).reshape(4, 4), want[0]["pose"])
