"""What the library asks of the caller's arena does not grow: programs size it
once, some to the byte."""
import dataclasses

import numpy as np
import pytest

from synth import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_12163_gb300 as rg
    rg.lib()
    return rg


# (trees, modes per leaf, frame, frames) -> bytes that creating the relocaliser has taken so far at most: 200 and 120
# modes per pixel (no colour masks), 40 (colour masks), six trees (no pixel records)
CREATED = {
    (5, 40, (95, 71), 1): 3305472,
    (5, 40, (640, 480), 2): 27930880,
    (3, 40, (640, 480), 2): 23233280,
    (5, 8, (640, 480), 2): 28451840,
    (6, 8, (640, 480), 2): 15081728,
}


@pytest.mark.parametrize("case", list(CREATED), ids=str)
def test_relocaliser(rg, case):
    trees, m_max, size, batch = case
    w = workloads.small_case()
    ctx = rg.Context(0, arena_bytes=1 << 28)
    scene = rg.Scene(ctx, w.room().lo, w.room().hi)
    f = rg.Forest.random(ctx, dict(w.forest, n_trees=trees, depth=6, m_max=m_max), 3)
    before = ctx.usage()[0]
    rel = rg.Relocaliser(f, scene, dict(w.ransac, n_trees_used=trees, k_top=40), size[0], size[1], batch)
    assert ctx.usage()[0] - before <= CREATED[case]
    rel.close()
    f.close()
    scene.close()
    ctx.close()


@pytest.mark.parametrize("trees,depth", [(1, 1), (5, 6), (3, 15), (16, 4)])
def test_adaptation(rg, trees, depth):
    """Two words per example and tree, and a point per grid pixel, whatever
    the number of leaves; again only for a larger frame."""
    import torch
    w = workloads.small_case()
    ctx = rg.Context(0, arena_bytes=1 << 28)
    f = rg.Forest.random(ctx, dict(w.forest, n_trees=trees, depth=depth, m_max=2, kappa=8, grid_step=4), 3)
    start = ctx.usage()[0]
    most = 0
    for size in ((4, 4), (96, 72), (160, 121), (95, 70), (640, 480)):
        K = dataclasses.replace(w.K, width=size[0], height=size[1])
        d = torch.full((size[1], size[0]), 2.0, device="cuda")
        f.adapt(d, torch.zeros(size[1], size[0], 3, dtype=torch.uint8, device="cuda"), K, np.eye(4))
        most = max(most, -(-size[0] // 4) * -(-size[1] // 4))
        asked = sum(-(-b // 256) * 256 for b in (4 * most * trees, 16 * most, 4 * most * trees))
        assert ctx.usage()[0] - start <= asked, size
    assert f.export()["res_count"].sum() == trees * (1 + 24 * 18 + 40 * 31 + 24 * 18 + 160 * 120)
    f.close()
    ctx.close()
