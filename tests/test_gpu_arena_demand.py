"""What the library asks of the caller's arena does not grow: programs size it
once, some to the byte."""
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
