"""Handles destroyed parents first, as a garbage collector that finalises a cycle may do."""
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_children_outlive_their_parents():
    ctx = gsp.Context(0)
    sc = I.cornell_box(width=16, height=16)
    for _ in range(20):  # freed memory is soon reused
        s = gsp.Scene(ctx, sc)
        r = gsp.Renderer(s, gsp.sppm_params(sc, 100, seed=3, r0_frac=0.05))
        r.run(1)
        r.sync()
        h, s.h = s.h, None
        gsp.gsp_scene_destroy(h)
        r.close()
    c2 = gsp.Context(0)
    s = gsp.Scene(c2, sc)
    h, c2.h = c2.h, None
    gsp.gsp_context_destroy(h)
    s.close()
    assert gsp.Scene(ctx, sc).trace(torch.from_numpy(I.random_rays(100, seed=1)).cuda())[0].numel() == 100
    ctx.sync()
