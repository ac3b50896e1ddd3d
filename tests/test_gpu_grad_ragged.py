"""The gradient at pixel and path counts that leave warps and blocks partly filled, with 17 materials,
against the oracle's FP64 gradient, to the tolerance of the other gradient tests."""
import numpy as np
import pytest

import oracle as O
from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,photons", [(37, 21, 20_001), (33, 1, 5000), (5, 3, 97)])
def test_ragged_sizes(w, h, photons):
    kw = dict(photons_per_pass=photons, seed=4, r0_frac=0.03)
    sc = I.grad_scene(width=w, height=h, plane_quads=48, sphere_n=8)
    orc = O.Sppm(sc, O.default_params(sc, **kw))
    orc.enable_grad()
    orc.run(2)
    g = orc.image() - 0.05 * np.random.default_rng(7).standard_normal((h, w, 3))
    ga_o, gl_o = orc.grad(g)
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, sc)
    r = gsp.Renderer(s, gsp.sppm_params(sc, **kw))
    r.enable_grad(2)
    r.run(2)
    ga, gl = (x.cpu().numpy() for x in r.grad(torch.from_numpy(g.astype(np.float32)).cuda()))
    r.sync()
    for x in (r, s, ctx):
        x.close()
    diffuse = sc.mats["type"] == I.DIFFUSE
    for a, b in ((ga[diffuse], ga_o[diffuse]), (gl, gl_o)):
        assert np.all(np.abs(a - b) <= 1e-3 * np.maximum(np.abs(b), 1e-3 * np.linalg.norm(b)))
    assert np.all(ga[~diffuse] == 0)
