"""Several passes in one call, whose hash grids are built on the tracing streams (small renderers, a grid
per trace set) or before each gather (larger ones, one grid), against the passes one call at a time: the
same kernels on the same data, so bit for bit, on both sides of the line and with the split of long queries."""
import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gsp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("make,w,h,photons", [
    (I.cornell_box, 37, 21, 700),
    (I.full_scene, 64, 48, 1 << 17),        # 2^22 deposit slots: a grid per trace set
    (I.full_scene, 64, 48, (1 << 17) + 1),  # one grid
    (I.full_scene, 512, 512, 60_000),       # long queries listed per trace set
])
def test_passes_together_equal_passes_alone(ctx, make, w, h, photons):
    sc = make(width=w, height=h) if make is I.cornell_box else make(width=w, height=h, plane_quads=32, sphere_n=9)
    s = gsp.Scene(ctx, sc)
    params = gsp.sppm_params(sc, photons, seed=3, r0_frac=0.03)
    got = []
    for calls in ((5,), (1, 1, 1, 1, 1), (2, 3)):
        r = gsp.Renderer(s, params)
        for n in calls:
            r.run(n)
        r.sync()
        got.append([r.image().cpu().numpy(), r.last_deposits()] + [np.asarray(v.cpu()) for v in r.state().values()
                                                                   if torch.is_tensor(v)])
        r.close()
    assert np.abs(got[0][0]).sum() > 0
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
    s.close()
