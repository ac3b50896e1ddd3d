"""The walk of the hit/miss links (a scene with a step limit follows its links; one link set has them only)
and the stack walk against every triangle in turn: a negative tmin with boxes that have no extent along one
axis, and coincident surfaces."""
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I
from test_gpu_coincident import one_plane, two_floors
from test_gpu_negative_tmin import every_triangle, floor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walk", ["links", "one set", "stack"])
@pytest.mark.parametrize("make", [lambda: floor(40), two_floors, one_plane], ids=["floor", "two_floors", "one_plane"])
def test_closest_hits(make, walk):
    sc = make()
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, sc, link_sets=1 if walk == "one set" else 6)
    if walk == "links":
        gsp.gsp_scene_set_step_limit(s.h, 2**31 - 1)
    rays = torch.from_numpy(I.random_rays(9001, seed=8)).cuda()
    for tmin in (0.0, -3.0, -1e6, -float("inf")):
        rays[:, 3] = tmin
        want = every_triangle(sc, rays)
        assert int((want >= 0).sum()) > 300
        for n in (1, 33, 9001):
            got = s.trace(rays[:n], method="stack" if walk == "stack" else "mtbvh")[0]
            assert torch.equal(got, want[:n]), (tmin, n)
    ctx.sync()
    ctx.close()
