"""Surfaces that coincide: the smallest (t, triangle index) of every triangle in turn, whichever way a ray is
walked (one lane, four lanes, a whole warp), so whatever its place in a call."""
import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I
from test_gpu_negative_tmin import every_triangle, floor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def two_floors():
    """Two floors at one height, differently divided."""
    a, b = floor(40), floor(31)
    a.verts[:, 1] = b.verts[:, 1] = 0.3
    b.verts[:, ::2] += np.float32(0.013)
    return I.Scene(verts=np.concatenate([a.verts, b.verts]), tris=np.concatenate([a.tris, b.tris + len(a.verts)]),
                   tri_mat=np.concatenate([a.tri_mat, b.tri_mat]), mats=a.mats, camera=a.camera)


def one_plane():
    """Triangles over one another in one plane."""
    sc = I.random_soup(2500, seed=3, size=0.2)
    sc.verts[:, 1] = 0.37
    return sc


@pytest.mark.parametrize("builder", ["host", "device"])
@pytest.mark.parametrize("make", [two_floors, one_plane])
def test_closest_hits(make, builder):
    sc = make()
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, sc, builder=builder)
    rays = torch.from_numpy(I.random_rays(9001, seed=8)).cuda()
    for tmin in (0.0, -3.0):
        rays[:, 3] = tmin
        want = every_triangle(sc, rays)
        assert int((want >= 0).sum()) > 300
        for n in (1, 7, 33, 4865, 9001):
            assert torch.equal(s.trace(rays[:n])[0], want[:n]), (tmin, n)
    ctx.sync()
    ctx.close()
