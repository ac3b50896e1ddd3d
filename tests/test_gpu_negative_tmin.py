"""Rays with a negative tmin, from just behind the origin to -inf, with unit and long directions: the
triangles of the default walk against every triangle in turn (Moller-Trumbore in FP32, operation by
operation), in a soup and in a floor whose boxes have no extent along one axis, for both builders, at ray
counts walked by one lane, four lanes and a whole warp per ray."""
import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def floor(g):
    """A g x g grid of squares at height 0."""
    sc = I.random_soup(1, seed=1)
    x = np.linspace(-1, 1, g + 1, dtype=np.float32)
    verts = np.stack(np.broadcast_arrays(x[:, None], np.float32(0), x[None, :]), -1).reshape(-1, 3)
    a = (np.arange(g)[:, None] * (g + 1) + np.arange(g)[None, :]).reshape(-1)
    tris = np.concatenate([np.stack([a, a + 1, a + g + 2], -1), np.stack([a, a + g + 2, a + g + 1], -1)])
    return I.Scene(verts=np.ascontiguousarray(verts), tris=tris.astype(np.int32),
                   tri_mat=np.zeros(len(tris), np.int32), mats=sc.mats, camera=sc.camera)


def fma(a, b, c):
    """FP32 a b + c rounded once (but for the rounding of the sum to FP64 before that)."""
    return (a.double() * b.double() + c.double()).float()


def every_triangle(sc, rays):
    """Index of the closest triangle of each ray, -1 for none (ties: the smallest index). The products and
    fused sums of the library's device code, in its order."""
    v = torch.from_numpy(sc.verts).cuda()[torch.from_numpy(sc.tris).cuda().long()]
    v0, e1, e2 = v[:, 0], v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
    out = []
    for r in rays.split(256):
        o, d = r[:, None, 0:3], r[:, None, 4:7]

        def cross(a, b):
            return tuple(fma(a[..., i], b[..., j], -(a[..., j] * b[..., i])) for i, j in ((1, 2), (2, 0), (0, 1)))

        def dot(a, b):
            return fma(a[..., 2], b[2], fma(a[..., 1], b[1], a[..., 0] * b[0]))

        p = cross(d, e2)
        det = dot(e1, p)
        f = 1.0 / det
        s = o - v0
        u = f * dot(s, p)
        q = cross(s, e1)
        w = f * dot(d, q)
        t = f * dot(e2, q)
        ok = (det != 0) & (u >= 0) & (w >= 0) & (u + w <= 1) & (t > r[:, None, 3]) & (t < r[:, None, 7])
        t = torch.where(ok, t, float("inf"))
        best = t.min(dim=1, keepdim=True).values
        first = (t == best).int().argmax(dim=1)
        out.append(torch.where(ok.any(dim=1), first, -1).int())
    return torch.cat(out)


@pytest.mark.parametrize("builder", ["host", "device"])
@pytest.mark.parametrize("make", [lambda: I.random_soup(3000, seed=2, size=0.1), lambda: floor(40)], ids=["soup", "floor"])
@pytest.mark.parametrize("length", [1.0, 20.0])
def test_closest_hits(make, builder, length):
    sc = make()
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, sc, builder=builder)
    rays = torch.from_numpy(I.random_rays(9001, seed=8)).cuda()
    rays[:, 4:7] *= length
    for tmin in (-0.5, -3.0, -1e6, -3.4028234663852886e38, -float("inf")):
        rays[:, 3] = tmin / length
        want = every_triangle(sc, rays)
        assert int((want >= 0).sum()) > 1000
        for n in (1, 7, 33, 4865, 9001):
            assert torch.equal(s.trace(rays[:n])[0], want[:n]), (tmin, n)
    ctx.sync()
    ctx.close()


@pytest.mark.parametrize("every", [2, 7, 400])
@pytest.mark.parametrize("n", [33, 9001, 700_000])
def test_among_other_rays(every, n):
    """Every second, seventh or 400th ray starts behind its origin: warps that change to the form of the walk for
    such rays, at their first rays and in between, give every ray the hit it has alone."""
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, I.random_soup(3000, seed=2, size=0.1))
    rays = torch.from_numpy(I.random_rays(n, seed=9)).cuda()
    ahead = s.trace(rays)
    rays[:, 3] = -2.0
    behind = s.trace(rays)
    some = torch.zeros(n, dtype=torch.bool, device="cuda")
    some[every - 1::every] = True
    rays[:, 3] = torch.where(some, -2.0, 0.0)
    mixed = s.trace(rays)
    for a, b, m in zip(ahead, behind, mixed):
        assert torch.equal(torch.where(some, b, a), m)
    ctx.sync()
    ctx.close()
