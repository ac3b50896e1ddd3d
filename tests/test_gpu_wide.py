"""The four-wide walk against the walk of the hit/miss links on the GPU (a scene with a step limit
follows its links): triangles and t bit for bit at the ray counts where the launch changes shape and
at the smallest trees, for both builders; renders bit for bit in every mode."""
import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LINKS = 2**31 - 1  # a step limit that nothing reaches


@pytest.fixture(scope="module")
def ctx():
    c = gsp.Context(0)
    yield c
    c.close()


def both(scene, rays):
    """(wide, links) results as int32 bit patterns"""
    out = []
    for limit in (0, LINKS):
        gsp.gsp_scene_set_step_limit(scene.h, limit)
        out.append([x.view(torch.int32).cpu().numpy() for x in scene.trace(rays, with_uv=True)])
    gsp.gsp_scene_set_step_limit(scene.h, 0)
    return out


@pytest.mark.parametrize("builder", ["host", "device"])
@pytest.mark.parametrize("ntris", [1, 5, 8, 9, 300, 20_000])
def test_closest_hits(ctx, ntris, builder):
    sc = I.random_soup(ntris, seed=ntris, size=0.1)
    s = gsp.Scene(ctx, sc, builder=builder)
    rays = I.random_rays(20_011, seed=5)
    rays[::3, 7] = 1.0   # finite tmax
    rays[::5, 3] = 0.3   # tmin past some hits
    rays[::7, 4] = 0.0   # axis-parallel
    rays = torch.from_numpy(rays).cuda()
    for n in (1, 2, 9, 31, 33, 129, 4865, 20_011):
        wide, links = both(s, rays[:n])
        for a, b in zip(wide, links):
            assert np.array_equal(a, b), n
    ctx.sync()


@pytest.mark.parametrize("per_warp", [32, 128])
@pytest.mark.parametrize("extra", [0, 1])
def test_long_calls_equal_their_parts(ctx, per_warp, extra):
    """The line between static and dynamic chunks (32 rays per warp) and the line between hits
    re-evaluated in the kernel and through a list (128) do not show in the results."""
    n = torch.cuda.get_device_properties(0).multi_processor_count * 32 * per_warp + extra
    sc = I.random_soup(3000, seed=2, size=0.1)
    s = gsp.Scene(ctx, sc)
    rays = torch.from_numpy(I.random_rays(n, seed=6)).cuda()
    whole = s.trace(rays, with_uv=True)
    part = 4000
    for k in range(0, n, part):
        for a, b in zip(whole, s.trace(rays[k:k + part].clone(), with_uv=True)):
            assert torch.equal(a[k:k + part].view(torch.int32), b.view(torch.int32)), k
    ctx.sync()


@pytest.mark.parametrize("photon_mode", [gsp.FULL_PATH, gsp.REGEN])
@pytest.mark.parametrize("make,w,h,photons", [(I.cornell_box, 37, 21, 700), (I.full_scene, 96, 64, 20_000),
                                              (I.shaded_scene, 64, 48, 9_000),
                                              (I.full_scene, 300, 201, 400_000)])  # pools refilled from the queue
def test_renders(ctx, make, w, h, photons, photon_mode):
    sc = make(width=w, height=h) if make is I.cornell_box else make(width=w, height=h, plane_quads=32, sphere_n=9)
    s = gsp.Scene(ctx, sc)
    images = []
    for limit in (0, LINKS):
        gsp.gsp_scene_set_step_limit(s.h, limit)
        r = gsp.Renderer(s, gsp.sppm_params(sc, photons, seed=3, r0_frac=0.03, photon_mode=photon_mode))
        r.run(3)
        r.sync()
        images.append(r.image())
        b = gsp.Renderer(s, gsp.sppm_params(sc, photons, seed=3, r0_frac=0.03, photon_mode=photon_mode))
        batch = gsp.Batch([b])
        batch.run(3)
        b.sync()
        images.append(b.image())
        batch.close()
    assert float(images[0].sum()) > 0
    for other in images[1:]:
        assert torch.equal(images[0], other)
