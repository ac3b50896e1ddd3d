"""Closest hits for page-locked host buffers on both sides of the line between one launch that writes
host memory itself and two halves with copies, and with result buffers that it cannot write to as
pairs of floats: the results of the same rays on the device, bit for bit."""
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, I.random_soup(3000, seed=2, size=0.1))
    yield s
    ctx.close()


@pytest.mark.parametrize("uv", [None, 0, 1])  # offset of the uv buffer in floats
@pytest.mark.parametrize("n", [1, 33, 5000, 1 << 18, (1 << 18) + 1])
def test_host_results(scene, n, uv):
    rays = torch.from_numpy(I.random_rays(n, seed=6))
    want = scene.trace(rays.cuda(), with_uv=True)
    tri = torch.empty(n, dtype=torch.int32).pin_memory()
    t = torch.empty(n).pin_memory()
    buf = torch.empty(2 * n + 1).pin_memory()
    out = None if uv is None else buf[uv:uv + 2 * n].view(n, 2)
    gsp.gsp_trace_closest_hit_host(scene.h, rays.pin_memory(), tri, t, out)
    for a, b in zip(want, (tri, t) if out is None else (tri, t, out)):
        assert torch.equal(a.cpu().view(torch.int32), b.contiguous().view(torch.int32))
