"""Host buffers that are page-locked in parts: a hole between two registrations, two registrations side by side,
the tail alone missing. Each gives the results of the same rays on the device, through whichever path takes
such a buffer."""
import mmap

import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PAGES = 12


@pytest.fixture(scope="module")
def scene():
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, I.random_soup(3000, seed=2, size=0.1))
    yield s
    ctx.close()


def pages():
    """A page-aligned array of PAGES pages."""
    n = PAGES * mmap.PAGESIZE
    a = np.zeros(n + mmap.PAGESIZE, np.uint8)
    start = -a.ctypes.data % mmap.PAGESIZE
    return a[start:start + n]


@pytest.mark.parametrize("which", ["rays", "tri", "t"])
@pytest.mark.parametrize("parts", [((0, 4), (8, 12)), ((0, 6), (6, 12)), ((0, 11),), ((0, 12),)],
                         ids=["hole", "side by side", "tail missing", "whole"])
def test_registered_parts(scene, which, parts):
    buf = pages()
    n = buf.nbytes // (32 if which == "rays" else 4)
    rays = torch.from_numpy(I.random_rays(n, seed=6))
    want = scene.trace(rays.cuda())
    host = {"rays": rays.pin_memory(), "tri": torch.empty(n, dtype=torch.int32).pin_memory(),
            "t": torch.empty(n).pin_memory()}
    mine = torch.from_numpy(buf.view(np.int32 if which == "tri" else np.float32)).view(host[which].shape)
    mine.copy_(host[which])
    host[which] = mine
    rt = torch.cuda.cudart()
    done = []
    try:
        for a, b in parts:
            at = buf.ctypes.data + a * mmap.PAGESIZE
            assert int(rt.cudaHostRegister(at, (b - a) * mmap.PAGESIZE, 0)) == 0
            done.append(at)
        gsp.gsp_trace_closest_hit_host(scene.h, host["rays"], host["tri"], host["t"])
    finally:
        for at in done:
            rt.cudaHostUnregister(at)
    assert torch.equal(want[0].cpu(), host["tri"])
    assert torch.equal(want[1].cpu(), host["t"])
