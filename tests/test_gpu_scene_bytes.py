"""What a scene's tree takes on the device: stats.device_bytes against the sizes of its arrays, counted from
the exported tree. The four-wide form is there for the scenes that are walked in it only."""
import numpy as np
import pytest

from paper_1505_06022_gb300 import gsp, inputs as I

pytestmark = pytest.mark.gpu


def wide_entries(nodes):
    """Internal nodes at even depth of a tree given in preorder (an internal node's second child is where the
    first one's miss link leads)."""
    words, miss = nodes.view(np.int32)[:, 7], nodes.view(np.int32)[:, 3]
    count, todo = 0, [(0, 0)]
    while todo:
        n, depth = todo.pop()
        if words[n] >= 0:
            continue
        count += depth % 2 == 0
        todo += [(n + 1, depth + 1), (int(miss[n + 1]), depth + 1)]
    return count


@pytest.mark.parametrize("builder", ["host", "device"])
@pytest.mark.parametrize("link_sets,scale", [(6, 1.0), (1, 1.0), (6, 1e9)])
def test_device_bytes(builder, link_sets, scale):
    sc = I.random_soup(700, seed=4, size=0.1)
    sc.verts *= np.float32(scale)
    ctx = gsp.Context(0)
    s = gsp.Scene(ctx, sc, builder=builder, link_sets=link_sets)
    nodes = gsp.bvh_export_full(s.h, sc.ntris)[0]
    nn = len(nodes)
    pairs = (nn - 1) // 2 if builder == "host" else sc.ntris - 1  # the device build has one per radix-tree node
    wide = wide_entries(nodes) if link_sets == 6 and scale == 1.0 else 0
    want = 32 * link_sets * (nn + 1) + 48 * sc.ntris + 64 * pairs + 128 * wide + 32 * sc.ntris
    assert s.stats["device_bytes"] == want
    ctx.sync()
    ctx.close()
