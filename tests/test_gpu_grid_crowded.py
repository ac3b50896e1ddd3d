"""Parts of the hash grid with more points than their block's lanes hold: counts around a part that is held, a
batch of points fetched at once and several batches, in one bucket and in a few, against the oracle, bit for
bit."""
import numpy as np
import pytest

import oracle as O
from paper_1505_06022_gb300 import gsp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spread", [0.0, 0.02])
@pytest.mark.parametrize("bits", [0, 9, 20])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 2047, 2048, 2049, 16_385, 300_007])
def test_order(n, bits, spread):
    rng = np.random.default_rng(n + bits)
    h = 0.05
    x = (0.01 + rng.normal(scale=spread, size=(n, 3))).astype(np.float32)
    x = x[O.hash_grid(x, h, 1 << bits)[3] == 0]  # a coordinate on a cell face may round to either cell
    _, order, starts, _ = O.hash_grid(x, h, 1 << bits)
    pos = torch.zeros((len(x), 4), dtype=torch.float32, device="cuda")
    pos[:, :3] = torch.from_numpy(x).cuda()
    ctx = gsp.Context(0)
    got_order, got_starts = gsp.gsp_hash_grid_build(ctx.h, pos, h, 1 << bits)
    ctx.sync()
    np.testing.assert_array_equal(got_order.cpu().numpy().view(np.uint32), order)
    np.testing.assert_array_equal(got_starts.cpu().numpy().view(np.uint32), starts)
    ctx.close()
