"""The hash grid at the sizes where its split into tiles and parts changes shape: input counts around a
tile, bucket counts from one to past the point where the radix sort takes over, inputs that crowd into
one bucket (a part larger than its block holds in registers), against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1505_06022_gb300 import gsp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("bits", [0, 1, 8, 9, 18, 19, 21, 22])
@pytest.mark.parametrize("n", [1, 255, 257, 3073, 150_001])
def test_matches_oracle(n, bits, crowded):
    rng = np.random.default_rng(n + bits)
    h = 0.5 if crowded else 0.01
    x = rng.normal(scale=0.05 if crowded else 1.0, size=(n, 3)).astype(np.float32)
    x = x[O.hash_grid(x, h, 1 << bits)[3] == 0]  # a coordinate on a cell face may round to either cell
    _, order, starts, _ = O.hash_grid(x, h, 1 << bits)
    pos = torch.zeros((len(x), 4), dtype=torch.float32, device="cuda")
    pos[:, :3] = torch.from_numpy(x).cuda()
    ctx = gsp.Context(0)
    for _ in range(2):  # the second build reuses the scratch
        got_order, got_starts = gsp.gsp_hash_grid_build(ctx.h, pos, h, 1 << bits)
    ctx.sync()
    np.testing.assert_array_equal(got_order.cpu().numpy().view(np.uint32), order)
    np.testing.assert_array_equal(got_starts.cpu().numpy().view(np.uint32), starts)
    ctx.close()
