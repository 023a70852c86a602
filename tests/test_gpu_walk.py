"""The warp walk over CGA positions (k_walk.cuh) at its edges: counts around a
lane group, a step and a warp's share; slabs and columns that open at every
position or never; output buffers off the 16-byte boundary.  Whole numbers, so
equality with the oracle's decode."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _voxels(shape, n):
    i = np.arange(n)
    if shape == "column":      # one column, one slab
        return np.stack([0 * i + 5, 0 * i + 9, i % 4096], 1)
    if shape == "row":         # a column per voxel, one slab
        return np.stack([0 * i + 5, i % 4096, 0 * i + 1], 1)
    if shape == "diagonal":    # a slab per voxel
        return np.stack([i % 4096, (7 * i) % 4096, (3 * i) % 4096], 1)
    if shape == "pairs":       # slabs and columns that open inside a lane group
        return np.stack([i // 40, (i // 3) % 4096, i % 3], 1)
    rng = np.random.default_rng(n)
    return rng.integers(0, 64, size=(n, 3))


@pytest.mark.parametrize("shape", ["column", "row", "diagonal", "pairs", "random"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 1023, 1025, 4096, 40_001])
def test_decode_at_step_edges(shape, n):
    pts = ((_voxels(shape, n) + 0.5) / 4096.0).astype(np.float32)
    og = oracle.grid_from_box([0, 0, 0], 1.0, 12)
    want = oracle.decode(oracle.build(pts, og)).astype(np.int64)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, 12))
    for off in (0, 1, 4):
        room = torch.full((off + 3 * n + 5,), -1, dtype=torch.int32, device="cuda")
        cga.cga_decode(a, out=room[off:])
        got = room.cpu().numpy()
        assert np.array_equal(got[off:off + want.size].reshape(-1, 3), want)
        assert np.all(got[:off] == -1) and np.all(got[off + want.size:] == -1)
