"""xz and yz projections where the joined bits can go wrong: slabs that end inside a
step, one slab over many warps, slabs of one voxel, columns that fill words, the
smallest and widest grids of the bitmap form.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _voxels(kind, bits):
    side, rng = 1 << bits, np.random.default_rng(bits)
    if kind == "slab":       # one slab, in full where the grid is small
        n = min(side * side, 60_000)
        yz = rng.choice(side * side, size=n, replace=False)
        return np.stack([np.full(n, side // 2), yz // side, yz % side], -1)
    if kind == "diagonal":   # a voxel a slab
        i = np.arange(side)
        return np.stack([i, i, side - 1 - i], -1)
    if kind == "columns":    # full columns, several slabs a step and a slab over steps
        x = np.repeat(np.arange(0, side, max(1, side // 9)), 3)
        y = rng.integers(0, side, size=len(x))
        z = np.arange(side)
        return np.stack([np.repeat(x, side), np.repeat(y, side), np.tile(z, len(x))], -1)
    return rng.integers(0, side, size=(40_000, 3))


@pytest.mark.parametrize("bits", [5, 6, 10, 12, 13])
@pytest.mark.parametrize("kind", ["slab", "diagonal", "columns", "random"])
def test_planes(kind, bits):
    pts = ((_voxels(kind, bits) + 0.5) / (1 << bits)).astype(np.float32)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, bits))
    o = oracle.build(pts, oracle.grid_from_box([0, 0, 0], 1.0, bits))
    for plane in ("xz", "yz"):
        got, want = cga.cga_project(a, plane).download(), oracle.project(o, plane)
        for lv in ("U_index", "U_pointer", "V_index"):
            assert np.array_equal(got[lv], getattr(want, lv)), (plane, lv)
