"""Rows of a merge found along the walk over its voxels: inputs that share nothing,
everything and every other voxel, slabs and columns that only one of them has, several
slabs in one step, the first and last places of the grid, an empty input.  Geometry and
rows equal the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")


def _pair(kind, bits):
    side, rng = 1 << bits, np.random.default_rng(bits)
    ends = np.array([[0, 0, 0], [0, 0, side - 1], [0, side - 1, 0], [side - 1] * 3])
    v = np.concatenate([rng.integers(0, side, size=(3000, 3)),
                        rng.integers(0, min(side, 12), size=(2000, 3))])
    if kind == "apart":      # by slabs
        return v[v[:, 0] % 2 == 0], v[v[:, 0] % 2 == 1]
    if kind == "columns":    # by columns of shared slabs
        return v[v[:, 1] % 2 == 0], v[v[:, 1] % 2 == 1]
    if kind == "same":
        return v, v[::-1]
    if kind == "ends":       # the grid's corners against the rest
        return ends, v
    if kind == "empty":
        return v, v[:0]
    if kind == "column":     # one column against half of it, and its neighbours
        z = np.arange(side)
        c = np.stack([np.full(side, side // 2), np.full(side, side // 3), z], -1)
        return c, np.concatenate([c[::2], c + [0, 1, 0], c - [1, 0, 0]])
    return v[:3500], v[1500:]


@pytest.mark.parametrize("policy", ["base", "average"])
@pytest.mark.parametrize("bits", [3, 6, 10, 13, 16])
@pytest.mark.parametrize("kind", ["apart", "columns", "same", "ends", "empty", "column", "overlap"])
def test_rows(kind, bits, policy):
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    rng, hs, os_ = np.random.default_rng(1), [], []
    for v in _pair(kind, bits):
        pts = ((v + 0.5) / (1 << bits)).astype(np.float32)
        rows = rng.integers(0, 256, size=(len(v), 3), dtype=np.uint8)
        hs.append(cga.cga_build_values(torch.from_numpy(pts).cuda(), torch.from_numpy(rows).cuda(), g))
        os_.append(oracle.build_values(pts, rows, og))
    for i, j in ((0, 1), (1, 0)):
        m = cga.cga_merge_values(hs[i], hs[j], policy=policy)
        o, ov = oracle.merge_values(*os_[i], *os_[j], policy=policy)
        d = m.download()
        for lv in LEVELS:
            assert np.array_equal(d[lv], getattr(o, lv)), lv
        assert np.array_equal(cga.cga_values(m).cpu().numpy(), ov)
