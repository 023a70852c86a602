"""The build by bins where it can go wrong, against the oracle's arrays: counts
around a job's and a block's capacity, clouds that fill one bin or one slab
(split jobs, duplicates, and the general sort behind them), every grid width, and
batches in which only some clouds need the general sort.  Equality."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")


def _cloud(kind, n, bits):
    rng = np.random.default_rng(31 * n + bits)
    side = 1 << bits
    v = rng.integers(0, side, size=(n, 3))
    if kind == "dups":         # almost everything in one voxel
        v[rng.random(n) < 0.97] = [side // 3, side // 2, side // 5]
    elif kind == "wall":       # one slab
        v[:, 0] = side // 2
    elif kind == "walls":      # two slabs, a thin rest
        v[:, 0] = np.where(rng.random(n) < 0.6, side // 4, side - 1)
        v[: n // 20] = rng.integers(0, side, size=(n // 20, 3))
    elif kind == "column":     # one column
        v[:, :2] = [side - 1, 0]
    elif kind == "zeros":      # a tenth of the returns invalid, at one point
        v[rng.random(n) < 0.1] = 0
    elif kind == "pole":       # a few columns side by side
        v[:, 0] = side // 2
        v[:, 1] = side // 2 + rng.integers(0, min(side // 2, 6), size=n)
    elif kind == "corner":     # a small cube at the far corner
        v = side - 1 - rng.integers(0, min(side, 40), size=(n, 3))
    return ((v + 0.5) / side).astype(np.float32)


def _same(handle, want):
    got = handle.download()
    for lv in LEVELS:
        assert np.array_equal(got[lv], getattr(want, lv)), lv


@pytest.mark.parametrize("bits", [1, 4, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16])
@pytest.mark.parametrize("kind", ["uniform", "dups", "wall", "walls", "column", "corner"])
def test_kinds_and_widths(kind, bits):
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    for n in (3000, 50_000):
        pts = _cloud(kind, n, bits)
        _same(cga.cga_build(torch.from_numpy(pts).cuda(), g), oracle.build(pts, og))


@pytest.mark.parametrize("n", [1, 2, 31, 511, 512, 513, 2047, 2049, 4095, 4096, 4097, 8191, 8192,
                               8193, 16_385])
@pytest.mark.parametrize("bits", [10, 12, 16])
def test_counts(n, bits):
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    for kind in ("uniform", "wall"):
        pts = _cloud(kind, n, bits)
        _same(cga.cga_build(torch.from_numpy(pts).cuda(), g), oracle.build(pts, og))


@pytest.mark.parametrize("kind,n,bits", [("wall", 400_000, 12), ("wall", 400_000, 16),
                                         ("wall", 1_200_000, 12), ("wall", 1_100_000, 15),
                                         ("walls", 500_000, 13), ("dups", 1_000_000, 12),
                                         ("corner", 300_000, 15), ("uniform", 1_500_000, 12),
                                         ("zeros", 131_072, 16), ("zeros", 1_200_000, 13),
                                         ("pole", 120_000, 12), ("pole", 120_000, 14),
                                         ("pole", 120_000, 16), ("dups", 120_000, 16),
                                         ("dups", 120_000, 10), ("dups", 60_000, 15),
                                         ("uniform", 700_000, 16)])
def test_large_skew(kind, n, bits):
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    pts = _cloud(kind, n, bits)
    for _ in range(2):
        _same(cga.cga_build(torch.from_numpy(pts).cuda(), g), oracle.build(pts, og))


def test_batch_where_some_clouds_need_the_general_sort():
    spec = [("uniform", 60_000, 12), ("wall", 1_200_000, 12), ("uniform", 0, 10), ("dups", 300_000, 16),
            ("wall", 250_000, 16), ("uniform", 1, 3), ("walls", 90_000, 14)]
    pts = [_cloud(*s) if s[1] else np.zeros((0, 3), np.float32) for s in spec]
    grids = [cga.grid_from_box([0, 0, 0], 1.0, s[2]) for s in spec]
    got = cga.cga_build_batch([torch.from_numpy(p).cuda() for p in pts], grids)
    for h, p, s in zip(got, pts, spec):
        _same(h, oracle.build(p, oracle.grid_from_box([0, 0, 0], 1.0, s[2])))


def test_non_finite_point_is_reported():
    for kind in ("uniform", "wall"):
        pts = _cloud(kind, 300_000, 12)
        pts[12345, 1] = np.nan
        a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, 12))
        assert a.status() == cga.ERR_NONFINITE
