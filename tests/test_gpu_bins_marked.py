"""Builds by bins whose cloud is marked for the general sort as soon as its bins are
counted (one x slab of more than 2^20 points) while other bins hold enough points for
jobs and splits of their own: alone, with attributes and in batches, in scratch that
holds old data (the library never clears a block that it is given).  Equality with the
oracle's arrays."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")
MARK = 1_100_000  # points of the large slab: above 2^20


ALLOCATORS = []  # handles call back into theirs when they are collected


class OldData:
    """An allocator whose blocks are full of what another program left there."""

    def __init__(self, old):
        self.held = {}
        ALLOCATORS.append(self)

        @ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
        def alloc(ctx, size, stream):
            words = (int(size) + 3) // 4
            if old == "small":   # a number of keys that fits a block, wherever it is read
                t = torch.randint(1, 3000, (words,), dtype=torch.int32, device="cuda")
            else:
                t = torch.full((words,), -1, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            self.held[t.data_ptr()] = t
            return t.data_ptr()

        @ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
        def free(ctx, p, stream):
            torch.cuda.synchronize()
            self.held.pop(p, None)

        self.arg = cga.Allocator(None, alloc, free)


def _cloud(kind, n, bits):
    rng = np.random.default_rng(7 * n + bits)
    side = 1 << bits
    v = rng.integers(0, side, size=(n, 3))
    v[:MARK, 0] = side // 2
    if kind == "second":   # the rest in another slab, which has to be split
        v[MARK:, 0] = side // 4
    return ((rng.permutation(v) + 0.5) / side).astype(np.float32)


def _grids(bits):
    return cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)


def _same(handle, want):
    got = handle.download()
    for lv in LEVELS:
        assert np.array_equal(got[lv], getattr(want, lv)), lv


@pytest.mark.parametrize("old", ["small", "ones"])
@pytest.mark.parametrize("bits", [10, 12, 16])
@pytest.mark.parametrize("kind,n", [("uniform", 3_000_000), ("second", MARK + 100_000)])
def test_alone(kind, n, bits, old):
    g, og = _grids(bits)
    pts = _cloud(kind, n, bits)
    mem = OldData(old)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), g, allocator=mem.arg)
    _same(a, oracle.build(pts, og))


@pytest.mark.parametrize("policy", ["average", "first"])
@pytest.mark.parametrize("bits", [12, 16])
def test_with_attributes(bits, policy):
    g, og = _grids(bits)
    n = MARK + 400_000
    pts = _cloud("uniform", n, bits)
    rows = np.random.default_rng(bits).integers(0, 256, size=(n, 3), dtype=np.uint8)
    mem = OldData("small")
    a = cga.cga_build_values(torch.from_numpy(pts).cuda(), torch.from_numpy(rows).cuda(), g,
                             policy=policy, allocator=mem.arg)
    want, want_rows = oracle.build_values(pts, rows, og, policy=policy)
    _same(a, want)
    assert np.array_equal(cga.cga_values(a).cpu().numpy(), want_rows)


@pytest.mark.parametrize("old", ["small", "ones"])
def test_in_a_batch(old):
    rng = np.random.default_rng(5)
    spec = [(50_000, 12), (MARK + 300_000, 12), (20_000, 16), (MARK + 200_000, 16), (9000, 10)]
    pts = [_cloud("second", n, b) if n > MARK else rng.random((n, 3), dtype=np.float32)
           for n, b in spec]
    mem = OldData(old)
    got = cga.cga_build_batch([torch.from_numpy(p).cuda() for p in pts],
                              [_grids(b)[0] for _, b in spec], allocator=mem.arg)
    for h, p, (_, b) in zip(got, pts, spec):
        _same(h, oracle.build(p, _grids(b)[1]))


@pytest.mark.parametrize("bits", [10, 12, 13, 16])
@pytest.mark.parametrize("n,zeros", [(600_000, 270_000), (3_000_000, 400_000), (2_000_000, 460_000),
                                     (700_000, 690_000)])
def test_many_points_in_one_voxel(n, zeros, bits):
    """More keys in one voxel's row than go by parts: a map of the row, or the mark."""
    g, og = _grids(bits)
    rng = np.random.default_rng(zeros + bits)
    v = rng.random((n, 3), dtype=np.float32)
    v[:zeros] = 0.625
    v[: zeros // 100, 2] = 0.626
    pts = rng.permutation(v)
    mem = OldData("small")
    a = cga.cga_build(torch.from_numpy(pts).cuda(), g, allocator=mem.arg)
    _same(a, oracle.build(pts, og))
    if n < 1_000_000:
        rows = rng.integers(0, 256, size=(n, 3), dtype=np.uint8)
        b = cga.cga_build_values(torch.from_numpy(pts).cuda(), torch.from_numpy(rows).cuda(), g,
                                 allocator=mem.arg)
        want, want_rows = oracle.build_values(pts, rows, og)
        _same(b, want)
        assert np.array_equal(cga.cga_values(b).cpu().numpy(), want_rows)
