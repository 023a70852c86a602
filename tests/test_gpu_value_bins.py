"""The Value array summed along with a build by bins, against the oracle byte for
byte: every channel count and policy, one and several jobs, voxels of more points
than 16-bit sums hold, split bins and their rows, clouds that the general sort takes
over, unaligned rows, and an allocator that refuses any one of the blocks."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")


def _cloud(kind, n, bits, channels):
    rng = np.random.default_rng(13 * n + bits + channels)
    side = 1 << bits
    v = rng.integers(0, side, size=(n, 3))
    if kind == "dups":       # nearly everything in one voxel
        v[rng.random(n) < 0.97] = [side // 3, side // 2, side // 5]
    elif kind == "few":      # a dozen points a voxel
        v = rng.integers(0, max(2, round((n / 12) ** (1 / 3))), size=(n, 3)) % side
    elif kind == "wall":     # one slab
        v[:, 0] = side // 2
    elif kind == "pole":     # a few columns
        v[:, 0] = side // 2
        v[:, 1] = side // 2 + rng.integers(0, 5, size=n)
    rows = rng.integers(0, 256, size=(n, channels), dtype=np.uint8)
    if n > 3:
        rows[rng.random(n) < 0.5] = 255
    return ((v + 0.5) / side).astype(np.float32), rows


def _same(got, want, rows):
    d = got.download()
    for lv in LEVELS:
        assert np.array_equal(d[lv], getattr(want, lv)), lv
    assert np.array_equal(cga.cga_values(got).cpu().numpy(), rows)


def _check(kind, n, bits, channels, policy, skip=0, allocator="torch"):
    pts, rows = _cloud(kind, n, bits, channels)
    # rows that start `skip` bytes into their block
    block = torch.zeros(skip + rows.size, dtype=torch.uint8, device="cuda")
    block[skip:] = torch.from_numpy(rows.reshape(-1)).cuda()
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    a = cga.cga_build_values(torch.from_numpy(pts).cuda(), block[skip:].view(n, channels), g,
                             policy=policy, allocator=allocator)
    _same(a, *oracle.build_values(pts, rows, og, policy=policy))


@pytest.mark.parametrize("policy", ["average", "first"])
@pytest.mark.parametrize("channels", [1, 2, 3, 4])
@pytest.mark.parametrize("kind,n,bits", [
    ("uniform", 3, 16), ("uniform", 5000, 10), ("uniform", 60_001, 16), ("uniform", 60_002, 12),
    ("few", 70_000, 13), ("few", 90_000, 16), ("dups", 9000, 12), ("dups", 70_003, 16),
    ("wall", 50_000, 11), ("pole", 100_000, 12), ("pole", 60_000, 16)])
def test_kinds(kind, n, bits, channels, policy):
    _check(kind, n, bits, channels, policy)


@pytest.mark.parametrize("policy", ["average", "first"])
@pytest.mark.parametrize("kind,n,bits", [("dups", 400_000, 16), ("wall", 1_200_000, 12),
                                         ("wall", 300_000, 16), ("uniform", 1_400_000, 12)])
def test_large_skew(kind, n, bits, policy):
    _check(kind, n, bits, 3, policy)


@pytest.mark.parametrize("skip", [1, 2, 3])
@pytest.mark.parametrize("channels", [1, 2, 3, 4])
def test_unaligned_rows(channels, skip):
    _check("few", 20_001, 12, channels, "average", skip)


@pytest.mark.parametrize("refused", [1, 2, 3, 4])
def test_any_block_refused_once(refused):
    calls, held = [0], {}

    @ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
    def alloc(ctx, size, stream):
        calls[0] += 1
        if calls[0] == refused:
            return None
        t = torch.empty(int(size), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    @ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    def free(ctx, p, stream):
        torch.cuda.synchronize()
        held.pop(p, None)

    for policy in ("average", "first"):
        calls[0] = 0
        _check("uniform", 30_000, 12, 3, policy, allocator=cga.Allocator(None, alloc, free))
        assert calls[0] > refused
    assert not held
