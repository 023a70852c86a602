"""k-means by cells (k_kmcells.cu) against the oracle's per-voxel passes: every
grid width, clouds that fill one cell (several chunks), one voxel per cell,
symmetric lattices whose voxels tie between centres, and runs cut short.  Whole
numbers, so equality."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _cloud(kind, n, bits):
    rng = np.random.default_rng(17 * n + bits)
    side = 1 << bits
    if kind == "uniform":
        v = rng.integers(0, side, size=(n, 3))
    elif kind == "corner":      # everything in one small corner of the grid
        v = rng.integers(0, min(side, 24), size=(n, 3)) + (side - min(side, 24))
    elif kind == "clusters":    # two dense balls far apart, a few strays
        c = rng.integers(0, 2, size=(n, 1)) * (side * 3 // 4)
        v = c + rng.integers(0, max(side // 64, 2), size=(n, 3))
        v[: n // 50] = rng.integers(0, side, size=(n // 50, 3))
    else:                       # a full lattice: ties on every bisecting plane
        k = min(side, max(2, round(n ** (1 / 3))))
        v = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return ((v + 0.5) / side).astype(np.float32)


@pytest.mark.parametrize("max_iter", [1, 2, 64])
@pytest.mark.parametrize("kind,n,bits", [
    ("uniform", 1, 1), ("uniform", 7, 2), ("lattice", 64, 3), ("lattice", 32768, 7),
    ("lattice", 20000, 10), ("uniform", 3000, 9), ("uniform", 40_000, 12), ("uniform", 20_000, 16),
    ("corner", 30_000, 10), ("corner", 30_000, 16), ("clusters", 60_000, 12),
    ("clusters", 60_000, 16)])
def test_matches_the_oracle(kind, n, bits, max_iter):
    pts = _cloud(kind, n, bits)
    og = oracle.grid_from_box([0, 0, 0], 1.0, bits)
    o = oracle.build(pts, og)
    want = oracle.kmeans(o, max_iter)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, bits))
    lab, cen, cnt, it = cga.cga_kmeans(a, max_iter)
    assert int(it.item()) == want[3]
    assert np.array_equal(lab.cpu().numpy(), want[0])
    assert np.array_equal(cen.cpu().numpy(), want[1])
    assert np.array_equal(cnt.cpu().numpy().astype(np.int64), np.asarray(want[2]).astype(np.int64))


def test_without_room_for_the_cells():
    """An allocator that refuses the large block still gets its answer."""
    import ctypes
    pts = _cloud("uniform", 5000, 10)
    og = oracle.grid_from_box([0, 0, 0], 1.0, 10)
    want = oracle.kmeans(oracle.build(pts, og), 64)
    refuse = {"on": False}
    held = {}

    @ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
    def alloc(ctx, n, stream):
        if refuse["on"] and n > 4096:
            return None
        t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    @ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    def free(ctx, p, stream):
        torch.cuda.synchronize()
        held.pop(p, None)

    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, 10),
                      allocator=cga.Allocator(None, alloc, free))
    torch.cuda.synchronize()
    refuse["on"] = True
    lab, cen, cnt, it = cga.cga_kmeans(a, 64)
    assert int(it.item()) == want[3]
    assert np.array_equal(lab.cpu().numpy(), want[0]) and np.array_equal(cen.cpu().numpy(), want[1])
    del lab, cen, cnt, it
    a.free()
