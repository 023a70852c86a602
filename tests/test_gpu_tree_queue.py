"""The breadth-first tree search at its edges, against the oracle's exhaustive
search: queues that overflow (a shell of voxels at one distance from the
query), starts from the position table with one to four cells per axis (queries
at cell borders, on every grid width), and a tree without the table (an
allocator that has no room for it).  Whole numbers, so equality."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _grids(bits):
    return (cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)), oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0)))


def _check(a, pts, og, q):
    q = np.ascontiguousarray(q, np.float32)
    oi, od = oracle.nn_brute(oracle.build(pts, og), og, q)
    for qq, rep in ((q, 1), (np.tile(q, (-(-8192 // len(q)), 1)), -(-8192 // len(q)))):
        idx, d2 = cga.cga_nn_query(a, torch.from_numpy(qq).cuda())
        assert np.array_equal(d2.cpu().numpy().view(np.uint64), np.tile(od, rep))
        assert np.array_equal(idx.cpu().numpy().view(np.uint32), np.tile(oi, rep))


@pytest.mark.parametrize("bits,radius", [(8, 100.0), (10, 400.0), (12, 1500.0), (16, 30000.0)])
def test_shell_overflows_the_queue(bits, radius):
    rng = np.random.default_rng(bits)
    c = (1 << bits) / 2
    d = rng.normal(size=(20_000, 3))
    pts = (c + radius * d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    g, og = _grids(bits)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), g)
    cga.cga_nn_prepare(a, "tree")
    q = c + rng.normal(0, radius / 200, size=(300, 3))
    q[:20] = c
    _check(a, pts, og, q)


@pytest.mark.parametrize("bits", [3, 5, 6, 8, 9, 11, 12, 14, 16])
@pytest.mark.parametrize("n", [40, 5000])
def test_starts_from_the_position_table(bits, n):
    rng = np.random.default_rng(100 * bits + n)
    side = 1 << bits
    v = rng.integers(0, side, size=(n, 3))
    pts = (v + 0.5).astype(np.float32)
    g, og = _grids(bits)
    a = cga.cga_build(torch.from_numpy(pts).cuda(), g)
    cga.cga_nn_prepare(a, "tree")
    cell = rng.choice([4, 16, 64, 256], size=(600, 1))
    edge = (v[rng.integers(0, n, 600)] // cell) * cell + rng.integers(-2, 3, size=(600, 3))
    near = v[rng.integers(0, n, 600)] + rng.integers(-20, 21, size=(600, 3))
    _check(a, pts, og, np.concatenate([edge, near]) + 0.5)


def test_without_room_for_the_position_table():
    rng = np.random.default_rng(9)
    pts = (rng.integers(0, 4096, size=(6000, 3)) + 0.5).astype(np.float32)
    g, og = _grids(12)
    most, held = {"n": None}, {}

    @ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
    def alloc(ctx, n, stream):
        if most["n"] is not None and n >= most["n"]:
            most["n"] = None  # one refusal: the tree with its table
            return None
        t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    @ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    def free(ctx, p, stream):
        torch.cuda.synchronize()
        held.pop(p, None)

    a = cga.cga_build(torch.from_numpy(pts).cuda(), g, allocator=cga.Allocator(None, alloc, free))
    cga.cga_nn_prepare(a)          # x directory and column table
    most["n"] = 200_000            # the next large block is the tree's
    cga.cga_nn_prepare(a, "tree")
    assert most["n"] is None
    _check(a, pts, og, np.concatenate([pts[:300] + 3, rng.uniform(0, 4096, size=(500, 3))]))
    a.free()
