"""Tree searches that begin in the query's own brick: queries on stored voxels and beside
them, ties between the own brick's voxels and a neighbouring brick's (the smaller key wins
on either side), empty own cells at every level, queries outside the grid.  Equality with
the exhaustive search."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _check(vox, q, bits):
    pts, q = (np.asarray(vox) + 0.5).astype(np.float32), np.asarray(q, np.float32)
    og = oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)))
    cga.cga_nn_prepare(a, "tree")
    idx, d2 = cga.cga_nn_query(a, torch.from_numpy(q).cuda())
    oi, od = oracle.nn_brute(oracle.build(pts, og), og, q)
    assert np.array_equal(d2.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(idx.cpu().numpy().view(np.uint32), oi)


@pytest.mark.parametrize("bits", [3, 4, 5, 6, 8, 11, 14, 15, 16])
def test_on_and_beside_stored_voxels(bits):
    rng = np.random.default_rng(bits)
    side = 1 << bits
    vox = rng.integers(0, side, size=(400, 3))
    cube = np.stack(np.meshgrid(*[np.arange(min(side, 11))] * 3, indexing="ij"), -1).reshape(-1, 3)
    vox = np.concatenate([vox, cube + max(0, side // 2 - 5)])
    near = vox[rng.integers(0, len(vox), size=800)]
    q = np.concatenate([near + 0.5, near + rng.integers(-3, 4, size=near.shape) + 0.5,
                        rng.uniform(-side, 2 * side, size=(400, 3))])
    _check(vox, q, bits)


@pytest.mark.parametrize("bits", [5, 9, 12, 16])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_ties_across_a_brick_border(bits, axis):
    side = 1 << bits
    lo = side // 2          # a border of bricks and of every coarser cell below the root
    vox, q = [], []
    for d in (1, 2, 3):
        a, b = [lo + 7, lo + 9, lo + 5], [lo + 7, lo + 9, lo + 5]
        a[axis], b[axis] = lo - d, lo + d
        vox += [a, b]
        c = list(a)
        c[axis] = lo
        q.append(np.array(c) + 0.5)     # b in its brick, a in the one below: equal distances
        c[axis] = lo - 1
        q.append(np.array(c) + 0.5)
    for i in range(len(q)):
        _check(vox[:2 * (i // 2) + 2], q, bits)
        _check(vox[2 * (i // 2):2 * (i // 2) + 2], q, bits)
