"""The fine nearest-neighbour search in 32-bit distances and where it hands over to
64 bits: nearest voxels 65535 voxels off and around it, along one axis and along
three, equal distances, queries far outside the grid; with and without the prepared
directory.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _check(vox, q, prepared, bits=16):
    pts, q = (np.asarray(vox) + 0.5).astype(np.float32), np.asarray(q, np.float32)
    og = oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)))
    if prepared:
        cga.cga_nn_prepare(a)
    idx, d2 = cga.cga_nn_query(a, torch.from_numpy(q).cuda())
    oi, od = oracle.nn_brute(oracle.build(pts, og), og, q)
    assert np.array_equal(d2.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(idx.cpu().numpy().view(np.uint32), oi)


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("corner", [[0, 0, 0], [65535, 65535, 65535], [0, 65535, 30000]])
def test_hand_over(corner, prepared):
    steps = [0, 1, 46340, 46341, 65534, 65535, 65536, 65537, 92681, 131071, 1 << 20]
    q = [[corner[0] + (s if k & 1 else 0), corner[1] + (s if k & 2 else 0),
          corner[2] + (s if k & 4 else 0)] for s in steps for k in range(1, 8)]
    q += [[corner[0] - s, corner[1] - s, corner[2]] for s in steps]
    q += [[np.nan, 0, 0], [0, np.inf, 0], [3e9, -3e9, 1]]
    q = np.array(q, np.float64)
    _check([corner], q, prepared)
    _check([corner, [65535 - c for c in corner]], q, prepared)


@pytest.mark.parametrize("prepared", [False, True])
def test_ties_and_crowds(prepared):
    rng = np.random.default_rng(5)
    lattice = np.stack(np.meshgrid(*[np.arange(100, 160, 6)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pole = np.stack([np.full(300, 40), np.full(300, 41), np.arange(300) * 3], -1)
    vox = np.concatenate([lattice, pole, rng.integers(0, 65536, size=(500, 3))])
    q = np.concatenate([lattice[::7] + 3, pole[::11] + 1, rng.uniform(0, 300, size=(300, 3)),
                        rng.uniform(-9e4, 16e4, size=(300, 3))])
    _check(vox, q, prepared)
