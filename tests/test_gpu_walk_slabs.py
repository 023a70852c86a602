"""The walk over CGA positions where many slabs open within one of its steps: from one
voxel a slab to hundreds, counts around the 32 slabs that are loaded at once and the 128
positions of a step, slabs ending with a step.  Decode against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slabs", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 500, 4000])
@pytest.mark.parametrize("per", [1, 2, 3, 4, 5, 31, 128, 130])
def test_slabs_of_equal_size(slabs, per):
    bits = 12
    x = np.repeat(np.arange(slabs) + 7, per)
    y = np.tile(np.arange(per) // 2, slabs)
    z = np.tile(np.arange(per) * 3, slabs)
    pts = (np.stack([x, y, z], -1) + 0.5).astype(np.float32)
    want = oracle.build(pts, oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0)))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)))
    assert np.array_equal(cga.cga_decode(a).cpu().numpy().astype(np.uint32), oracle.decode(want))


def test_slabs_of_any_size():
    bits = 16
    rng = np.random.default_rng(4)
    sizes = rng.choice([1, 1, 1, 2, 7, 40, 129, 700], size=3000)
    x = np.repeat(np.sort(rng.choice(1 << bits, size=len(sizes), replace=False)), sizes)
    pts = (np.stack([x, rng.integers(0, 9, len(x)), rng.integers(0, 1 << bits, len(x))], -1) +
           0.5).astype(np.float32)
    want = oracle.build(pts, oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0)))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)))
    assert np.array_equal(cga.cga_decode(a).cpu().numpy().astype(np.uint32), oracle.decode(want))
    for plane in ("xz", "yz"):
        got, o = cga.cga_project(a, plane).download(), oracle.project(want, plane)
        for lv in ("U_index", "U_pointer", "V_index"):
            assert np.array_equal(got[lv], getattr(o, lv)), (plane, lv)
