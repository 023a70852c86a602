"""Averages of a voxel that holds about 2^16 points, where a count and a sum no longer
fit one 32-bit word of k_bin_values, and about 257, where two sums no longer do: alone in
its column and beside voxels of one point, every channel count, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
ROWS = ((255, 255, 255, 255), (7, 0, 200, 128), (128, 128, 128, 1))


@pytest.mark.parametrize("bits", [12, 16])
@pytest.mark.parametrize("count", [257, 258, 65_000, 65_280, 65_281, 65_282, 65_400, 65_409,
                                   65_500, 65_535, 65_536, 65_793])
def test_crowded_voxel(count, bits):
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    side = 1 << bits
    rng = np.random.default_rng(count + bits)
    voxel = np.array([side // 3, side // 2, side // 4])
    for beside in (0, 3):   # voxels of one point in the crowded one's column
        rest = rng.integers(0, side, size=(1500, 3))
        rest[:, 0] = np.where(rest[:, 0] >> (bits - 4) == voxel[0] >> (bits - 4), 0, rest[:, 0])
        v = np.concatenate([np.broadcast_to(voxel, (count, 3)), rest] +
                           [voxel[None] + [0, 0, k + 1] for k in range(beside)])
        order = rng.permutation(len(v))
        pts = ((v[order] + 0.5) / side).astype(np.float32)
        d_pts = torch.from_numpy(pts).cuda()
        for row in ROWS:
            rows = np.concatenate([np.broadcast_to(np.array(row, np.uint8), (count, 4)),
                                   rng.integers(0, 256, size=(len(v) - count, 4), dtype=np.uint8)])
            rows = rows[order]
            for channels in (1, 2, 3, 4):
                r = np.ascontiguousarray(rows[:, :channels])
                a = cga.cga_build_values(d_pts, torch.from_numpy(r).cuda(), g, policy="average")
                want, want_rows = oracle.build_values(pts, r, og, policy="average")
                assert a.info()["u"] == want.u
                assert np.array_equal(cga.cga_values(a).cpu().numpy(), want_rows), (beside, row, channels)
