"""k-means runs of few passes, which go voxel by voxel: the oracle's results on both
sides of the rule, and no tables of cells where one or two passes cannot pay for them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga, synth

pytestmark = pytest.mark.gpu
BY_CELLS = 7  # launches by cells, whatever the passes


@pytest.mark.parametrize("n,bits", [(1, 16), (100, 10), (1000, 16), (3000, 12), (10_000, 10),
                                    (60_000, 16), (60_000, 9)])
def test_both_sides_of_the_rule(n, bits):
    pts = synth.uniform_cube(n, seed=n + bits)
    o = oracle.build(pts, oracle.grid_from_box([0, 0, 0], 1.0, bits))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.grid_from_box([0, 0, 0], 1.0, bits))
    u = a.info()["u"]
    by_cells = []
    for max_iter in (1, 2, 3, 4, 5, 7, 9, 12):
        before = cga.kernel_launches()
        lab, cen, cnt, it = cga.cga_kmeans(a, max_iter, u=u)
        launches = cga.kernel_launches() - before
        assert launches in (BY_CELLS, 3 + 2 * max_iter)
        by_cells.append(max_iter != 2 and launches == BY_CELLS)
        want = oracle.kmeans(o, max_iter)
        assert int(it.item()) == want[3]
        assert np.array_equal(lab.cpu().numpy(), want[0])
        assert np.array_equal(cen.cpu().numpy(), want[1])
        assert np.array_equal(cnt.cpu().numpy().astype(np.int64),
                              np.asarray(want[2]).astype(np.int64))
    assert not by_cells[0] and by_cells[-1]   # (2 passes: as many launches either way)
