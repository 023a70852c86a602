"""Searches whose warps take their block's next query when they are free: query
counts around a block's and a wave's warps, with one query in a hundred far more
expensive than the rest.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
COUNTS = [1, 7, 8, 9, 31, 33, 1000, 7295, 7297, 9001]


def _world():
    rng = np.random.default_rng(12)
    pts = rng.random((4000, 3)).astype(np.float32) * np.float32([0.5, 0.5, 0.05])
    g, og = cga.grid_from_box([0, 0, 0], 1.0, 12), oracle.grid_from_box([0, 0, 0], 1.0, 12)
    return cga.cga_build(torch.from_numpy(pts).cuda(), g), oracle.build(pts, og), og


def _queries(m):
    rng = np.random.default_rng(m)
    q = rng.random((m, 3)).astype(np.float32) * np.float32([0.5, 0.5, 0.05])
    q[::100] += np.float32(0.45)
    return q


def _same(got, want):
    for g, w in zip(got, want):
        g = g.cpu().numpy()
        assert np.array_equal(g.view(np.uint32 if g.itemsize == 4 else np.uint64), w)


@pytest.mark.parametrize("m", COUNTS)
@pytest.mark.parametrize("prepare", [None, (), (3,), "tree"])
def test_nearest(m, prepare):
    a, o, og = _world()
    if prepare is not None:
        cga.cga_nn_prepare(a, prepare)
    q = _queries(m)
    _same(cga.cga_nn_query(a, torch.from_numpy(q).cuda()), oracle.nn_brute(o, og, q))


@pytest.mark.parametrize("m", COUNTS)
def test_k_nearest_and_radius(m):
    a, o, og = _world()
    cga.cga_nn_prepare(a)
    q = _queries(m)
    d = torch.from_numpy(q).cuda()
    _same(cga.cga_knn(a, d, 3), oracle.knn(o, og, q, 3))
    _same(cga.cga_knn(a, d[:99].contiguous(), 40), oracle.knn(o, og, q[:99], 40))
    _same(cga.cga_radius(a, d, 5000), oracle.radius(o, og, q, 5000))
