"""Both arithmetic forms of the radius and k-NN searches where one hands over to
the other: radii around 2^31, queries whose neighbours lie 65535 voxels off and
more, clouds with fewer voxels than k, columns around the length that is measured
voxel by voxel, slabs with more hits than a lane keeps; with and without the
prepared directory.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _setup(bits, vox, prepared):
    pts = (np.asarray(vox) + 0.5).astype(np.float32)
    og = oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0))
    a = cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0)))
    if prepared:
        cga.cga_nn_prepare(a)
    return a, oracle.build(pts, og), og


def _columns(bits, heights):
    v = [[3 + 2 * i, 5, z] for i, h in enumerate(heights) for z in range(h)]
    v += [[3, 5 + 3 * j, 2 * j] for j in range(1, 12)]
    return np.array(v)


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("k", [1, 8, 32, 33, 400])
def test_knn_near_and_far(k, prepared):
    rng = np.random.default_rng(k)
    vox = np.concatenate([rng.integers(0, 65536, size=(150, 3)), rng.integers(0, 40, size=(900, 3)),
                          rng.integers(65500, 65536, size=(50, 3))])
    a, o, og = _setup(16, vox, prepared)
    q = np.concatenate([rng.uniform(0, 40, size=(60, 3)), rng.uniform(0, 65536, size=(60, 3)),
                        rng.uniform(-3e5, 3e5, size=(60, 3)), [[-65535.5] * 3, [65536.5, 0.5, 0.5],
                        [np.nan, 0, 0], [1e9, -1e9, 5]]]).astype(np.float32)
    gi, gd = cga.cga_knn(a, torch.from_numpy(q).cuda(), k)
    oi, od = oracle.knn(o, og, q, k)
    assert np.array_equal(gd.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(gi.cpu().numpy().view(np.uint32), oi)


@pytest.mark.parametrize("k", [5, 32, 64])
def test_knn_of_fewer_voxels_than_k(k):
    a, o, og = _setup(16, [[1, 2, 3], [65535, 65535, 65535], [7, 7, 7]], True)
    q = np.array([[0, 0, 0], [-2e5, 0, 0], [65535, 0, 65535], [np.inf, 0, 0]], np.float32)
    gi, gd = cga.cga_knn(a, torch.from_numpy(q).cuda(), k)
    oi, od = oracle.knn(o, og, q, k)
    assert np.array_equal(gd.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(gi.cpu().numpy().view(np.uint32), oi)


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("r2", [0, 1, 9, 36, 400, (1 << 31) - 1, 1 << 31, 65535 ** 2 + 5, 1 << 34])
def test_radius_forms(r2, prepared):
    rng = np.random.default_rng(r2 % 1000)
    vox = np.concatenate([_columns(16, [1, 3, 4, 5, 6, 7, 9, 40]),
                          rng.integers(0, 65536, size=(40, 3))])
    a, o, og = _setup(16, vox, prepared)
    q = np.concatenate([vox[rng.integers(0, len(vox), 60)] + rng.integers(-4, 5, size=(60, 3)),
                        rng.uniform(-7e4, 1.4e5, size=(30, 3)),
                        [[-46341.0, 5.0, 2.0], [3.0, 5.0, -65536.0], [np.nan, 1, 1], [1e9, 5, 5]]])
    q = q.astype(np.float32)
    off, gi, gd = cga.cga_radius(a, torch.from_numpy(q).cuda(), r2)
    oo, oi, od = oracle.radius(o, og, q, r2)
    assert np.array_equal(off.cpu().numpy().view(np.uint64), oo)
    assert np.array_equal(gi.cpu().numpy().view(np.uint32), oi)
    assert np.array_equal(gd.cpu().numpy().view(np.uint64), od)
