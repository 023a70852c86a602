"""Merge tiles of several cuts: inputs whose columns are shared, interleaved, apart or
crowded at one end (so that tiles take their most columns from one side), one to dozens
of voxels a column, every partition, sizes around the cuts and a wave of tiles, and a
batch of such pairs.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")
BITS = 12


def _side(cols, per, rng):
    """Voxels of the columns (key x << 12 | y), 1 to per of each."""
    c = np.repeat(cols, rng.integers(1, per + 1, size=len(cols)))
    z = rng.integers(0, 1 << BITS, size=len(c))
    return ((np.stack([c >> BITS, c & 0xFFF, z], -1) + 0.5) / (1 << BITS)).astype(np.float32)


def _pair(kind, n, per):
    rng = np.random.default_rng(n + per)
    c = np.sort(rng.choice(1 << 22, size=2 * n, replace=False))
    a, b = {"same": (c[:n], c[:n]), "mixed": (c[0::2], c[1::2]), "apart": (c[:n], c[n:]),
            "few": (c, c[:: max(1, n // 3)]),
            "ends": (c[:n], np.concatenate([c[:2], c[n - 5:]]))}[kind]
    return _side(a, per, rng), _side(b, per, rng)


def _same(h, o):
    d = h.download()
    for lv in LEVELS:
        assert np.array_equal(d[lv], getattr(o, lv)), lv


def _grids():
    return cga.grid_from_box([0, 0, 0], 1.0, BITS), oracle.grid_from_box([0, 0, 0], 1.0, BITS)


@pytest.mark.parametrize("half", [512, 1024, 2048])
@pytest.mark.parametrize("per", [1, 5, 60])
@pytest.mark.parametrize("kind", ["same", "mixed", "apart", "few", "ends"])
def test_pairs(kind, per, half):
    g, og = _grids()
    try:
        for n in (1, 128, 129, 1023, 1025, 7 * 512, 40_000):
            pts = _pair(kind, n, per if n < 40_000 else min(per, 12))
            a, b = (cga.cga_build(torch.from_numpy(p).cuda(), g) for p in pts)
            cap = len(pts[0]) + len(pts[1])
            cga.tuning_set(BITS, cap, {"radix_bits": 8, "sort_threads": 512, "merge_half": half})
            _same(cga.cga_merge(a, b), oracle.merge(*(oracle.build(p, og) for p in pts)))
            cga.tuning_set(BITS, cap, None)
    finally:
        for k in range(1, 24):
            cga.tuning_set(BITS, 1 << k, None)


def test_batch():
    g, og = _grids()
    pairs = [_pair("mixed", 30_000, 3), _pair("same", 9000, 40), _pair("few", 2, 1),
             _pair("apart", 20_000, 1)]
    hs = [[cga.cga_build(torch.from_numpy(p).cuda(), g) for p in pair] for pair in pairs]
    got = cga.cga_merge_batch([h[0] for h in hs], [h[1] for h in hs])
    for m, pair in zip(got, pairs):
        _same(m, oracle.merge(*(oracle.build(p, og) for p in pair)))
