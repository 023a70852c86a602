"""Builds on coarse grids on both sides of the rule that sends them by bins or to the
general sort, alone, in batches on either side of half the points, and with attributes.
Equality with the oracle's arrays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")


def _cloud(n, bits, seed):
    rng = np.random.default_rng(seed)
    v = rng.integers(0, 1 << bits, size=(n, 3))
    v[: n // 3] = v[: n // 3] % max(1, (1 << bits) // 7)   # a crowded corner
    return ((v + 0.5) / (1 << bits)).astype(np.float32)


def _grids(bits):
    return cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)


def _same(handle, want):
    got = handle.download()
    for lv in LEVELS:
        assert np.array_equal(got[lv], getattr(want, lv)), lv


@pytest.mark.parametrize("bits", [1, 2, 3, 5, 6, 7, 8])
def test_around_the_rule(bits):
    g, og = _grids(bits)
    edges = [512 << bits, 8192 << bits]
    for n in sorted({e + d for e in edges for d in (-1, 0)}):
        if n > 2_100_000:
            continue
        pts = _cloud(n, bits, n)
        _same(cga.cga_build(torch.from_numpy(pts).cuda(), g), oracle.build(pts, og))


@pytest.mark.parametrize("bits", [4, 7])
def test_with_attributes(bits):
    g, og = _grids(bits)
    n = (512 << bits) + 777
    pts = _cloud(n, bits, n)
    rows = np.random.default_rng(n).integers(0, 256, size=(n, 3), dtype=np.uint8)
    a = cga.cga_build_values(torch.from_numpy(pts).cuda(), torch.from_numpy(rows).cuda(), g)
    want, want_rows = oracle.build_values(pts, rows, og)
    _same(a, want)
    assert np.array_equal(cga.cga_values(a).cpu().numpy(), want_rows)


@pytest.mark.parametrize("fine", [30_000, 200_000])
def test_batches(fine):
    spec = [(6, 90_000), (12, fine), (16, 5000), (3, 100)]
    pts = [_cloud(n, b, n) for b, n in spec]
    got = cga.cga_build_batch([torch.from_numpy(p).cuda() for p in pts], [_grids(b)[0] for b, _ in spec])
    for h, p, (b, _) in zip(got, pts, spec):
        _same(h, oracle.build(p, _grids(b)[1]))
