"""Point builds that do not go by bins (dense grids: more than four blocks' worth of
points a bin) under every sort shape, alone and as batches in which one such cloud takes
the others, of up to 48-bit keys, along to the general sort.  Equality with the oracle's
arrays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga, synth

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")
DENSE = [(3, 300_001), (4, 600_003), (6, 2_200_000)]   # more than 2^bits * 32768 points


@pytest.fixture(params=[(8, 256), (8, 512), (9, 512)], ids=["8x256", "8x512", "9x512"])
def shape(request):
    t = dict(zip(("radix_bits", "sort_threads", "merge_half"), (*request.param, 1024)))

    def every_entry(value):
        for bits in range(1, 17):
            for nb in range(32):
                cga.tuning_set(bits, (1 << (nb - 1)) if nb else 0, value)

    every_entry(t)
    yield t
    every_entry(None)


def _grids(bits):
    return cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)


def _same(handle, want):
    got = handle.download()
    for lv in LEVELS:
        assert np.array_equal(got[lv], getattr(want, lv)), lv


@pytest.mark.parametrize("bits,n", DENSE)
def test_dense_grid(shape, bits, n):
    assert n >> bits > 32768
    g, og = _grids(bits)
    pts, xform = synth.uniform_cube(n, seed=n, lo=-0.02, extent=1.04), synth.rigid_xform(seed=n)
    d = torch.from_numpy(pts).cuda()
    _same(cga.cga_build(d, g), oracle.build(pts, og))
    _same(cga.cga_build(d, g, xform=xform), oracle.build(pts, og, xform=xform))


def test_batch_with_a_dense_grid(shape):
    spec = [(12, 70_000), (4, 600_003), (16, 50_001), (9, 4097), (14, 20_000), (11, 1), (15, 0)]
    pts = [synth.uniform_cube(n, seed=20 + i) for i, (_, n) in enumerate(spec)]
    got = cga.cga_build_batch([torch.from_numpy(p).cuda() for p in pts],
                              [_grids(b)[0] for b, _ in spec])
    for h, p, (b, _) in zip(got, pts, spec):
        _same(h, oracle.build(p, _grids(b)[1]))
