"""Batches and pipelines of one small cloud among many empty ones: their tables do not
fit the scratch of a build by bins, so that the general sort runs, under every digit
width (with 9-bit digits 36-, 42- and 45-bit keys take other pass counts than with 8).
Equality with the oracle's arrays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga, synth

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")
EMPTY = 40


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


@pytest.mark.parametrize("bits", [9, 11, 12, 14, 15, 16])
def test_one_cloud_among_empty_ones(shape, bits):
    g, og = _grids(bits)
    n = 4096
    pts = synth.uniform_cube(n, seed=bits)
    xform = synth.rigid_xform(seed=50 + bits)
    want = oracle.build(pts, og)
    empty = torch.zeros((0, 3), dtype=torch.float32, device="cuda")
    at = EMPTY // 3
    clouds = [empty] * EMPTY
    clouds[at] = torch.from_numpy(pts).cuda()
    grids = [g] * EMPTY
    got = cga.cga_build_batch(clouds, grids)
    for i, h in enumerate(got):
        assert h.info()["u"] == (want.u if i == at else 0)
    _same(got[at], want)
    pipe = cga.Pipeline(clouds, grids, [xform] * EMPTY, [None] * EMPTY)
    pipe.run_graph()
    torch.cuda.synchronize()
    _same(pipe.view(at, "merged"), oracle.merge(want, oracle.build(pts, og, xform=xform)))
    pipe.free()
