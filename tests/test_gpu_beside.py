"""Calls on one stream while a long kernel of another stream holds a place on the GPU:
they need no more of the chip at once than is free, so they end before it does."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2110_11616_gb300 import cga, synth

pytestmark = pytest.mark.gpu


def _ends_beside(call):
    """Whether call's work ends while a one-thread kernel of 0.4 s or more, started before
    it on another stream, still runs."""
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(mine):
        call()   # loads the kernels and fills the allocator's cache
        call()
    torch.cuda.synchronize()
    busy, done = torch.cuda.Event(), torch.cuda.Event()
    with torch.cuda.stream(other):
        torch.cuda._sleep(800_000_000)   # cycles, of at most 2070 MHz
        busy.record()
    time.sleep(0.02)
    with torch.cuda.stream(mine):
        kept = call()
        done.record()
    while not done.query() and not busy.query():
        time.sleep(0.001)
    ended = done.query() and not busy.query()
    torch.cuda.synchronize()
    del kept
    return ended


@pytest.mark.parametrize("n,bits", [(131_072, 16), (600_000, 12), (2_000_000, 12)])
def test_build(n, bits):
    g = cga.grid_from_box([0, 0, 0], 1.0, bits)
    pts = torch.from_numpy(synth.uniform_cube(n, seed=bits)).cuda()
    torch.cuda.synchronize()
    assert _ends_beside(lambda: cga.cga_build(pts, g))


def test_build_that_the_general_sort_takes_over():
    g = cga.grid_from_box([0, 0, 0], 1.0, 12)
    v = np.random.default_rng(1).random((1_500_000, 3), dtype=np.float32)
    v[:1_200_000, 0] = 0.4   # one x slab
    pts = torch.from_numpy(v).cuda()
    torch.cuda.synchronize()
    assert _ends_beside(lambda: cga.cga_build(pts, g))


@pytest.mark.parametrize("n,bits", [(60_000, 12), (2_000_000, 12)])
def test_kmeans(n, bits):
    pts = torch.from_numpy(synth.uniform_cube(n, seed=bits)).cuda()
    a = cga.cga_build(pts, cga.grid_from_box([0, 0, 0], 1.0, bits))
    u = a.info()["u"]
    torch.cuda.synchronize()
    assert _ends_beside(lambda: cga.cga_kmeans(a, 64, u=u))
