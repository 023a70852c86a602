"""Fine nearest-neighbour calls whose long queries are finished by the whole block:
counts for every number of rounds, around the sorted calls and beyond what a block
keeps, near, far and invalid queries, answers beyond 32-bit distances, with and without
the prepared directory, one CGA and batches.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga

pytestmark = pytest.mark.gpu


def _world(bits, n, seed):
    rng = np.random.default_rng(seed)
    side = 1 << bits
    v = np.concatenate([rng.integers(0, side, size=(n, 3)),
                        rng.integers(0, min(side, 90), size=(n, 3)),
                        np.stack([np.full(n, side // 2), rng.integers(0, side, n),
                                  rng.integers(0, side, n)], -1)])
    pts = (v + 0.5).astype(np.float32)
    og = oracle.Grid(bits, 1.0, (0.0, 0.0, 0.0))
    return (cga.cga_build(torch.from_numpy(pts).cuda(), cga.make_grid(bits, 1.0, (0.0, 0.0, 0.0))),
            oracle.build(pts, og), og)


def _queries(bits, m):
    rng = np.random.default_rng(m)
    side = 1 << bits
    q = rng.uniform(0, side, size=(m, 3))
    q[::3] = rng.integers(0, 100, size=(len(q[::3]), 3))
    q[5::41] = rng.uniform(-4 * side, 5 * side, size=(len(q[5::41]), 3))
    q[7::97] = [np.nan, 1, 2]
    q[11::89, 0] = 3e5
    return q.astype(np.float32)


def _same(got, want):
    assert np.array_equal(got[1].cpu().numpy().view(np.uint64), want[1])
    assert np.array_equal(got[0].cpu().numpy().view(np.uint32), want[0])


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("bits,n", [(8, 700), (16, 700), (16, 1)])
@pytest.mark.parametrize("m", [1, 2, 150, 1824, 1825, 7296, 7300, 20_000, 117_000])
def test_counts(m, bits, n, prepared):
    a, o, og = _world(bits, n, 3)
    if prepared:
        cga.cga_nn_prepare(a)
    q = _queries(bits, m)
    _same(cga.cga_nn_query(a, torch.from_numpy(q).cuda()), oracle.nn_window(o, og, q))


def test_batch():
    worlds = [_world(b, n, b) for b, n in ((6, 300), (12, 900), (16, 500))]
    cga.cga_nn_prepare(worlds[1][0])
    qs = [_queries(b, m) for b, m in ((6, 4096), (12, 17), (16, 5000))]
    got = cga.cga_nn_query_batch([w[0] for w in worlds], [torch.from_numpy(q).cuda() for q in qs])
    for r, (a, o, og), q in zip(got, worlds, qs):
        _same(r, oracle.nn_window(o, og, q))
