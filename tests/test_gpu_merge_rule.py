"""Merges whose partition comes from the size rule, at the sizes where the rule
changes its mind (150k points; four points per grid column; 3M points of a fine
grid) and on columns that only one input holds.  Equality with the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2110_11616_gb300 import cga, synth

pytestmark = pytest.mark.gpu
LEVELS = ("X_index", "X_pointer", "Y_index", "Y_pointer", "Z_index")


@pytest.mark.parametrize("bits,na,nb", [
    (10, 74_999, 75_000), (10, 75_000, 75_000), (8, 131_071, 131_072), (8, 131_072, 131_072),
    (14, 100, 149_901), (16, 1_499_999, 1_500_000), (16, 1_500_000, 1_500_000), (3, 5000, 1)])
def test_rule_edges(bits, na, nb):
    a, b = synth.uniform_cube(na, seed=na + bits), synth.uniform_cube(nb, seed=nb + 7)
    b = b * np.float32(0.7) + np.float32(0.2)
    g, og = cga.grid_from_box([0, 0, 0], 1.0, bits), oracle.grid_from_box([0, 0, 0], 1.0, bits)
    m = cga.cga_merge(cga.cga_build(torch.from_numpy(a).cuda(), g),
                      cga.cga_build(torch.from_numpy(b).cuda(), g))
    want, got = oracle.merge(oracle.build(a, og), oracle.build(b, og)), m.download()
    for lv in LEVELS:
        assert np.array_equal(got[lv], getattr(want, lv)), lv
