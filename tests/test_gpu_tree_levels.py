"""The fixed-point prefix sums on both sides of 1,048,576 points, where the block
sums need a second level of blocks: the same tree and midpoints as the oracle."""
import numpy as np
import pytest

import oracle
from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1048576, 1049601])
def test_tree_of_two_levels_of_block_sums(n):
    y = inputs.spread_embedding((np.arange(n) * 7919) % 37, 2, rho_hi=10.0)
    with HyperbolicTSNE(precision="fp32") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        g = t.get_tree()
    o = oracle.tree_export(y, 0, which=1)
    for k in ("depth", "prefix", "count", "first"):
        assert np.array_equal(g[k], o[k]), k
    assert np.all(np.abs(g["ycell"] - o["ycell"]) <= 4 * np.spacing(np.abs(o["ycell"])))
