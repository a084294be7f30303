"""The key sort by ranks: on both sides of every tile-size boundary (512, 1024,
2048 and 4096 keys per tile) and of its limit, with many equal keys, the sorted
keys build the oracle's tree."""
import numpy as np
import pytest

import oracle
from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 63, 65, 511, 512, 513, 1025, 8192, 8193, 32768, 32769, 90000, 90001, 150000,
                               150001])
@pytest.mark.parametrize("ties", [False, True])
def test_tree_of_the_sorted_keys(n, ties):
    y = inputs.spread_embedding((np.arange(n) * 7919) % 37, n % 5, rho_hi=10.0)
    if ties and n > 2:  # every point three times, the copies far apart in index
        y = y[np.arange(n) % (n // 3 + 1)]
    with HyperbolicTSNE(precision="fp32") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        g = t.get_tree()
    o = oracle.tree_export(y, 0, which=1)
    for k in ("depth", "prefix", "count", "first"):
        assert np.array_equal(g[k], o[k]), k


@pytest.mark.parametrize("n", [2000, 4096])
def test_small_sorts_wait_for_nothing(n):
    """The wait test's limit applies to sorts of more than 4096 keys only."""
    y = inputs.spread_embedding(np.arange(n) % 37, 3, rho_hi=8.0)
    with HyperbolicTSNE(precision="fp32") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        g, _ = t.grad(0.5)
        t._check(t._lib.hts_set_wait_test(t._ctx, 8))
        h, _ = t.grad(0.5)
        t._check(t._lib.hts_set_wait_test(t._ctx, 0))
    assert np.array_equal(g, h)
