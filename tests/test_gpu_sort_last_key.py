"""A point's key can be 2^64 - 1, the value that fills the last sorted tile: the
outermost point of the 64th embedding at an angle that rounds to a full turn
(the end of a circle laid out by linspace).  Wherever it lies in its tile, once
or several times, the sorted keys build the oracle's trees."""
import numpy as np
import pytest

import oracle
from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu

TOP = np.uint64(2 ** 64 - 1)


# tiles of 512 (one and several), 1024, 2048 and 4096 keys, and the radix sort
@pytest.mark.parametrize("n", [500, 2000, 20000, 60000, 131072, 150001])
@pytest.mark.parametrize("where", ["first", "middle", "last", "thrice"])
def test_last_key_is_a_point(n, where):
    off = np.concatenate([5 * np.arange(64), [n]])
    y = inputs.spread_embedding(np.arange(n) % 37, 3, rho_hi=8.0)
    m = n - off[63]
    at = off[63] + {"first": [0], "middle": [m // 2], "last": [m - 1], "thrice": [7, m // 3, m - 40]}[where]
    y[at] = [0.9999 * np.cos(2.0 * np.pi), 0.9999 * np.sin(2.0 * np.pi)]  # (y = -2.4e-16)
    y[off[63]:] *= np.minimum(1.0, 0.9999 / np.linalg.norm(y[off[63]:], axis=1))[:, None]
    with HyperbolicTSNE(precision="fp32") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        t.set_segments(off)
        keys, _ = t.get_keys()
        assert np.array_equal(np.flatnonzero(keys == TOP), at)
        g = t.get_tree()
    pos = 0
    for s in range(64):
        o = oracle.tree_export(y[off[s]:off[s + 1]], 0, which=1)
        sl = slice(pos, pos + len(o["depth"]))
        for k in ("depth", "prefix", "count"):
            assert np.array_equal(g[k][sl], o[k]), (s, k)
        assert np.array_equal(g["first"][sl], np.where(o["first"] >= 0, o["first"] + off[s], -1)), s
        pos += len(o["depth"])
    assert pos == len(g["depth"])
