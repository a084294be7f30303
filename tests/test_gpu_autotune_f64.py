"""Autotuning a float64 context keeps the listed walk where it is the faster one
(N = 3001: about 0.4 ms against 0.8 ms and more at every cut depth), with or
without counting: the tuned context gives the untuned one's bits, which the
direct walk's order of sums does not."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counted", [False, True])
def test_autotune_keeps_the_listed_walk(counted):
    n = 3001
    with HyperbolicTSNE(precision="fp64") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(inputs.spread_embedding(np.arange(n) % 7, 5, rho_hi=9.0))
        g, z = t.grad(0.5)
        t.set_counters(counted)
        assert t.autotune(0.5, 3)[0] == 256  # (a listed walk has no block size to tune)
        t.set_counters(False)
        g2, z2 = t.grad(0.5)
        assert np.array_equal(g, g2) and z == z2
        t.set_walk_split(1)
        g2, z2 = t.grad(0.5)
        assert not np.array_equal(g, g2)
