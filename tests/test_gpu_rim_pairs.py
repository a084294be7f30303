"""Points so close to the rim that a cell's 1 - |y|^2 rounds to 0 in float32 mode
(its conformal factor is infinite): a cell that no point accepts has no part in
the sums, listed or counted."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE

pytestmark = pytest.mark.gpu


# one to five interactions a point: the sums take them four at a time
@pytest.mark.parametrize("n", [2, 3, 4, 5, 6])
def test_cluster_at_the_rim(n):
    a = 0.3 + 1e-11 * np.arange(n)
    y = (1.0 - 1e-11) * np.stack([np.cos(a), np.sin(a)], 1)
    with HyperbolicTSNE(precision="fp32") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        for depth in (-1, 0):
            t.set_walk_split(depth)
            g, z = t.grad(0.05)
            t.set_counters(True)
            g2, z2 = t.grad(0.05)
            assert t.get_counters()[0] == 0  # no cell accepted: exact pairs only
            t.set_counters(False)
            assert np.isfinite(g).all() and np.array_equal(g, g2) and z == z2, depth
