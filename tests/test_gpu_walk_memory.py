"""The interaction lists are taken by the first call that walks a tree with them:
not by a context that only computes exact gradients, and not by batches, which
never list."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu

MB = 1 << 20


def free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def context(n, precision):
    t = HyperbolicTSNE(precision=precision)
    t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
    t.set_Y(inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=8.0))
    return t


# lists: 175 MB at 32,768 points, by the sizes of list_pages
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_lists_are_taken_by_the_first_listed_walk(precision):
    n = 32768
    with context(n, precision) as t:  # (kernels are loaded, pools warm)
        for theta in (0.0, 0.5):
            t.grad(theta)
    with context(n, precision) as t:
        f0 = free()
        t.grad(0.0)
        f1 = free()
        g, z = t.grad(0.5)
        f2 = free()
        g2, z2 = t.grad(0.5)
        assert free() == f2
        assert np.array_equal(g, g2) and z == z2
    assert f0 - f1 < 8 * MB and f1 - f2 > 160 * MB


def test_batches_take_no_lists():
    n = 32768
    for k in range(2):
        with context(n, "fp32") as t:
            t.set_segments(np.array([0, 5000, n]))
            f0 = free()
            t.grad(0.5)
            assert k == 0 or f0 - free() < 8 * MB


def test_tree_export_before_any_walk():
    n = 3000
    with context(n, "fp64") as t:
        a = t.get_tree()
        t.grad(0.5)
        b = t.get_tree()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
