"""Counting the walk's work does not change its results, in float64 neither (whose
counting walk adds in another order than the listed sums)."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


# one and several blocks that sum a chunk; a depth that was asked for (direct)
@pytest.mark.parametrize("form", ["exact", "paper"])
@pytest.mark.parametrize("n,depth", [(2049, -1), (20011, -1), (2049, 2)])
def test_counting_keeps_the_bits(n, depth, form):
    with HyperbolicTSNE(precision="fp64", grad_form=form) as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=9.0))
        t.set_walk_split(depth)
        g, z = t.grad(0.5)
        t.set_counters(True)
        g2, z2 = t.grad(0.5)
        assert t.get_counters()[3] >= n and t.get_counters()[1] > 0
    assert np.array_equal(g, g2) and z == z2


# The listed sums against the direct walk (depth 0): the same terms in another
# order, n 2^-53 of their sizes' sum at most.
@pytest.mark.parametrize("n", [1, 33, 64, 2049, 9729, 20001])
@pytest.mark.parametrize("rho,theta", [(0.0, 0.5), (12.0, 0.2), (9.0, 1.0)])
def test_listed_against_direct(n, rho, theta):
    y = inputs.initial_embedding(n, 3) if rho == 0.0 else inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=rho)
    if n >= 700:
        y[5:45] = y[5]  # one leaf of the deepest level holds 40 points
    with HyperbolicTSNE(precision="fp64") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(y)
        g, z = t.grad(theta)
        t.set_walk_split(0)
        g2, z2 = t.grad(theta)
    assert abs(z - z2) <= 1e-12 * abs(z2)
    assert np.linalg.norm(g - g2) <= 1e-12 * np.linalg.norm(g2) + 1e-300


@pytest.mark.parametrize("n,listed", [(262144, True), (262145, False)])
def test_limit_of_the_float64_lists(n, listed):
    with HyperbolicTSNE(precision="fp64") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(inputs.spread_embedding(np.arange(n) % 37, 3, rho_hi=9.0))
        g, z = t.grad(0.8)
        t.set_walk_split(0)
        g2, z2 = t.grad(0.8)
    assert np.array_equal(g, g2) is not listed
    assert abs(z - z2) <= n * 2.0 ** -53 * abs(z2)
    assert np.linalg.norm(g - g2) <= n * 2.0 ** -53 * np.linalg.norm(g2)
