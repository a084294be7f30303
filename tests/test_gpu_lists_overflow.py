"""Interaction lists that do not fit their pages, in float64: a tight cluster with
outliers at nested distances is cut into a few units only (a cut stops at eight
ancestors), so that at theta = 0.005 the pools of two chunks run out (9,728
points: 48 of the 256).  Their chunks are walked directly by one of the two
blocks that sum a chunk; the other adds nothing."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu

N, THETA = 9728, 0.005


def nested_cluster():
    rng = np.random.default_rng(0)
    c = np.array([0.31, 0.17])
    y = c + 1e-6 * rng.standard_normal((N, 2))
    k = np.arange(40)
    a = rng.uniform(0.0, 2.0 * np.pi, 40)
    y[:40] = c + (0.5 * 2.0 ** (-0.5 * k))[:, None] * np.stack([np.cos(a), np.sin(a)], 1)
    return y


# The same terms in another order: off by n 2^-53 (1.1e-12) of the sum of their
# sizes at most, and that is within 8 times the result here (the terms of a
# point grow with the distance and mostly point away from the cluster).
TOL = 1e-11


@pytest.mark.parametrize("form", ["exact", "paper"])
def test_overflow_after_a_call_that_left_sums(form):
    with HyperbolicTSNE(precision="fp64", grad_form=form) as t:
        t.set_P(np.zeros(N + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(inputs.spread_embedding(np.arange(N) % 7, 3, rho_hi=9.0))
        t.grad(0.5)
        t.set_Y(nested_cluster())
        g, z = t.grad(THETA)
        t.set_walk_split(0)  # the direct walk
        g2, z2 = t.grad(THETA)
    assert abs(z - z2) <= TOL * abs(z2)
    assert np.linalg.norm(g - g2) <= TOL * np.linalg.norm(g2)


def test_overflow_gives_the_same_bits_again():
    """131,071 points at theta = 0.2: pools of 16 chunks run out, and which chunk
    finds its pool empty depends on timing."""
    n = 131071
    with HyperbolicTSNE(precision="fp64") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(inputs.spread_embedding(np.arange(n) % 20, 3, rho_hi=6.0))
        g, z = t.grad(0.2)
        for _ in range(5):
            h, y = t.grad(0.2)
            assert np.array_equal(g, h) and z == y
