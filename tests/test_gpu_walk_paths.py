"""The ways a float32 walk is run give the same bits: the counting walk visits
and adds one interaction at a time with the general pair term; small problems
list their interactions first and sum them by blocks; embeddings close to the
origin take the pair term's series without the logarithm."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


def embedding(n, rho, buckets):
    y = inputs.initial_embedding(n, 3) if rho == 0.0 else inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=rho)
    if buckets and n >= 700:
        y[5:45] = y[5]      # one leaf of the deepest level holds 40 points
        y[600:633] = y[600]
    return y


def both(y, theta, depth, split_rule="equal_length", grad_form="exact", offsets=None):
    n = len(y)
    with HyperbolicTSNE(split_rule=split_rule, grad_form=grad_form) as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        if offsets is not None:
            t.set_segments(offsets)
        t.set_walk_split(depth)
        g, z = t.grad(theta)
        z = t.segment_Z() if offsets is not None else z
        t.set_counters(True)
        g2, z2 = t.grad(theta)
        z2 = t.segment_Z() if offsets is not None else z2
    return g, z, g2, z2


# one point; one and two 32-point chunks and their remainders; both sides of
# the listing's size limit (32,768)
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 2049, 32768, 32769])
@pytest.mark.parametrize("rho,theta", [(0.0, 0.5), (9.0, 0.2), (9.0, 1.0)])
def test_same_bits_as_the_counting_walk(n, rho, theta):
    y = embedding(n, rho, buckets=rho > 0)
    for depth in (-1, 0, 2):
        g, z, g2, z2 = both(y, theta, depth)
        assert np.array_equal(g, g2) and z == z2, depth


@pytest.mark.parametrize("rule,form", [("equal_area", "exact"), ("equal_length", "paper")])
@pytest.mark.parametrize("n,rho", [(3000, 0.0), (3000, 6.0), (40000, 0.0)])
def test_same_bits_options(rule, form, n, rho):
    g, z, g2, z2 = both(embedding(n, rho, buckets=False), 0.5, -1, rule, form)
    assert np.array_equal(g, g2) and z == z2


def test_same_bits_segments_near_and_far():
    """Segments at the origin and spread ones share chunks: a chunk takes the
    series only if all of its segments allow it."""
    parts = [embedding(k, r, False) for k, r in ((45, 0.0), (37, 9.0), (1, 0.0), (900, 0.0), (700, 11.0), (64, 0.0))]
    off = np.concatenate([[0], np.cumsum([len(p) for p in parts])])
    g, z, g2, z2 = both(np.concatenate(parts), 0.5, -1, offsets=off)
    assert np.array_equal(g, g2) and np.array_equal(z, z2)


def test_lists_that_do_not_fit():
    """theta = 0.01 accepts next to nothing: every chunk lists about n
    interactions, more than its pool holds, and is walked directly."""
    g, z, g2, z2 = both(embedding(32768, 8.0, False), 0.01, 0)
    assert np.array_equal(g, g2) and z == z2


# float64: the counting walk is the direct one (a ring per warp), the other
# listed up to 262,144 points (several blocks per chunk below 304 chunks).
# The same terms in another order: n 2^-53 of the terms' sum at most.
@pytest.mark.parametrize("n", [1, 33, 64, 2049, 9729, 20001])
@pytest.mark.parametrize("rho,theta", [(0.0, 0.5), (12.0, 0.2), (9.0, 1.0)])
def test_float64_listed_and_direct(n, rho, theta):
    y = embedding(n, rho, buckets=rho > 0)
    with HyperbolicTSNE(precision="fp64") as t:
        t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32))
        t.set_Y(y)
        g, z = t.grad(theta)
        t.set_counters(True)
        g2, z2 = t.grad(theta)
        accepted = t.get_counters()[:2].copy()
        t.set_counters(False)
        t.set_counters(True)
        t.set_walk_split(1)
        t.grad(theta)
        assert np.array_equal(t.get_counters()[:2], accepted)  # the same interactions, cut or not
    assert abs(z - z2) <= 1e-12 * abs(z2)
    assert np.linalg.norm(g - g2) <= 1e-12 * np.linalg.norm(g2) + 1e-300
