"""A point that has diverged (a step that reported HTS_ENUMERIC left it not finite)
and the gradients of the points beside it."""
import numpy as np
import pytest

from paper_2401_13708_gb300 import HtsError, HyperbolicTSNE, inputs

pytestmark = pytest.mark.gpu


def diverged(precision, n, at, theta, offsets=None, split_rule="equal_length"):
    """A context whose point `at` is not finite after a step; its other points."""
    y = inputs.spread_embedding(np.arange(n) % 7, 3, rho_hi=6.0)
    t = HyperbolicTSNE(precision=precision, split_rule=split_rule)
    t.set_P(np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
    t.set_Y(y)
    if offsets is not None:
        t.set_segments(offsets)
    v = np.zeros((n, 2))
    v[at] = np.inf  # (the step to a point at infinity is not a number; one of NaN moves nothing)
    t.set_state(vel=v)
    with pytest.raises(HtsError):
        t.step(1, theta, 1.0, 0.0, 1.0)
    y = t.get_Y()
    assert np.array_equal(np.flatnonzero(~np.isfinite(y).all(1)), [at])
    return t, y


# the diverged point in the block of 64 points that the boundary divides
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_exact_gradient_of_the_other_embedding(precision):
    n, off = 200, np.array([0, 90, 200])
    t, y = diverged(precision, n, 80, 0.0, off)
    with t:
        g, _ = t.grad(0.0)
    assert np.isfinite(g[90:]).all() and not np.isfinite(g[:90]).any()
    with HyperbolicTSNE(precision=precision) as t:
        t.set_P(np.zeros(111, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float64))
        t.set_Y(y[90:])
        h, _ = t.grad(0.0)
    # the same terms in float32 (float64) sums of another order: 110 roundings each
    eps = 2.0 ** (-24 if precision == "fp32" else -53)
    assert np.linalg.norm(g[90:] - h) <= 110.0 * 8.0 * eps * np.linalg.norm(h)


# listed, direct (float32 above 32,768 points; a depth in float64), and the
# embedding beside it in a batch
@pytest.mark.parametrize("precision,n,depth", [("fp32", 2000, -1), ("fp32", 33000, -1), ("fp64", 2000, -1),
                                               ("fp64", 2000, 0), ("fp64", 12000, -1)])
def test_tree_gradient_of_its_own_embedding(precision, n, depth):
    t, y = diverged(precision, n, 17, 0.0)
    with t:
        t.set_walk_split(depth)
        g, z = t.grad(0.5)
        assert not np.isfinite(g).any() and not np.isfinite(z)
    off = np.array([0, 90, n])
    t, y = diverged(precision, n, 80, 0.0, off)
    with t:
        g, _ = t.grad(0.5)
        z = t.segment_Z()
    assert np.isfinite(g[90:]).all() and np.isfinite(z[1])
    assert not np.isfinite(g[:90]).any() and not np.isfinite(z[0])
