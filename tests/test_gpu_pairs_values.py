"""Window pair counts where a pair has no direction or a separation far below one.

Tolerances: FP64 sums of at most 5e4 pairs, 1e-12 of the shell's Q_0 (the same pairs, the same
operations but for a power of two); 1e-6 where a separation is replaced by a larger parallel one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _q(pos, w, observer, edges, box=0.0):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    return L.window_q_pairs(t(pos), t(w), None, observer, np.asarray(edges, dtype=np.float64), alpha=0.5, box=box)


def test_monopole_with_a_point_at_the_observer():
    """Q_0 does not depend on the observer, also where a line of sight does not exist."""
    rng = np.random.default_rng(2)
    pos, w = rng.uniform(0, 100, (3, 200)), rng.uniform(0.5, 1.5, 200)
    edges = np.linspace(0, 60, 7)
    want = _q(pos, w, (50.0, 50.0, -300.0), edges)
    got = _q(pos, w, tuple(pos[:, 17]), edges)
    np.testing.assert_allclose(got[0], want[0], rtol=1e-12)


@pytest.mark.parametrize("exponent", [-20, -150, -154, -155, -156, -158])
def test_separations_near_the_underflow_threshold(exponent):
    """Two points 10^exponent apart have the multipoles of two points 1e-6 apart in the same direction."""
    d = np.array([0.3, -0.5, 0.7])
    w, edges, observer = np.array([1.0, 2.0]), (0.0, 1.0), (3.0, 2.0, -10.0)
    pair = lambda s: np.stack([np.zeros(3), d * s], axis=1)
    want, got = _q(pair(1e-6), w, observer, edges), _q(pair(10.0 ** exponent), w, observer, edges)
    np.testing.assert_allclose(got, want, atol=1e-6 * want[0].max())


@pytest.mark.parametrize("power", [-40, -60, -70, -71, -72, -76])
@pytest.mark.parametrize("periodic", [False, True])
def test_shells_in_a_small_unit(power, periodic):
    """Every length times a power of two: the same pairs in the same shells."""
    rng = np.random.default_rng(5)
    pos, w = rng.uniform(0, 1, (3, 300)), rng.uniform(0.5, 1.5, 300)
    edges, observer, u = np.linspace(0, 0.45, 10), np.array([0.5, 0.4, -3.0]), 2.0 ** power
    want = _q(pos, w, tuple(observer), edges, 1.0 if periodic else 0.0)
    got = _q(pos * u, w, tuple(observer * u), edges * u, u if periodic else 0.0) * u ** 3
    assert (np.abs(got - want) <= 1e-12 * np.abs(want[0])).all()
