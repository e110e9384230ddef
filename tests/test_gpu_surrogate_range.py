"""The decoding (pre (mu + sum_q w_q base_q + sd y) + theta_5 shot - ref) / sigma over the values that FP64 maps
may hold: other units, empty error bars, baselines that span many binades.

Tolerance: the result is stored in FP32 (2^-24 of it; 2^-23 allows for the decoding's own rounding), and
2^-40 of the sum of the magnitudes of the terms, sum_q |w_q base_q| among them, for what a sum in pairs of
floats (about 2^-44 of the same sum) would leave.  The network's part is left out (sd = 0) but in the
last test.
"""
import numpy as np
import pytest

from paper_2202_11839_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

ROWS = [20, 640]   # both prediction kernels


def _net(seed=5):
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    return L, L.Surrogate(L.flatten_params(S.surrogate_init(seed)), batch=32)


def _dev(a):
    import torch
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _theta(rows, rng):
    th = np.column_stack([rng.uniform(0.5, 3, rows), rng.uniform(1, 3, rows), rng.uniform(0.6, 1, rows),
                          rng.uniform(-1, 1, rows), rng.uniform(-1, 1, rows), rng.uniform(0.5, 2, rows)])
    return np.ascontiguousarray(th)


def _lagrange(v, nodes):
    xs = -np.cos(np.pi * np.arange(nodes) / (nodes - 1))
    return np.stack([np.prod([(v - xs[j]) / (xs[i] - xs[j]) for j in range(nodes) if j != i], axis=0)
                     for i in range(nodes)], axis=-1)


# the fed inputs are the parameters themselves (lo = -1, hi = 1), so that a node is hit exactly
LO, HI = np.full(6, -1.0), np.full(6, 1.0)


def _predict(net, theta, mu, shot, ref, sigma, base, nodes, sd=None):
    keep = [_dev(a) for a in (mu, np.zeros(320) if sd is None else sd, shot, ref, sigma, base)]
    kw = dict(base=keep[5], base_nodes=nodes, base_in=(3, 4)) if base is not None else {}
    net.set_map(LO, HI, (0, 0, 0, 1, 1, 0), *keep[:5], **kw)
    return net.predict(_dev(theta)).double().cpu().numpy()


def _want(theta, mu, shot, ref, sigma, base, nodes, part=0.0):
    """The decoding in FP64 and the sum of the magnitudes of its terms, both over sigma."""
    A, b, s8, sh = theta[:, 0:1], theta[:, 1:2], theta[:, 2:3], theta[:, 5:6]
    pre = np.concatenate([np.repeat(A * b * s8 ** 2, 80, 1), np.repeat(A * A * s8 ** 2, 240, 1)], axis=1)
    u, mag = mu + part + np.zeros((len(theta), 320)), np.abs(mu) + np.abs(part) + np.zeros((len(theta), 320))
    if base is not None:
        la, lb = _lagrange(theta[:, 3], nodes), _lagrange(theta[:, 4], nodes)
        w = (la[:, :, None] * lb[:, None, :]).reshape(len(theta), -1)
        u, mag = u + w @ base, mag + np.abs(w) @ np.abs(base)
    rf = 0.0 if ref is None else ref
    sg = 1.0 if sigma is None else sigma
    with np.errstate(divide="ignore", invalid="ignore"):
        return (pre * u + sh * shot - rf) / sg, (np.abs(pre) * mag + np.abs(sh * shot) + np.abs(rf)) / np.abs(sg)


def _close(got, want, mag):
    with np.errstate(invalid="ignore"):
        return np.abs(got - want) <= 2.0 ** -23 * np.abs(want) + 2.0 ** -40 * mag


@pytest.mark.parametrize("rows", ROWS)
@pytest.mark.parametrize("unit", [1e-200, 1e-60, 1e-42, 1e-30, 1e30, 1e45, 1e150])
def test_other_units(rows, unit):
    L, net = _net()
    rng = np.random.default_rng(rows)
    mu, shot, ref = rng.standard_normal((3, 320)) * unit
    sigma = rng.uniform(0.5, 2, 320) * unit
    base = rng.standard_normal((16, 320)) * unit
    theta = _theta(rows, rng)
    args = (theta, mu, shot, ref, sigma, base, 4)
    want, mag = _want(*args)
    assert _close(_predict(net, *args), want, mag).all()
    # amplitudes instead: the curves of another unit of the parameters
    theta[:, 0] = rng.uniform(0.5, 1, rows) * 1e25
    mu, shot, ref, base = mu / unit, shot / unit, None, base / unit
    args = (theta, mu, shot, ref, np.where(np.arange(320) < 80, 1e25, 1e50), base, 4)
    want, mag = _want(*args)
    assert _close(_predict(net, *args), want, mag).all()
    net.close()


@pytest.mark.parametrize("rows", ROWS)
def test_empty_and_infinite_error_bars(rows):
    """sigma = 0: an infinity of the difference's sign; an infinite mean or sigma as in FP64."""
    L, net = _net()
    rng = np.random.default_rng(7)
    mu, shot, ref = rng.standard_normal((3, 320))
    sigma = np.ones(320)
    sigma[3::7] = 0.0
    sigma[5::7] = np.inf
    mu[4::40] = np.inf
    theta = _theta(rows, rng)
    args = (theta, mu, shot, ref, sigma, None, 0)
    want, mag = _want(*args)
    got = _predict(net, *args)
    fin = np.isfinite(want)
    assert (~fin).any() and np.array_equal(got[~fin], want[~fin], equal_nan=True)
    assert _close(got, want, mag)[fin].all()
    net.close()


@pytest.mark.parametrize("rows", ROWS)
@pytest.mark.parametrize("nodes", [2, 3, 5, 8])
def test_baselines_of_many_binades(rows, nodes):
    """One node's value far below the others of its column, parameters on that node and near it."""
    L, net = _net()
    rng = np.random.default_rng(nodes)
    base = rng.standard_normal((nodes * nodes, 320)) * 2.0 ** rng.integers(0, 60, 320)
    base[0] = rng.uniform(0.1, 1.0, 320) / 3.0
    theta = _theta(rows, rng)
    theta[:, 3:5] = -1.0
    theta[rows // 4:, 3] = -1.0 + 2.0 ** -rng.integers(3, 50, rows - rows // 4).astype(float)
    theta[rows // 2:, 4] = -1.0 + 2.0 ** -rng.integers(3, 50, rows - rows // 2).astype(float)
    args = (theta, np.zeros(320), np.zeros(320), None, None, base, nodes)
    want, mag = _want(*args)
    assert _close(_predict(net, *args), want, mag).all()
    net.close()


@pytest.mark.parametrize("rows", ROWS)
def test_the_network_part_in_another_unit(rows):
    """sd and sigma in a unit beyond FP32, against the same curves in units of one."""
    L, net = _net()
    rng = np.random.default_rng(11)
    theta = _theta(rows, rng)
    zero, unit = np.zeros(320), 2.0 ** 200
    sd = rng.uniform(0.5, 2, 320)
    plain = _predict(net, theta, zero, zero, None, np.ones(320), None, 0, sd=sd)
    scaled = _predict(net, theta, zero, zero, None, np.full(320, unit), None, 0, sd=sd * unit)
    assert np.isfinite(plain).all() and np.abs(plain).max() > 0
    np.testing.assert_allclose(scaled, plain, rtol=2.0 ** -23)
    net.close()
