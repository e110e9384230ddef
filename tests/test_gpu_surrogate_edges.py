"""The surrogate's row-chain kernels at the edges of their tiles: groups of 16 rows on clusters,
groups of 32 rows in one CTA, weight tiles and minibatch panels of 128 rows, and the baseline as
digit products for every number of Lobatto nodes.

Tolerances.  Gradients and outputs: both sides round the operands to BF16, the GPU may round to
the neighbour (2^-8 on that element), a few 1e-3 norm-wise.  The decoded baseline: weights and
base values are 48-bit fixed-point numbers relative to the largest of their row and column, and
products below 2^-48 of the two maxima are dropped (at most 15 of them on each of 64 terms:
below 2^-38); the prediction is stored in FP32.
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2202_11839_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _net(batch, seed=5):
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    rng = np.random.default_rng(seed)
    layers = [(w, (rng.standard_normal(b.shape) * 0.05).astype(np.float32)) for w, b in S.surrogate_init(seed)]
    return L, L.Surrogate(L.flatten_params(layers), batch=batch), layers, rng


def _dev(a, dtype=np.float64):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def _lagrange(v, nodes):
    xs = -np.cos(np.pi * np.arange(nodes) / (nodes - 1))
    return np.array([np.prod([(v - xs[j]) / (xs[i] - xs[j]) for j in range(nodes) if j != i])
                     for i in range(nodes)])


@pytest.mark.parametrize("batch", [32, 96, 128, 160, 288])
def test_gradients_of_ragged_minibatches(batch):
    L, net, layers, rng = _net(batch)
    n = batch + 17
    x = rng.uniform(-1, 1, (n, 6)).astype(np.float32)
    y = rng.standard_normal((n, 320)).astype(np.float32)
    idx = rng.permutation(n)[:batch].astype(np.int32)
    g, loss = net.gradients(_dev(x, np.float32), _dev(y, np.float32), _dev(idx, np.int32))
    ws = [w.astype(np.float64) for w, _ in layers]
    bs = [b.astype(np.float64) for _, b in layers]
    rl, gws, gbs = M.loss_and_grads(ws, bs, x[idx].astype(np.float64), y[idx].astype(np.float64))
    assert abs(loss - rl) <= 1e-4 * rl
    for li, (gw, gb) in enumerate(L.unflatten_params(g)):
        assert np.linalg.norm(gw - gws[li]) < 5e-3 * np.linalg.norm(gws[li]), li
        assert np.linalg.norm(gb - gbs[li]) < 5e-3 * np.linalg.norm(gbs[li]), li
    net.close()


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 31, 33, 607, 608, 609, 640, 1000])
def test_predict_rows(rows):
    """Ragged row counts on both prediction kernels, against the oracle's network."""
    import torch
    L, net, layers, rng = _net(1024)
    lo, hi = S.SURROGATE_RANGES[:, 0], S.SURROGATE_RANGES[:, 1]
    one, zero = np.ones(320), np.zeros(320)
    maps = [_dev(zero), _dev(one), _dev(zero), _dev(zero), _dev(one)]
    net.set_map(lo, hi, (1,) * 6, *maps)
    theta = S.latin_hypercube(rows, seed=rows)
    got = net.predict(_dev(theta)).double().cpu().numpy()
    assert got.shape == (rows, 320)
    x = (2 * (theta - lo) / (hi - lo) - 1).astype(np.float32).astype(np.float64)
    ref, _ = M.forward([w.astype(np.float64) for w, _ in layers], [b.astype(np.float64) for _, b in layers], x)
    A, b, s8 = theta[:, 0:1], theta[:, 1:2], theta[:, 2:3]
    pre = np.concatenate([np.repeat(A * b * s8 ** 2, 80, 1), np.repeat(A * A * s8 ** 2, 240, 1)], axis=1)
    want = pre * ref
    err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(pre * np.abs(ref).max(), axis=1)
    assert err.max() < 5e-3, err.max()
    net.close()


@pytest.mark.parametrize("nodes", [0, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("rows", [33, 640])
def test_baseline_digits(nodes, rows):
    """The decoding without the network's part (sd = 0): columns whose base spans many binades or
    is zero, parameters inside and outside of the box (Lagrange weights above one)."""
    L, net, layers, rng = _net(1024)
    lo, hi = S.SURROGATE_RANGES[:, 0], S.SURROGATE_RANGES[:, 1]
    theta = S.latin_hypercube(rows, seed=3)
    theta[::5, 3:5] = lo[3:5] + (hi - lo)[3:5] * rng.uniform(-0.5, 1.5, (len(theta[::5]), 2))
    theta[1, 3:5] = lo[3:5]        # on a node: one weight is 1, the others 0
    mu, shot, sig = rng.standard_normal(320), rng.uniform(0, 5, 320), rng.uniform(1.0, 3.0, 320)
    base = rng.standard_normal((max(nodes, 1) ** 2, 320)) * 2.0 ** rng.integers(-30, 30, 320)
    base[:, 7] = 0.0
    base[0, 11] = 1e6
    keep = [_dev(mu), _dev(np.zeros(320)), _dev(shot), _dev(sig), _dev(base.reshape(-1))]
    kw = dict(base=keep[4], base_nodes=nodes, base_in=(3, 4)) if nodes else {}
    net.set_map(lo, hi, (1,) * 6, keep[0], keep[1], keep[2], None, keep[3], **kw)
    got = net.predict(_dev(theta)).double().cpu().numpy()
    A, b, s8, sh = theta[:, 0:1], theta[:, 1:2], theta[:, 2:3], theta[:, 5:6]
    pre = np.concatenate([np.repeat(A * b * s8 ** 2, 80, 1), np.repeat(A * A * s8 ** 2, 240, 1)], axis=1)
    x = 2 * (theta - lo) / (hi - lo) - 1
    bl, big = np.zeros((rows, 320)), np.zeros((rows, 320))
    for r in range(rows if nodes else 0):
        w = np.outer(_lagrange(x[r, 3], nodes), _lagrange(x[r, 4], nodes)).reshape(-1)
        bl[r] = w @ base
        big[r] = np.abs(w).max() * np.abs(base).max(axis=0)
    want = (pre * (mu + bl) + sh * shot) / sig
    tol = 2.0 ** -22 * np.abs(want) + 2.0 ** -34 * (pre * (np.abs(mu) + big) + sh * shot) / sig
    assert (np.abs(got - want) <= tol).all(), (np.abs(got - want) / tol).max()
    net.close()
