"""FP32 arrays of the surrogate that start at any float (a view at an odd offset): outputs of
infer and predict, targets of train and gradients.

Nothing is rounded differently for another address, so the results are those of 16-byte aligned arrays
bit for bit; the losses are FP64 atomic sums in any order (1e-12).
"""
import numpy as np
import pytest

from paper_2202_11839_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _net(batch=96, seed=5):
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    return L, L.Surrogate(L.flatten_params(S.surrogate_init(seed)), batch=batch)


def _at(offset, shape):
    """A float array whose first element lies `offset` floats after a 256-byte boundary, and the buffer
    of sentinels around it."""
    import torch
    n = int(np.prod(shape))
    buf = torch.full((n + 8,), -7.0, dtype=torch.float32, device="cuda")
    return buf[offset:offset + n].view(shape), buf


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("rows", [1, 9, 16, 33, 640, 650])
def test_outputs_at_any_float(rows, offset):
    import torch
    L, net = _net()
    lo, hi = S.SURROGATE_RANGES[:, 0], S.SURROGATE_RANGES[:, 1]
    one, zero = (torch.full((320,), v, dtype=torch.float64, device="cuda") for v in (1.0, 0.0))
    base = torch.linspace(-1.0, 1.0, 16 * 320, dtype=torch.float64, device="cuda")
    net.set_map(lo, hi, (1,) * 6, zero, one, zero, None, one, base=base, base_nodes=4)
    theta = torch.from_numpy(S.latin_hypercube(rows, seed=rows)).cuda()
    x = net.encode(theta)
    for call, arg in ((net.infer, x), (net.predict, theta)):
        want = call(arg).cpu().numpy()
        view, buf = _at(offset, (rows, 320))
        call(arg, out=view)
        assert np.array_equal(view.cpu().numpy(), want)
        rest = torch.cat([buf[:offset], buf[offset + rows * 320:]])
        assert bool((rest == -7.0).all())
    net.close()


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_targets_at_any_float(offset):
    import torch
    batch, n = 96, 130
    rng = np.random.default_rng(offset)
    x = torch.from_numpy(rng.uniform(-1, 1, (n, 6)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.standard_normal((n, 320)).astype(np.float32)).cuda()
    sched = torch.from_numpy(np.concatenate([rng.permutation(n)[:batch] for _ in range(3)]).astype(np.int32)).cuda()
    got = []
    for off in (0, offset):
        L, net = _net(batch)
        yv, _ = _at(off, (n, 320))
        yv.copy_(y)
        xv, _ = _at(off, (n, 6))
        xv.copy_(x)
        g, loss = net.gradients(xv, yv, sched[:batch])
        losses = torch.zeros(3, dtype=torch.float64, device="cuda")
        net.train(xv, yv, sched, 1e-3, losses)
        got.append((g, net.params(), loss, losses.cpu().numpy()))
        net.close()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    np.testing.assert_allclose(got[0][2], got[1][2], rtol=1e-12)
    np.testing.assert_allclose(got[0][3], got[1][3], rtol=1e-12)
