"""Window multipoles through the z pass that multiplies by the window's transform and through the
reach masks: randoms confined to a few planes and pencils (most tiles empty) and filling the box,
on both FFT kernels (a pencil or a pair of pencils per thread).

Tolerance: FP64 against the oracle at 1e-10 and FP32 at 1e-5 of |Q_0| + |Q_l|, as in the parity
test."""
import numpy as np
import pytest

from oracle import lpp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec,tol,slab", [(8, 1, 1e-10, None), (64, 1, 1e-10, (0.4, 0.55)), (64, 0, 1e-5, (0.0, 0.1)),
                                             (128, 0, 1e-5, (0.7, 0.8)), (32, 0, 1e-5, None)])
@pytest.mark.parametrize("scheme", [2, 3])
def test_confined_randoms(n, prec, tol, slab, scheme):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    box = 400.0
    dt = np.float64 if prec == L.LPP_FP64 else np.float32
    rng = np.random.default_rng(n + scheme)
    pos = rng.uniform(0.0, box, (3, 2000))
    if slab:
        pos[1:] = box * (slab[0] + (slab[1] - slab[0]) * rng.random((2, 2000)))
    pos = pos.astype(dt)
    w, nbar = rng.uniform(0.8, 1.2, 2000).astype(dt), rng.uniform(0.5, 2.0, 2000).astype(dt)
    obs = (200.0, 180.0, -300.0)
    edges = np.linspace(0.0, 0.35 * box, 6)
    plan = L.Plan(n, box, np.linspace(0, 0.1, 3), observer=obs, scheme=scheme, precision=prec, moments=1,
                  max_shapes=10, max_randoms=2000)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    plan.assign(L.LPP_RANDOMS, t(pos), t(w), t(nbar))
    q, _, points, _ = plan.window_q(edges)
    q2, _, _, _ = plan.window_q(edges)
    plan.close()
    ref = O.window_multipoles(n, box, (0, 0, 0), obs, pos, w, nbar, 1.0, edges, scheme=scheme)
    np.testing.assert_array_equal(points, ref.n_points)
    scale = np.abs(ref.q[0])[None, :] + np.abs(ref.q)
    for got in (q, q2):
        assert (np.abs(got - ref.q) <= tol * np.where(scale > 0, scale, 1.0)).all()
