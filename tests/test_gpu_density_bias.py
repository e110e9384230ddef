"""The density field of data minus alpha randoms in FP32, whose difference magnifies a common rounding of
all randoms: particles with one offset within their cells along x, alpha exact in FP32 with an odd
mantissa.

Tolerance: 1e-6 of the FP64 path's shell value.  A relative bias b of the randoms' weights moves the lowest
shell's P_dd, whose modes see the footprint's whole weight against the shot noise of 1.9M particles, by
about 2 b sqrt(8.4e5) 0.6 = 1.1e3 b.  A rounding that all particles share is up to 3e-8 (3e-5), one
that differs between them averages to 2e-10 (2e-7); the FP32 transforms add a few 1e-7.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interlace", [False, True])
@pytest.mark.parametrize("offset", [0.05, 0.1, 0.2, 0.3])
def test_randoms_with_one_offset(offset, interlace):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    n, n_rand, n_data = 256, 1 << 20, 838861   # about one particle per cell of the footprint
    rng = np.random.default_rng(int(100 * offset))

    def points(count):
        x = rng.integers(128, 255, count) + np.round(offset * 2 ** 16) / 2 ** 16
        return np.stack([x, rng.uniform(66, 194, count), rng.uniform(66, 194, count)]).astype(np.float32)
    data, rand = points(n_data), points(n_rand)
    raw = {}
    for prec, dt in ((L.LPP_FP64, np.float64), (L.LPP_FP32, np.float32)):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda()
        plan = L.Plan(n, float(n), np.linspace(0.5, 3.5, 4) * 2 * np.pi / n, observer=(128.0, 128.0, -900.0), scheme=3,
                      interlace=interlace, precision=prec, moments=1, max_shapes=n_data, max_randoms=n_rand)
        plan.assign(L.LPP_SHAPES, t(data), None, None, None, L.LPP_SHAPE_NONE)
        plan.assign(L.LPP_RANDOMS, t(rand), None, t(np.full(n_rand, 0.1)))
        raw[prec] = plan.multipoles().raw[0].real
        plan.close()
    err = np.abs(raw[L.LPP_FP32] - raw[L.LPP_FP64]) / np.abs(raw[L.LPP_FP64])
    assert err.max() < 1e-6, err
