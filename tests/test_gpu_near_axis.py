"""Harmonic weights of galaxies whose line of sight all but coincides with the grid's z axis: the squares
of its x and y components underflow in FP32.

Tolerance: FP32 against the FP64 path at 1e-5 of the per-bin scale, as in the parity tests."""
import numpy as np
import pytest

from tests import parity_util as U
from tests.test_gpu_parity import TOL32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0.0, 1e-30, 1e-22, 1e-20, 3e-20, 1e-19, 1e-17, 1e-12, 1e-6, 1e-3])
def test_lines_of_sight_close_to_the_axis(offset):
    from paper_2202_11839_gb300 import lpp as L
    n, box, count = 32, 500.0, 400
    rng = np.random.default_rng(3)
    pos = np.stack([offset * rng.uniform(0.3, 1.0, count), offset * rng.uniform(0.3, 1.0, count),
                    rng.uniform(0.0, box, count)]).astype(np.float32)
    cat = dict(pos=pos, w=rng.uniform(0.5, 1.5, count).astype(np.float32),
               shape=rng.standard_normal((6, count)).astype(np.float32))
    cfg = dict(n=n, box=box, observer=(0.0, 0.0, -40.0), pole=(0.0, 1.0, 0.0), scheme=3, interlace=True,
               k_edges=U.default_edges(n, box, 6))
    g64 = U.run_gpu(cfg, {k: v.astype(np.float64) for k, v in cat.items()}, L.LPP_FP64)
    g32 = U.run_gpu(cfg, cat, L.LPP_FP32)
    pp = np.abs(g64.raw[U.O.M_INDEX[("plus", 0)]].real) / g64.norm_auto
    pd = np.abs(g64.raw[U.O.M_INDEX[("dd", 0)]].real) / g64.norm_dd
    sc = np.abs(g64.p) + np.sqrt(pp * pd)[None, :]
    err = np.abs(g32.p - g64.p) / np.where(sc > 0, sc, 1.0)
    assert err.max() < TOL32, err.max(axis=1)
