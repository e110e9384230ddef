"""The fused assignment and transform passes with particles on the faces of the box, of the cells
and of the tiles, over grids from one tile to many, for every assignment order, interlaced and
not, in both precisions.

Tolerances: the FP64 path against the oracle at 1e-10 and the FP32 path against the FP64 path at
1e-5 of the per-bin scale |P| + sqrt(P_+^(0) P_dd^(0)), as in the parity tests.
"""
import numpy as np
import pytest

from tests import parity_util as U
from tests.test_gpu_parity import TOL32, TOL64

pytestmark = pytest.mark.gpu


def _catalogue(n, box, count, seed, n_rand=0):
    """Float32 positions; a third of them on faces of cells, half cells and the box."""
    cat = U.make_case("faces", n, count, seed, box=box, n_rand=n_rand, dtype=np.float32)
    rng = np.random.default_rng(seed)
    for key in ("pos", "rpos"):
        if key not in cat:
            continue
        p = cat[key]
        for ax in range(3):
            sel = rng.random(p.shape[1]) < 0.33
            grid = rng.integers(0, 2 * n, sel.sum()) * (0.5 * box / n)
            grid[::5] = np.where(rng.random(grid[::5].size) < 0.5, 0.0, box)
            grid[1::5] = np.where(rng.random(grid[1::5].size) < 0.5, np.nextafter(np.float32(box), np.float32(0)), 1e-30)
            p[ax, sel] = grid.astype(np.float32)
    return cat


def _cfg(n, box, scheme, interlace, nb=6, frac=1.0, **kw):
    return dict(n=n, box=box, observer=(box / 2, box / 2, -800.0), scheme=scheme, interlace=interlace,
                k_edges=U.default_edges(n, box, nb, frac), **kw)


@pytest.mark.parametrize("scheme", [2, 3])
@pytest.mark.parametrize("interlace", [False, True])
@pytest.mark.parametrize("n", [8, 16, 32])
def test_fp64_faces(n, scheme, interlace):
    cat = _catalogue(n, 256.0, 900, seed=n + scheme, n_rand=1500)
    cfg = _cfg(n, 256.0, scheme, interlace, nb=3)
    from paper_2202_11839_gb300 import lpp as L
    cat64 = {k: v.astype(np.float64) for k, v in cat.items()}
    U.assert_parity(U.run_gpu(cfg, cat64, L.LPP_FP64), U.run_oracle(cfg, cat64), TOL64, f"faces {n}")


@pytest.mark.parametrize("scheme", [2, 3])
@pytest.mark.parametrize("interlace", [False, True])
@pytest.mark.parametrize("n,nb,frac", [(16, 1, 0.3), (32, 4, 1.0), (64, 8, 1.0), (64, 1, 0.1), (128, 8, 1.0),
                                       (256, 5, 0.25)])
def test_fp32_matches_fp64_faces(n, nb, frac, scheme, interlace):
    from paper_2202_11839_gb300 import lpp as L
    cat = _catalogue(n, 512.0, 20_000, seed=n + scheme, n_rand=30_000)
    cfg = _cfg(n, 512.0, scheme, interlace, nb, frac)
    g64 = U.run_gpu(cfg, {k: v.astype(np.float64) for k, v in cat.items()}, L.LPP_FP64)
    g32 = U.run_gpu(cfg, cat, L.LPP_FP32)
    np.testing.assert_array_equal(g32.n_modes, g64.n_modes)
    pp = np.abs(g64.raw[U.O.M_INDEX[("plus", 0)]].real) / g64.norm_auto
    pd = np.abs(g64.raw[U.O.M_INDEX[("dd", 0)]].real) / g64.norm_dd
    sc = np.abs(g64.p) + np.sqrt(pp * pd)[None, :]
    err = np.abs(g32.p - g64.p) / np.where(sc > 0, sc, 1.0)
    assert err.max() < TOL32, err.max(axis=1)


@pytest.mark.parametrize("n", [64, 128])
def test_one_slot_matches_two_slot_small_grids(n):
    """fused_slots = 1 against the default on grids of a few tiles."""
    from paper_2202_11839_gb300 import lpp as L
    cat = _catalogue(n, 512.0, 30_000, seed=n, n_rand=20_000)
    cfg = _cfg(n, 512.0, 3, True, 8)
    two = U.run_gpu(cfg, cat, L.LPP_FP32)
    one = U.run_gpu(dict(cfg, fused_slots=1), cat, L.LPP_FP32)
    assert two.extra["path"]["two_slot_launches"] > 0
    assert one.extra["path"]["two_slot_launches"] == 0
    pp = np.abs(one.raw[U.O.M_INDEX[("plus", 0)]].real) / one.norm_auto
    pd = np.abs(one.raw[U.O.M_INDEX[("dd", 0)]].real) / one.norm_dd
    sc = np.abs(one.p) + np.sqrt(pp * pd)[None, :]
    assert (np.abs(one.p - two.p) / np.where(sc > 0, sc, 1.0)).max() < TOL32
