"""Window pair counts at the edges of the kernel's tiles of 128 points, from one shell to the
largest number of shells, with points on shell edges and pairs without separation.

Tolerance: FP64 sums of at most 2.6e5 pairs; 1e-10 of |Q_0| + |Q_l| per shell, as for the larger
catalogues."""
import numpy as np
import pytest

from oracle import lpp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 257, 511])
@pytest.mark.parametrize("shells", [1, 40, 45, 256])
def test_tile_and_shell_edges(n, shells, periodic):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    rng = np.random.default_rng(n + shells)
    box = 400.0 if periodic else 0.0
    pos = rng.uniform(0.0, 400.0, (3, n))
    if n > 100:
        pos[:, 5] = pos[:, 60]                                       # no separation
        pos[:, 61], pos[:, 7] = (100.0, 120.0, 130.0), (100.0, 150.0, 170.0)   # 50 apart, exactly
        pos[:, 100] = pos[:, 3]
    w = rng.uniform(0.5, 1.5, n)
    nbar = rng.uniform(0.5, 2.0, n) * 1e-4
    obs = (200.0, 200.0, -900.0)
    edges = np.linspace(0.0, 200.0, shells + 1) if shells != 45 else np.sort(rng.uniform(3.0, 190.0, 46))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    q = L.window_q_pairs(t(pos), t(w), t(nbar), obs, edges, alpha=0.3, box=box)
    ref = O.window_pair_count_shells(pos, w, nbar, 0.3, obs, edges, box=box)
    scale = np.abs(ref[0])[None, :] + np.abs(ref)
    assert (np.abs(q - ref) <= 1e-10 * np.where(scale > 0, scale, 1e-290)).all()
