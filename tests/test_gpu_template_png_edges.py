"""Templates with the spin-2 non-Gaussian response: the FP64 matrix products of three and more sets over all
their tile shapes (one to nine tiles of 8 rows a warp, whole slabs or column segments), ragged counts of sets
and tiles that straddle the families, against the oracle and against calls of one set.

Tolerance: that of the parity test, 1e-10 of the value with a floor of 1e-3 of the family's largest.
"""
import numpy as np
import pytest

from oracle import template_oracle as T
from paper_2202_11839_gb300 import synthetic as S
from tests.test_gpu_template import FAMILY_SCALE, _window_table

pytestmark = pytest.mark.gpu

PNG = (-180.0, 0.17, 0.3)


def _scale(ref):
    return np.stack([np.abs(ref[j]) + 1e-3 * np.abs(ref[FAMILY_SCALE[kind]]).max()
                     for j, (kind, _) in enumerate(T.SLOTS)])


# with 305 sets all shells are in one group: 14 rows a shell; 1 to 4 shells take column segments, more whole
# slabs (2 tiles a warp from 5 shells on, 9 from 37)
@pytest.mark.parametrize("bins", [1, 2, 3, 4, 7, 13, 18, 22, 27, 32, 36, 40, 41, 60])
def test_tile_shapes(bins):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    edges = np.linspace(0.0, 0.2, bins + 1)
    params = S.latin_hypercube(305, seed=bins)
    th = torch.from_numpy(params).cuda()
    tm = L.Template(q, s, edges, shot_plus=1234.5)
    tm.set_png(*PNG)
    single = np.stack([tm(th[i:i + 1]).cpu().numpy()[0] for i in range(305)])
    mix = T.mixing_table()
    for i in (0, 1):
        ref = np.stack(T.template(params[i], q, s, edges, shot_plus=1234.5, mixing=mix, png=PNG))
        assert (np.abs(single[i] - ref) <= 1e-10 * _scale(ref)).all(), i
    for mask in (None, L.TEMPLATE_EB_SLOTS):
        if mask is not None:
            tm.set_slots(mask)
        for n in (2, 3, 8, 9, 33, 305):
            out = tm(th[:n]).cpu().numpy()
            for i in range(n):
                want = single[i] if mask is None else np.where(
                    [[bool((mask >> j) & 1)] for j in range(L.LPP_N_MOMENTS)], single[i], 0.0)
                assert (np.abs(out[i] - want) <= 1e-10 * _scale(single[i])).all(), (mask, n, i)
    tm.close()
