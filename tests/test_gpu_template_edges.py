"""The three template kernels (one or two sets with plain multiply-adds, FP64 matrix products,
products of base-256 digits) at the edges of their groups of sets and columns.

Tolerance: that of the parity test, 1e-10 of the value with a floor of 1e-3 of the family's
largest value.  FP64 sums of 2000 samples round at about 2000 x 1.1e-16 of their terms; seven
base-256 digits hold a factor to 2^-55 of the largest in its row or column.
"""
import numpy as np
import pytest

from oracle import template_oracle as T
from paper_2202_11839_gb300 import synthetic as S
from tests.test_gpu_template import FAMILY_SCALE, _window_table

pytestmark = pytest.mark.gpu


def _scale(ref):
    """Error scale per slot and shell of one parameter set's curves."""
    return np.stack([np.abs(ref[j]) + 1e-3 * np.abs(ref[FAMILY_SCALE[kind]]).max()
                     for j, (kind, _) in enumerate(T.SLOTS)])


@pytest.mark.parametrize("bins", [1, 7, 40, 41])
def test_set_counts_agree(bins):
    """Any number of sets gives each set's curves as a call of its own does (that call against
    the oracle for the first sets), with all slots and with a mask."""
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    edges = np.linspace(0.0, 0.2, bins + 1)
    params = S.latin_hypercube(300, seed=bins)
    params[::7, 0] = 0.0                       # no intrinsic alignment: exact zeros
    params[3::11, 0] *= 1e-6
    th = torch.from_numpy(params).cuda()
    tm = L.Template(q, s, edges, shot_plus=1234.5)
    single = np.stack([tm(th[i:i + 1]).cpu().numpy()[0] for i in range(300)])
    mix = T.mixing_table()
    for i in range(3):
        ref = np.stack(T.template(params[i], q, s, edges, shot_plus=1234.5, mixing=mix))
        sc = _scale(ref)
        assert (np.abs(single[i] - ref) <= 1e-10 * sc).all(), i
    for mask in (None, L.TEMPLATE_EB_SLOTS):
        if mask is not None:
            tm.set_slots(mask)
        for n in (2, 3, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 300):
            out = tm(th[:n]).cpu().numpy()
            for i in range(n):
                sc = _scale(single[i])
                want = single[i] if mask is None else np.where(
                    [[bool((mask >> j) & 1)] for j in range(L.LPP_N_MOMENTS)], single[i], 0.0)
                assert (np.abs(out[i] - want) <= 1e-10 * sc).all(), (mask, n, i)
    tm.close()
