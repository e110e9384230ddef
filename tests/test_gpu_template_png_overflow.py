"""A response so large that the shape spectra overflow leaves the families that carry less of it alone.

Tolerance: that of the parity test, 1e-10 of the value with a floor of 1e-3 of the family's largest."""
import numpy as np
import pytest

from oracle import template_oracle as T
from paper_2202_11839_gb300 import synthetic as S
from tests.test_gpu_template import _window_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f_nl,families", [(1e200, ("dd", "cross")), (float("inf"), ("dd",))])
@pytest.mark.parametrize("bins", [1, 7, 40])
def test_overflow_stays_in_its_family(f_nl, families, bins):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    th = torch.from_numpy(S.latin_hypercube(9, seed=3)).cuda()
    tm = L.Template(q, s, np.linspace(0.0, 0.2, bins + 1))
    tm.set_png(f_nl)
    single = np.stack([tm(th[i:i + 1]).cpu().numpy()[0] for i in range(9)])
    slots = [j for j, (kind, _) in enumerate(T.SLOTS) if kind in families]
    assert np.isfinite(single[:, slots]).all() and not np.isfinite(single[:, 4]).any()
    for n in (3, 9):
        got = tm(th[:n]).cpu().numpy()
        for i in range(n):
            for j in slots:
                ref = single[i, j]
                fam = np.abs(single[i, 0 if T.SLOTS[j][0] == "dd" else 1]).max()
                assert (np.abs(got[i, j] - ref) <= 1e-10 * (np.abs(ref) + 1e-3 * fam)).all(), (n, i, j)
    tm.close()
