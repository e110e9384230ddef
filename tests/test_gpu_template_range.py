"""Templates of parameters far outside of the emulator's box, whose spectra vary by many powers of two
against the reference of the digit products: calls of three and more sets (digits) against calls of one
set (FP64 multiply-adds of the same spectra and operator).

Tolerance: both are FP64 sums of 2048 products, at most some 24 roundings deep (8 columns a lane, the lanes,
the slabs, the normalisation): 24 x 2^-53 = 2.7e-15 of the sum of the products' magnitudes on
each side; 1e-14 of it between them.  The magnitudes come from the operator's rows, formed here by
transposing the oracle's chain.
"""
import numpy as np
import pytest

from oracle import template_oracle as T
from paper_2202_11839_gb300 import synthetic as S
from tests.test_gpu_template import _window_table

pytestmark = pytest.mark.gpu

BINS = 9


def _magnitudes(params, q, s, edges):
    """sum_n |op[n] P(k_n)| per slot and shell of one parameter set."""
    k, r, delta = T.log_grid()
    kin, kr0 = k[:T.N_IN], k[0] * r[0]
    transform = lambda x, ell, bias: np.real(np.fft.fft(np.fft.fft(x) * T.fftlog_kernel(ell, bias, delta, kr0))) / T.N_FFT
    qr, mix, model, p = T.q_on_r(q, s, r), T.mixing_table(), T.model_multipoles(params), T.linear_pk(params)[:T.N_IN]
    out = np.zeros((len(T.SLOTS), len(edges) - 1))
    for i, (kind, L) in enumerate(T.SLOTS):
        for b in range(len(edges) - 1):
            sel = (kin >= edges[b]) & (kin < edges[b + 1])
            x = np.zeros(T.N_FFT)
            x[:T.N_IN][sel] = kin[sel] ** 3 / np.sum(kin[sel] ** 3) * 4 * np.pi * kin[sel] ** -T.Q_FWD
            back = transform(x, L, T.Q_FWD) * r ** (3 - T.Q_FWD) * r ** -T.Q_INV / (2 * np.pi ** 2)
            row = np.zeros(T.N_IN)
            for lp, c in model[kind].items():
                qx = sum(mix[(kind, L, lp)][j] * qr[j] for j in range(5))
                row += (-1) ** (lp // 2) * transform(c * qx * back, lp, T.Q_INV)[:T.N_IN]
            out[i, b] = np.abs(row * kin ** (3 - T.Q_INV) * T.taper() * p).sum()
    return out


@pytest.mark.parametrize("n", [3, 16, 70])
def test_spectra_far_from_the_reference(n):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    edges = np.linspace(0.0, 0.2, BINS + 1)
    far = [(3.0, 0.2), (-3.0, 0.2), (8.0, 0.2), (-8.0, 0.2), (20.0, 0.2), (-20.0, 0.2), (2.0, 5.0), (-1.0, 0.002), (0.0, 0.2)]
    params = S.latin_hypercube(n, seed=n)
    for i in range(n):
        params[i, 3:5] = far[i % len(far)] if i % 3 or n == 3 else params[i, 3:5]
    params[:, 5] = 0.0
    th = torch.from_numpy(params).cuda()
    tm = L.Template(q, s, edges)
    many = tm(th).cpu().numpy()
    single = np.stack([tm(th[i:i + 1]).cpu().numpy()[0] for i in range(n)])
    tm.close()
    for i in range(min(n, 20)):
        mag = _magnitudes(params[i], q, s, edges)
        assert (np.abs(many[i] - single[i]) <= 1e-14 * mag).all(), params[i, 3:5]


def test_no_spectrum_is_no_number():
    """A set without a spectrum (Gamma = NaN) leaves the others of its call alone."""
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    params = S.latin_hypercube(20, seed=1)
    th = torch.from_numpy(params).cuda()
    tm = L.Template(q, s, np.linspace(0.0, 0.2, BINS + 1))
    want = tm(th).cpu().numpy()
    th[7, 4] = float("nan")
    got = tm(th).cpu().numpy()
    tm.close()
    assert np.isnan(got[7]).all()
    keep = np.arange(20) != 7
    assert np.array_equal(got[keep], want[keep])
