"""Calls of different sizes from several host threads at once, each with its own handle and stream: every
call succeeds and gives what it gives alone, bit for bit."""
import threading

import numpy as np
import pytest

from paper_2202_11839_gb300 import synthetic as S
from tests.test_gpu_template import _window_table

pytestmark = pytest.mark.gpu


def _together(calls, want, repeats):
    errors = []

    def work(call, ref):
        try:
            for _ in range(repeats):
                got = call()
            assert np.array_equal(got.cpu().numpy() if hasattr(got, "cpu") else got, ref)
        except Exception as e:   # noqa: BLE001 - reported below
            errors.append(e)
    threads = [threading.Thread(target=work, args=a) for a in zip(calls, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("png", [0.0, -100.0])
def test_templates_of_different_sizes(png):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    q, s = _window_table()
    calls, want, keep = [], [], []
    for bins, sets in ((60, 400), (1, 3), (40, 16), (3, 64)):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            tm = L.Template(q, s, np.linspace(0.0, 0.2, bins + 1), stream=st)
            tm.set_png(png)
            th = torch.from_numpy(S.latin_hypercube(sets, seed=bins)).cuda()
            out = torch.empty((sets, L.LPP_N_MOMENTS, bins), dtype=torch.float64, device="cuda")
        st.synchronize()

        def call(tm=tm, th=th, out=out, st=st):
            tm(th, out=out)
            st.synchronize()
            return out
        calls.append(call)
        want.append(call().cpu().numpy().copy())
        keep.append((tm, st))
    _together(calls, want, 400)


def test_pair_counts_of_different_sizes():
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    rng = np.random.default_rng(1)
    calls, want = [], []
    for shells in (256, 1, 40):
        pos = torch.from_numpy(rng.uniform(0, 100, (3, 100))).cuda()   # one tile: the sums have one order
        st = torch.cuda.Stream()
        torch.cuda.synchronize()

        def call(pos=pos, st=st, edges=np.linspace(0, 90, shells + 1)):
            return L.window_q_pairs(pos, None, None, (50.0, 50.0, -300.0), edges, stream=st)
        calls.append(call)
        want.append(call())
    _together(calls, want, 400)
