"""The surrogate's copy of the map's baseline: formed wherever it may not be there.  Predictions are
functions of the network, the map and the parameters alone, so two orders of calls agree bit for
bit."""
import ctypes as C

import numpy as np
import pytest

from paper_2202_11839_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _net(stream=None):
    import torch
    from paper_2202_11839_gb300 import lpp as L
    L.load_library()
    flat = L.flatten_params(S.surrogate_init(3))
    net = L.Surrogate(flat, batch=32, stream=stream)
    lo, hi = S.SURROGATE_RANGES[:, 0], S.SURROGATE_RANGES[:, 1]
    rng = np.random.default_rng(1)
    t = lambda a: torch.from_numpy(a).cuda()
    net.set_map(lo, hi, (1,) * 6, t(rng.standard_normal(320)), t(np.ones(320)), t(np.zeros(320)),
                base=t(rng.standard_normal(16 * 320)), base_nodes=4)
    return L, net, flat, t(S.latin_hypercube(40, seed=2))


def test_predict_after_a_new_workspace():
    """set_workspace (new parameters, Adam reset) keeps the map: the baseline is not lost with the
    old contents of the workspace."""
    import torch
    L, net, flat, theta = _net()
    want = net.predict(theta).cpu().numpy()
    other = torch.empty_like(net.workspace)
    size = net.workspace.numel() - 256
    for ws in (net.workspace, other):
        addr = ws.data_ptr() + (-ws.data_ptr()) % 256
        assert L.load_library().lpp_surrogate_set_workspace(
            net.h, C.c_void_p(addr), C.c_size_t(size), flat.ctypes.data_as(C.POINTER(C.c_float)),
            C.c_void_p(net.stream.cuda_stream)) == L.LPP_OK
        assert np.array_equal(net.predict(theta).cpu().numpy(), want)
    net.close()


def test_predict_after_a_capture():
    """A first predict that is only captured forms nothing: the next one outside of the graph, before the graph
    has run, and the graph itself give the same curves."""
    import torch
    _, ref, _, theta = _net()
    want = ref.predict(theta).cpu().numpy()
    ref.close()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        _, net, _, theta = _net(stream=st)
        out = torch.zeros((40, 320), dtype=torch.float32, device="cuda")
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            net.predict(theta, out=out)
        eager = net.predict(theta)
        st.synchronize()
        assert np.array_equal(eager.cpu().numpy(), want)
        graph.replay()
        st.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
    net.close()
