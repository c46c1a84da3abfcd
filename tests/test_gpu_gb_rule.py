"""Which GB energies and gradients run as one cluster launch."""
import ctypes as C

import pytest

from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _captured_nodes(call):
    import torch
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    h, graph, n = C.c_void_p(st.cuda_stream), C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
    try:
        call(st.cuda_stream)
    finally:
        assert cu.cuStreamEndCapture(h, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    cu.cuGraphDestroy(graph)
    return n.value


@pytest.mark.parametrize("n,n_rep,cluster", [
    (237, 1, True), (512, 64, True), (40, 160, True), (20, 300, True), (237, 128, True), (513, 1, False),
    (512, 128, False), (40, 256, False), (128, 224, False), (20, 640, False), (60, 2048, False), (4, 20000, False)])
def test_one_launch_where_it_pays(n, n_rep, cluster):
    import torch
    s = synth.make_system(n, n, n_ph=0, n_redox=0)
    x, q, rho = (torch.tensor(a, dtype=torch.float32, device="cuda:0").expand(n_rep, *a.shape).contiguous()
                 for a in (s.x, s.q, s.rho))
    scr = torch.tensor(s.screen, dtype=torch.float32, device="cuda:0")
    up, ws = torch.ones(n_rep, dtype=torch.float64, device="cuda:0"), cphremd._workspace(n_rep, n, "cuda:0")
    for call in (lambda st: cphremd.gb_energy(x, q, rho, scr, workspace=ws, stream=st),
                 lambda st: cphremd.gb_energy_backward(x, q, rho, scr, up, workspace=ws, stream=st)):
        call(None)  # (its output's memory is then at hand)
        assert (_captured_nodes(call) == 1) == cluster
