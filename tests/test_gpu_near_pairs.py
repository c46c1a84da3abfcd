"""The GB energy and its gradient at the edges of their kernels: the cluster
kernel for small replicas, and the symmetric pair kernels, whose near pairs (half
of the warp steps of small chains meet one) are evaluated apart from the tile
loop, with work items of 2 to 16 j-tiles."""
import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _rel(a, b):
    return np.sqrt(((a - b) ** 2).mean()) / max(np.sqrt((b ** 2).mean()), 1e-6)


@pytest.mark.parametrize("rgbmax", [0.0, 9.0])
@pytest.mark.parametrize("n", [2, 31, 33, 64, 65, 255, 257, 300])
def test_energy_and_gradient_at_tile_edges(n, rgbmax):
    """One replica and 1300 against the oracle, at the repository's bars (energy
    1e-6, gradients 1e-5 RMS relative); where the two run different kernels they
    sum the same FP32 pair terms in another order, so they agree to a few
    roundings (2e-6)."""
    import torch
    s, x, q, rho = synth.config_c5(n_rep=1300, n=n, seed=90 + n)
    gb = cphremd.default_gb()
    gb.rgbmax = rgbmax
    t = [torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in (x, q, rho)]
    scr = torch.tensor(s.screen, dtype=torch.float32, device="cuda:0")
    up = torch.ones(1300, dtype=torch.float64, device="cuda:0")
    E = cphremd.gb_energy(*t, scr, gb=gb).cpu().numpy()
    g = [a.cpu().numpy().astype(np.float64) for a in cphremd.gb_energy_backward(*t, scr, up, gb=gb)]
    for r in (0, 1299):
        one = [a[r:r + 1].contiguous() for a in t]
        E1 = cphremd.gb_energy(*one, scr, gb=gb).item()
        g1 = [a.cpu().numpy().astype(np.float64)[0] for a in cphremd.gb_energy_backward(*one, scr, up[:1], gb=gb)]
        Eo, *go = oracle.gb_grad(*(a[r].astype(np.float32).astype(np.float64) for a in (x, q, rho)),
                                 s.screen.astype(np.float32).astype(np.float64), oracle.GBParams(rgbmax=rgbmax))
        for e in (E[r], E1):
            assert abs(e - Eo) <= 1e-6 * abs(Eo), (r, e, Eo)
        for a, b, o in zip(g, g1, go):
            assert _rel(a[r], o) <= 1e-5 and _rel(b, o) <= 1e-5
            assert _rel(a[r], b) <= 2e-6


@pytest.mark.parametrize("n,n_rep", [(512, 1), (513, 1), (544, 2), (577, 1), (801, 3), (33, 24000), (65, 6000)])
def test_symmetric_kernels_at_tile_edges(n, n_rep):
    """Past the cluster kernel's sizes: work items of 2 j-tiles (a few replicas
    of over 512 atoms) and of 8 or 16 (many small ones); 512 is its largest."""
    import torch
    s, x, q, rho = synth.config_c5(n_rep=n_rep, n=n, seed=70 + n)
    t = [torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in (x, q, rho)]
    scr = torch.tensor(s.screen, dtype=torch.float32, device="cuda:0")
    up = torch.ones(n_rep, dtype=torch.float64, device="cuda:0")
    E = cphremd.gb_energy(*t, scr).cpu().numpy()
    g = [a.cpu().numpy().astype(np.float64) for a in cphremd.gb_energy_backward(*t, scr, up)]
    for r in {0, n_rep - 1}:
        Eo, *go = oracle.gb_grad(*(a[r].astype(np.float32).astype(np.float64) for a in (x, q, rho)),
                                 s.screen.astype(np.float32).astype(np.float64))
        assert abs(E[r] - Eo) <= 1e-6 * abs(Eo), (r, E[r], Eo)
        for a, o in zip(g, go):
            assert _rel(a[r], o) <= 1e-5
