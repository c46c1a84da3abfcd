"""The GB energy's pair kernels at the edges of their tiles: near pairs (half
of the warp steps of these small chains meet one) evaluated apart from the tile
loop, with work items of 2 j-tiles (one replica) and of 16 (1300 replicas)."""
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
    """Both item sizes against the oracle, at the repository's bars (energy
    1e-6, gradients 1e-5 RMS relative); the two sum the same FP32 pair terms in
    another order, so they agree to a few roundings (2e-6)."""
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
