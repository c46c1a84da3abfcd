"""Without an offset a Born radius is infinite where the tanh of its rational form
has saturated.  Such atoms have no GB energy of their own or with any other."""
import numpy as np
import pytest

from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _gb(kappa):
    gb = cphremd.default_gb()
    gb.offset, gb.alpha, gb.kappa = 0.0, 1000.0, kappa  # every atom's tanh is 1
    return gb


@pytest.mark.parametrize("kappa", [0.0, 0.1])
@pytest.mark.parametrize("n", [237, 600, 2003])
def test_gb_energy(n, kappa):
    import torch
    s, x, q, rho = synth.config_c5(n_rep=2, n=n, seed=5)
    t = [torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in (x, q, rho)]
    scr = torch.tensor(s.screen, dtype=torch.float32, device="cuda:0")
    assert cphremd.gb_energy(*t, scr, gb=_gb(kappa)).tolist() == [0.0, 0.0]
    _, dq, _ = cphremd.gb_energy_backward(*t, scr, torch.ones(2, dtype=torch.float64, device="cuda:0"), gb=_gb(kappa))
    assert not dq.any()


@pytest.mark.parametrize("kappa", [0.0, 0.1])
@pytest.mark.parametrize("n", [150, 600, 2003])
@pytest.mark.parametrize("prec,shape", [(cphremd.PREC_FP32, 0), (cphremd.PREC_FP32, 1), (cphremd.PREC_FP64, None)])
def test_engine(n, prec, shape, kappa):
    s = synth.make_system(n, 3, n_ph=2)
    grid = synth.Grid(np.array([-0.2]), np.array([7.0]), np.array([300.0]), np.zeros(1, np.int32), order=("E",))
    e = cphremd.init_system([s], grid, seed=1, precision=prec, gb=_gb(kappa))
    if shape is not None:
        e.set_tile_shape(0, shape)
    e.evaluate()
    t = e.energies()[0]
    assert t[0] == 0.0 and np.isfinite(t).all() and np.isinf(e.born_radii()).all()
    e.mc_titrate()
    assert all(np.isfinite(r.dU) for r in e.mc_records())
