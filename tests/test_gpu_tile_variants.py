"""The FP32 pair passes at the edges of their tiles in each form that a grid's
size selects: four CTAs to a work item (one walker) or one (1300 walkers), near
pairs queued, and one warp per atom from the staged operands."""
import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu

FORCE_RMS, ENERGY_REL, R_REL = 1e-5, 1e-6, 5e-6  # the engine's bars


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


@pytest.mark.parametrize("kappa,rgbmax", [(0.0, 0.0), (0.1, 9.0)])
@pytest.mark.parametrize("n", [33, 64, 129, 257, 1025])
def test_pair_passes_at_tile_edges(n, kappa, rgbmax):
    s = synth.make_system(n, 40 + n, n_ph=0)
    gb = cphremd.default_gb()
    gb.kappa, gb.rgbmax = kappa, rgbmax
    terms, Fo, Ro, _ = oracle.energy(oracle.OSystem(s), s.x, s.q, oracle.GBParams(kappa=kappa, rgbmax=rgbmax))
    # a term that cancels is held to the sum of its pairs' magnitudes (FP32 fixes
    # each pair to ~1e-7 of itself): Coulomb, and with it the total
    iu = np.triu_indices(n, 1)
    d = np.linalg.norm(s.x[iu[0]] - s.x[iu[1]], axis=1)
    scale = np.abs(terms)
    scale[1] = 332.05 * np.sum(np.abs(s.q[iu[0]] * s.q[iu[1]]) / d)
    scale[5] = scale[:5].sum()
    for W, shape in ((1, cphremd.SHAPE_SYMMETRIC), (1, cphremd.SHAPE_WARP_PER_ATOM),
                     (1300 if n < 1000 else 70, cphremd.SHAPE_SYMMETRIC)):
        grid = synth.Grid(np.linspace(-0.3, -0.1, W), np.array([7.0]), np.array([300.0]), np.zeros(W, np.int32),
                          order=("E",))
        eng = cphremd.init_system([s], grid, seed=2, gb=gb)
        eng.set_tile_shape(0, shape)
        eng.evaluate()
        eng.status()
        F, R, E = eng.forces(), eng.born_radii(), eng.energies()
        for w in {0, W - 1}:
            sl = eng.walker_slice(w)
            assert np.sqrt(((F[sl] - Fo) ** 2).mean()) <= FORCE_RMS * np.sqrt((Fo ** 2).mean()), (W, shape, w)
            np.testing.assert_allclose(R[sl], Ro, rtol=R_REL)
            for t in range(6):
                assert abs(E[w][t] - terms[t]) <= ENERGY_REL * scale[t] + 1e-9, (W, shape, t, E[w][t], terms[t])
