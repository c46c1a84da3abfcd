"""FP32 on one warp per atom: an extended molecule keeps the precision of a compact
one, however far from the walker's first atom a pair lies."""
import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


@pytest.mark.parametrize("kappa,rgbmax", [(0.0, 0.0), (0.1, 12.0)])
@pytest.mark.parametrize("n", [1203, 2003])
def test_a_fibre_of_a_thousand_angstrom(n, kappa, rgbmax):
    """The repository's bars: radii 5e-6, forces 1e-5 RMS relative."""
    s = synth.make_system(n, 3, n_ph=0)
    i = np.arange(n)  # zigzag steps of 1.5 A, 1.25 A along the axis
    s.x = np.stack([1.25 * i, 0.7 * (-1.0) ** i, 0.8 * (i % 4 // 2)], 1) + np.array([3.3, -7.7, 11.1])
    s.x += 0.05 * np.random.default_rng(n).standard_normal(s.x.shape)
    gb = cphremd.default_gb()
    gb.kappa, gb.rgbmax = kappa, rgbmax
    grid = synth.Grid(np.array([-0.2]), np.array([7.0]), np.array([300.0]), np.zeros(1, np.int32), order=("E",))
    e = cphremd.init_system([s], grid, seed=1, gb=gb)
    e.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    e.evaluate()
    _, Fo, Ro, _ = oracle.energy(oracle.OSystem(s), s.x, s.q, oracle.GBParams(kappa=kappa, rgbmax=rgbmax))
    np.testing.assert_allclose(e.born_radii(), Ro, rtol=5e-6)
    F = e.forces()
    assert np.sqrt(((F - Fo) ** 2).mean()) <= 1e-5 * np.sqrt((Fo ** 2).mean())
