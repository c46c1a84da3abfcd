"""Which walkers run whole steps in one cluster launch, and what the others keep."""
import numpy as np
import pytest

from oracle.run import shake_clusters
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _grid(W):
    return synth.Grid(np.linspace(-0.3, -0.1, W) if W > 1 else np.array([-0.2]), np.array([7.0]), np.array([300.0]),
                      np.zeros(W, np.int32), order=("E",))


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("tol", [1e-14, 1e-15])
def test_constraints_settle_at_tight_tolerances(tol, seed):
    """|d^2 - d0^2| <= 2 tol d0^2 as SHAKE's FP64 sees it; 2e-15 for this test's own
    evaluation of d^2 (some roundings of 1e-16 each way)."""
    s = synth.add_hydrogens(synth.make_system(128, 8 + seed, n_ph=2), 0.55, 8)
    e = cphremd.init_system([s], _grid(4), seed=seed, shake=True, shake_tol=tol)
    e.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    for _ in range(10):
        e.run(10)
        e.status()
    for w in range(4):
        x = e.positions()[e.walker_slice(w)]
        for heavy, hs in shake_clusters(s):
            for h, d0 in hs:
                d2 = ((x[heavy] - x[h]) ** 2).sum()
                assert abs(d2 - d0 * d0) <= (2 * tol + 2e-15) * d0 * d0
