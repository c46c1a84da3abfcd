"""A Born radius that is not a number stays one: short functions and clamps hide nothing."""
import numpy as np
import pytest

from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 600])
@pytest.mark.parametrize("prec,shape", [(cphremd.PREC_FP32, 0), (cphremd.PREC_FP32, 1), (cphremd.PREC_FP64, None)])
def test_radii_that_are_not_numbers(prec, shape, n):
    """A coefficient of the rational form that is not a number (set-up takes it)."""
    build.build()
    s = synth.make_system(n, 3, n_ph=0)
    grid = synth.Grid(np.array([-0.2]), np.array([7.0]), np.array([300.0]), np.zeros(1, np.int32), order=("E",))
    gb = cphremd.default_gb()
    gb.gamma = float("nan")
    e = cphremd.init_system([s], grid, seed=1, precision=prec, gb=gb)
    if shape is not None:
        e.set_tile_shape(0, shape)
    e.evaluate()
    assert np.isnan(e.born_radii()).all()
