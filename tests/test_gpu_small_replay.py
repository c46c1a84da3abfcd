"""Captured schedule periods of the small-walker kernel (cluster launches with
programmatic attributes between sweeps and exchanges) against direct launches."""
import numpy as np
import pytest

from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


@pytest.mark.parametrize("shake", [False, True])
def test_replayed_schedule_periods_change_no_bit(shake):
    """A period of 24 steps replays as a captured graph from step 1 on: two whole
    periods and some steps in one call, one launch per replica, and single
    steps, which never replay."""
    s = synth.make_system(110, 9, n_ph=2)
    if shake:
        s = synth.add_hydrogens(s, 0.5, 9)
    grid = synth.Grid(np.linspace(-0.3, -0.1, 4), np.array([7.0]), np.array([300.0]), np.zeros(4, np.int32), order=("E",))
    out = []
    for how in ("one", "single", "replica"):
        e = cphremd.init_system([s], grid, seed=5, mc_ph_every=4, mc_redox_every=6, exchange_every=8, shake=shake,
                                shake_tol=1e-8)
        e.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
        assert e.time_passes(reps=1)[2] == 0
        if how == "replica":
            e.set_launch_mode(cphremd.LAUNCH_PER_REPLICA)
        for n in [1 + 2 * 24 + 5] if how != "single" else [1] * 54:
            e.run(n)
        e.status()
        out.append([e.positions(), e.velocities(), e.site_states(), e.condition_map(), e.accept_stats(), e.visits(),
                    e.occupancy()[0], e.forces(), e.born_radii(), e.energies()])
    for o in out[1:]:
        for u, v in zip(out[0], o):
            np.testing.assert_array_equal(u, v)
