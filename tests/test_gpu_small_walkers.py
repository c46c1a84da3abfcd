"""Whole MD steps of small walkers in one cluster launch (FP32, one warp per
atom): forces against the oracle at the edges of the kernel's sizes, steps
against the FP64 engine, and the same bits however the steps are split into
launches, with titration sweeps, exchanges and constraints in between."""
import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _engine(s, W, prec=cphremd.PREC_FP32, **kw):
    grid = synth.Grid(np.linspace(-0.3, -0.1, W) if W > 1 else np.array([-0.2]), np.array([7.0]), np.array([300.0]),
                      np.zeros(W, np.int32), order=("E",))
    eng = cphremd.init_system([s], grid, seed=5, precision=prec, **kw)
    if prec == cphremd.PREC_FP32:
        eng.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    return eng


@pytest.mark.parametrize("kappa,rgbmax", [(0.0, 0.0), (0.1, 9.0)])
@pytest.mark.parametrize("n", [17, 33, 160, 161, 256, 257, 512, 513])
def test_forces_and_steps(n, kappa, rgbmax):
    s = synth.make_system(n, 60 + n, n_ph=0)
    gb = cphremd.default_gb()
    gb.kappa, gb.rgbmax = kappa, rgbmax
    terms, Fo, Ro, _ = oracle.energy(oracle.OSystem(s), s.x, s.q, oracle.GBParams(kappa=kappa, rgbmax=rgbmax))
    a = _engine(s, 2, gb=gb)
    a.evaluate()
    for w in range(2):
        sl = a.walker_slice(w)
        F, R = a.forces()[sl], a.born_radii()[sl]
        assert np.sqrt(((F - Fo) ** 2).mean()) <= 1e-5 * np.sqrt((Fo ** 2).mean())
        np.testing.assert_allclose(R, Ro, rtol=5e-6)
        iu = np.triu_indices(n, 1)
        d = np.linalg.norm(s.x[iu[0]] - s.x[iu[1]], axis=1)
        scale = np.abs(terms)  # a cancelling sum is held to the sum of its pairs' magnitudes
        scale[1] = 332.05 * np.sum(np.abs(s.q[iu[0]] * s.q[iu[1]]) / d)
        scale[5] = scale[:5].sum()
        assert (np.abs(a.energies()[w] - terms) <= 1e-6 * scale + 1e-9).all()
    # four steps against FP64: displacement and velocity to the force bar
    b = _engine(s, 2, cphremd.PREC_FP64, gb=gb)
    x0 = b.positions()
    for e in (a, b):
        e.step_replicas(4)
        e.status()
    for u, v in ((a.velocities(), b.velocities()), (a.positions() - x0, b.positions() - x0)):
        assert np.sqrt(((u - v) ** 2).mean()) <= 1e-5 * np.sqrt((v ** 2).mean())


@pytest.mark.parametrize("shake", [False, True])
def test_the_split_into_launches_changes_no_bit(shake):
    """24 steps with sweeps every 4 (pH) and 6 (redox) and an attempt every 8:
    one call, single steps, one launch per replica, and FP64 for the counts."""
    s = synth.make_system(150, 9, n_ph=2)
    if shake:
        s = synth.add_hydrogens(s, 0.5, 9)
    kw = dict(mc_ph_every=4, mc_redox_every=6, exchange_every=8, shake=shake, shake_tol=1e-8)
    out = []
    for how in ("one", "single", "replica"):
        e = _engine(s, 4, **kw)
        if how == "replica":
            e.set_launch_mode(cphremd.LAUNCH_PER_REPLICA)
        for n in [24] if how != "single" else [1] * 24:
            e.run(n)
        e.status()
        out.append([e.positions(), e.velocities(), e.site_states(), e.condition_map(), e.accept_stats(), e.visits(),
                    e.occupancy()[0], e.forces(), e.born_radii(), e.energies()])
    for o in out[1:]:
        for u, v in zip(out[0], o):
            np.testing.assert_array_equal(u, v)
    d = _engine(s, 4, cphremd.PREC_FP64, **kw)
    d.run(24)
    np.testing.assert_array_equal(out[0][5].sum(), d.visits().sum())
    np.testing.assert_array_equal(out[0][6].sum(), d.occupancy()[0].sum())
