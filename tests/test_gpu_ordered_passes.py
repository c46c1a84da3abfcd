"""The pair passes over every ordered pair at the edges of their batches and
tiles: FP32 (systems too large for the small-walker kernel) and FP64 with one
and with four warps per atom; and titration sweeps that accept more atoms than
they keep in shared memory, or that have more sites than a block has threads."""
import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth

pytestmark = pytest.mark.gpu

# (force RMS, energy, Born radius) relative bars of each mode
BARS = {cphremd.PREC_FP32: (1e-5, 1e-6, 5e-6), cphremd.PREC_FP64: (1e-10, 1e-10, 1e-11)}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _grid(W):
    return synth.Grid(np.linspace(-0.3, -0.1, W), np.array([7.0]), np.array([300.0]), np.zeros(W, np.int32), order=("E",))


def _check(n, prec, W, kappa, rgbmax):
    s = synth.make_system(n, 80 + n, n_ph=0)
    gb = cphremd.default_gb()
    gb.kappa, gb.rgbmax = kappa, rgbmax
    terms, Fo, Ro, _ = oracle.energy(oracle.OSystem(s), s.x, s.q, oracle.GBParams(kappa=kappa, rgbmax=rgbmax))
    iu = np.triu_indices(n, 1)
    d = np.linalg.norm(s.x[iu[0]] - s.x[iu[1]], axis=1)
    scale = np.abs(terms)  # a cancelling sum is held to the sum of its pairs' magnitudes
    scale[1] = 332.05 * np.sum(np.abs(s.q[iu[0]] * s.q[iu[1]]) / d)
    scale[5] = scale[:5].sum()
    eng = cphremd.init_system([s], _grid(W), seed=2, gb=gb, precision=prec)
    if prec == cphremd.PREC_FP32:
        eng.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    eng.evaluate()
    eng.status()
    bf, be, br = BARS[prec]
    for w in {0, W - 1}:
        sl = eng.walker_slice(w)
        assert np.sqrt(((eng.forces()[sl] - Fo) ** 2).mean()) <= bf * np.sqrt((Fo ** 2).mean())
        np.testing.assert_allclose(eng.born_radii()[sl], Ro, rtol=br)
        assert (np.abs(eng.energies()[w] - terms) <= be * scale + 1e-9).all()


@pytest.mark.parametrize("kappa,rgbmax", [(0.0, 0.0), (0.0, 9.0), (0.1, 0.0), (0.1, 9.0)])
@pytest.mark.parametrize("n,W", [(513, 1), (640, 3), (643, 2), (1025, 1), (1153, 1)])
def test_fp32_at_batch_edges(n, W, kappa, rgbmax):
    _check(n, cphremd.PREC_FP32, W, kappa, rgbmax)


@pytest.mark.parametrize("kappa,rgbmax", [(0.0, 0.0), (0.1, 9.0)])
@pytest.mark.parametrize("many", [False, True])  # four warps per atom up to 2048 atoms, else one
@pytest.mark.parametrize("n", [17, 31, 33, 128, 129, 160, 257])
def test_fp64_at_tile_edges(n, many, kappa, rgbmax):
    _check(n, cphremd.PREC_FP64, 2048 // n + 1 if many else 1, kappa, rgbmax)


@pytest.mark.parametrize("prec", [cphremd.PREC_FP32, cphremd.PREC_FP64])
@pytest.mark.parametrize("n_ph,atoms", [(32, (56, 64)), (262, (6, 6))])
def test_sweeps_that_accept_many_sites(n_ph, atoms, prec):
    """dU and decisions against the oracle's full recomputation: 2e-6 relative and
    1e-4 kcal/mol (FP32), 1e-9 (FP64); a decision within the exponent's error bound
    ends a walker's comparison, as the later sites see other charges."""
    fp64 = prec == cphremd.PREC_FP64
    s = synth.make_system(2200, 7, n_ph=n_ph, ph_atoms=atoms)
    grid = synth.Grid(np.array([-0.2]), np.array([1.0]), np.array([300.0]), np.zeros(1, np.int32), order=("E",))
    eng = cphremd.init_system([s], grid, seed=11, precision=prec)
    eng.mc_titrate(cphremd.MC_BOTH)
    recs = eng.mc_records()
    W = oracle.Walkers([s], grid, seed=11, gb=oracle.GBParams())
    oracle.mc_sweep(W, 0, "ph", 0)
    oracle.mc_sweep(W, 0, "redox", 0)
    taken, same = 0, True
    for (w, k, a, b, dU, x, lnu, acc) in W.mc_log:
        r = recs[k]
        assert (r.walker, r.site, r.frm, r.to, r.lnu) == (w, k, a, b, lnu)
        if same:
            assert abs(r.dU - dU) <= (1e-9 if fp64 else 2e-6) * max(1.0, abs(dU)) + (1e-9 if fp64 else 1e-4), k
            same = abs(lnu - x) > (1e-9 if fp64 else 2e-4) * max(1.0, abs(x))
        if same:
            assert bool(r.accepted) == bool(acc), k
            taken += len(s.sites[k].atoms) if acc else 0
    assert taken > 768 or n_ph > 256  # the sweep's shared memory holds 768 atoms, its block 256 threads
