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


@pytest.mark.parametrize("n,W,shake,cluster", [
    (160, 1, False, True), (160, 8, False, True), (120, 28, False, True), (237, 14, False, True),
    (480, 1, False, False), (360, 8, False, False), (237, 1, False, False), (80, 20, False, False),
    (160, 45, False, True), (160, 64, False, False), (120, 384, False, False), (128, 4, True, True), (128, 60, True, True),
    (84, 128, True, False)])
def test_cluster_launches_only_where_they_pay(n, W, shake, cluster):
    """One walker holds eight SMs: many of them, or large ones, run the separate
    launches.  cph_time_passes times what the steps run (the cluster kernel
    is one launch), and the autotuner keeps to the rule."""
    s = synth.add_hydrogens(synth.make_system(n, 8, n_ph=2), 0.55, 8) if shake else synth.make_system(n, 1, n_ph=2)
    e = cphremd.init_system([s], _grid(W), seed=3, shake=shake, shake_tol=1e-8)
    e.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    ms = e.time_passes(reps=2)
    assert ms[0] > 0 and (ms[1] == ms[2] == 0) == cluster
    e.autotune()
    if cluster:
        assert e.tile_shapes()[0] == cphremd.SHAPE_WARP_PER_ATOM


@pytest.mark.parametrize("n", [140, 200, 250])
def test_constrained_walkers_of_all_sizes(n):
    """With hydrogens 262 to 458 atoms: more than one atom to a warp.  Forces
    against the oracle and four steps against FP64, at the repository's bars."""
    import oracle
    s = synth.add_hydrogens(synth.make_system(n, 8, n_ph=2), 0.55, 8)
    o = oracle.OSystem(s)
    o.bond_k[(s.mass[s.bonds] < 2.0).any(axis=1)] = 0.0  # a constrained bond has no harmonic term
    q = s.q.copy()
    for t in s.sites:
        q[t.atoms] = t.q[t.init_state]
    _, Fo, Ro, _ = oracle.energy(o, s.x, q, oracle.GBParams())
    a = cphremd.init_system([s], _grid(2), seed=5, shake=True, shake_tol=1e-8)
    a.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
    assert a.time_passes(reps=1)[2] == 0
    a.evaluate()
    sl = a.walker_slice(1)
    np.testing.assert_allclose(a.born_radii()[sl], Ro, rtol=5e-6)
    F = a.forces()[sl]
    assert np.sqrt(((F - Fo) ** 2).mean()) <= 1e-5 * np.sqrt((Fo ** 2).mean())
    b = cphremd.init_system([s], _grid(2), seed=5, precision=cphremd.PREC_FP64, shake=True, shake_tol=1e-8)
    for e in (a, b):
        e.step_replicas(4)
        e.status()
    v, w = a.velocities(), b.velocities()
    assert np.sqrt(((v - w) ** 2).mean()) <= 1e-5 * np.sqrt((w ** 2).mean())


def _captured_kernels(call):
    """Nodes that call(stream) puts on a capturing stream."""
    import ctypes as C

    import torch
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    h, graph, n = C.c_void_p(st.cuda_stream), C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0  # thread-local
    try:
        call(st.cuda_stream)
    finally:
        assert cu.cuStreamEndCapture(h, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    cu.cuGraphDestroy(graph)
    return n.value


def test_long_runs_stay_divided_into_launches():
    """At most 1000 steps to a launch, and the same bits however a run is cut."""
    s = synth.make_system(60, 1, n_ph=2)
    kw = dict(mc_ph_every=0, mc_redox_every=0, exchange_every=0)

    def engine():
        e = cphremd.init_system([s], _grid(2), seed=3, **kw)
        e.set_tile_shape(0, cphremd.SHAPE_WARP_PER_ATOM)
        return e

    a, b, c = engine(), engine(), engine()
    assert _captured_kernels(lambda st: a.step_replicas(2500, stream=st)) == 4  # 1000, 1000, 500, and the counter's
    assert _captured_kernels(lambda st: a.run(2001, stream=st)) == 4
    a = engine()
    a.step_replicas(2500)
    for n in (700, 1000, 800):
        b.step_replicas(n)
    c.run(2500)
    for e in (a, b, c):
        e.status()
        assert e.get_step() == 2500
    for get in ("positions", "velocities", "forces", "born_radii", "visits"):
        np.testing.assert_array_equal(getattr(a, get)(), getattr(b, get)())
        np.testing.assert_array_equal(getattr(a, get)(), getattr(c, get)())
