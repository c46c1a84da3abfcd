"""What a user of this framework has it do, as timed cases.

Engine cases go through ``cphremd.init_system`` / ``Engine`` (molecular dynamics
with titration and exchanges, single sweeps and evaluations), the others through
``cphremd.gb_energy`` and ``cphremd.GBEnergy`` (energies and gradients of GPU
tensors).  The molecules are the seeded chains of ``synth``: one molecule per
size, as a user's program has one molecule, and the seed gives its conformation,
charges and velocities.

Results of the FP32 mode carry FP32 precision and are kept as float32, the way
trajectory files and float32 training programs hold them; the FP64 mode's are
kept as float64.
"""
import functools
import math

import numpy as np
import torch

from paper_1809_07726_gb300 import cphremd, synth

KB = 0.0019872041  # kcal / (mol K)
ACCEL = 418.4      # (kcal/mol/A)/amu -> A/ps^2
COULOMB = 332.0522173
MAX_PAIRS = 128 * 8000 * 7999 // 2  # unordered pairs of the largest gradient case


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The smallest call: the GB energy of one conformation of the paper's
        # system size (237 atoms), as in scoring or a minimiser's line search.
        dict(name="gb_1x237", kind="energy", n_rep=1, n=237),
        # Energy and gradient of a small batch of ragged conformations: one
        # step of a force-field or charge fit.
        dict(name="grad_16x1203", kind="grad", n_rep=16, n=1203),
        # The differentiation workload: 128 replicas of an 8000-atom protein.
        dict(name="grad_128x8000", kind="grad", n_rep=128, n=8000),
        # Plain C(pH,E)MD of one 160-atom heme peptide in FP64: 100 steps, a
        # titration sweep every 10.
        dict(name="md_fp64_1x160", kind="md", n=160, walkers=1, fp64=True, steps=100, shake=False, dims=1),
        # E-REMD of the same peptide, 8 replicas in FP32: one exchange period.
        dict(name="eremd_8x160", kind="md", n=160, walkers=8, fp64=False, steps=100, shake=False, dims=1),
        # The peptide with hydrogens (246 atoms), bonds to hydrogen constrained.
        dict(name="shake_4x246", kind="md", n=246, walkers=4, fp64=False, steps=50, shake=True, dims=1),
        # One replica of a 2000-atom protein: the plain MD run of a single
        # molecule, which one replica alone has to spread over the GPU.
        dict(name="md_1x2003", kind="md", n=2003, walkers=1, fp64=False, steps=20, shake=False, dims=1),
        # E,pH-REMD: 8 x 8 replicas of a 2400-atom protein, one titration period.
        dict(name="ephremd_64x2400", kind="md", n=2400, walkers=64, fp64=False, steps=10, shake=False, dims=2),
        # The titration sweep alone (both kinds) over the same 64 replicas.
        dict(name="mc_64x2400", kind="mc", n=2400, walkers=64),
        # MD steps of the 3D E,T,pH workload between two attempts: 384 replicas
        # of 500, 2000 and 8000 atoms in one engine.
        dict(name="remd3d_384", kind="md3d", steps=8),
        # Energies and forces with the other options of the GB model: OBC
        # model II, salt and a Born-radius cutoff.
        dict(name="eval_salt_8x1203", kind="eval", n=1203, walkers=8, fp64=False, kappa=0.1, rgbmax=12.0, obc2=True),
        # FP64 energies and forces of two conformations: reference values.
        dict(name="eval_fp64_2x1203", kind="eval", n=1203, walkers=2, fp64=True, kappa=0.0, rgbmax=0.0, obc2=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "grad", "md", "md", "mc", "eval"])
    if kind in ("energy", "grad"):
        n = _log(rng, 60, 6000)
        return dict(kind=kind, n_rep=_log(rng, 1, max(1, min(128, MAX_PAIRS // (n * n)))), n=n)
    if kind == "mc":
        return dict(kind="mc", n=_log(rng, 300, 3000), walkers=_log(rng, 2, 64))
    fp64 = rng.random() < 0.3
    if kind == "eval":
        return dict(kind="eval", n=_log(rng, 120, 1500 if fp64 else 4000), walkers=_log(rng, 1, 6 if fp64 else 16),
                    fp64=fp64, kappa=rng.choice([0.0, 0.0, 0.05, 0.1]), rgbmax=rng.choice([0.0, 0.0, 8.0, 12.0]),
                    obc2=rng.random() < 0.3)
    shake = rng.random() < 0.25
    n = _log(rng, 100, 400 if fp64 or shake else 3000)
    return dict(kind="md", n=n, walkers=_log(rng, 1, 4 if fp64 else 32), fp64=fp64,
                steps=_log(rng, 5, 100 if n < 500 else 20), shake=shake, dims=rng.choice([1, 2]))


# ------------------------------------------------------------------ molecules
@functools.lru_cache(maxsize=None)
def _molecule(n, shake=False):
    """The chain of this size: about one pH site per 125 atoms and one redox site."""
    if shake:  # about n atoms once the hydrogens are on
        heavy = max(40, round(n * 128 / 246))
        return synth.add_hydrogens(synth.make_system(heavy, 8, n_ph=2, ph_pka=[4.4, 4.85]), 0.55, 8)
    if n < 400:
        n_ph = 2 if n >= 40 else 0
        return synth.make_system(n, 1, n_ph=n_ph, ph_pka=[4.4, 4.85][:n_ph], n_redox=1 if n >= 40 else 0)
    return synth.make_system(n, 2, n_ph=n // 125, ph_states=(2, 4), ph_atoms=(6, 12))


def _grid(walkers, dims):
    nE = walkers
    if dims == 2:  # the most nearly square E x pH grid
        nE = max(d for d in range(1, int(math.isqrt(walkers)) + 1) if walkers % d == 0)
    npH = walkers // nE
    E = np.linspace(-0.35, -0.05, nE) if nE > 1 else np.array([-0.2])
    pH = 3.5 + 0.5 * np.arange(npH) if npH > 1 else np.array([7.0])
    order = tuple(k for k, m in (("E", nE), ("pH", npH)) if m > 1) or ("E",)
    return synth.Grid(E, pH, np.array([300.0]), np.zeros(walkers, np.int32), order=order)


def _gb(case):
    g = cphremd.default_gb()
    if case.get("obc2"):
        g.alpha, g.beta, g.gamma = 1.0, 0.8, 4.85
    g.kappa, g.rgbmax = case.get("kappa", 0.0), case.get("rgbmax", 0.0)
    return g


def _conformations(systems, grid, seed, width):
    """Every walker's positions, shifted from the molecule's by `width` A, and
    thermal velocities, from the seed."""
    rng = np.random.default_rng(seed)
    mols = [systems[s] for s in grid.system_of_slot]
    x = np.concatenate([m.x for m in mols])
    x = x + width * rng.standard_normal(x.shape)
    m = np.concatenate([m.mass for m in mols])
    v = rng.standard_normal(x.shape) * np.sqrt(KB * 300.0 * ACCEL / m)[:, None]
    return x, v


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    if case["kind"] in ("energy", "grad"):
        m, n_rep, n = _molecule(case["n"]), case["n_rep"], case["n"]
        dev = torch.device("cuda")
        gen = torch.Generator(dev).manual_seed(seed)

        def around(a, width):
            t = torch.tensor(a, dtype=torch.float32, device=dev).expand(n_rep, *a.shape)
            return t + width * torch.randn(t.shape, generator=gen, device=dev)

        st = dict(x=around(m.x, 0.05), q=around(m.q, 0.02), rho=around(m.rho, 0.0),
                  screen=torch.tensor(m.screen, dtype=torch.float32, device=dev))
        if case["kind"] == "grad":
            for k in ("x", "q", "rho"):
                st[k].requires_grad_(True)
        return dict(case=case, **st)
    if case["kind"] == "md3d":
        systems, grid = _config3d()
    else:
        systems = [_molecule(case["n"], case.get("shake", False))]
        grid = _grid(case["walkers"], case.get("dims", 1))
    fp64 = case.get("fp64", False)
    # constrained bonds start at their lengths
    x, v = _conformations(systems, grid, seed, 0.0 if case.get("shake") else 0.03)
    eng = cphremd.init_system(systems, grid, seed=seed, gb=_gb(case), shake=case.get("shake", False), shake_tol=1e-8,
                              precision=cphremd.PREC_FP64 if fp64 else cphremd.PREC_FP32)
    eng.set_positions(x)
    eng.set_velocities(v)
    if not fp64:
        eng.autotune()
    return dict(case=case, eng=eng, dtype=np.float64 if fp64 else np.float32)


@functools.lru_cache(maxsize=None)
def _config3d():
    return synth.config_c4()


# ------------------------------------------------------------------ run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "energy":
        E = cphremd.gb_energy(state["x"], state["q"], state["rho"], state["screen"])
        return E.float()
    if kind == "grad":
        x, q, rho = state["x"], state["q"], state["rho"]
        E = cphremd.GBEnergy.apply(x, q, rho, state["screen"])
        g = torch.autograd.grad(E.sum(), (x, q, rho))
        return [E.detach().float(), *g]
    eng, dt = state["eng"], state["dtype"]
    if kind == "eval":
        eng.evaluate()
        return [eng.energies().astype(dt, copy=False), eng.forces().astype(dt, copy=False),
                eng.born_radii().astype(dt, copy=False)]
    if kind == "mc":
        eng.mc_titrate()
        return [eng.site_states(), eng.charges()]
    if kind == "md3d":
        eng.step_replicas(case["steps"])
    else:
        eng.run(case["steps"])
    return [eng.positions().astype(dt, copy=False), eng.velocities().astype(dt, copy=False), eng.site_states(),
            eng.condition_map()]


# ------------------------------------------------------------------ work
def _sizes(case):
    """(atoms per walker, walkers) of each molecule."""
    if case["kind"] == "md3d":
        return [(500, 128), (2000, 128), (8000, 128)]
    if case["kind"] in ("energy", "grad"):
        return [(case["n"], case["n_rep"])]
    return [(_molecule(case["n"], case.get("shake", False)).n, case["walkers"])]


def work(case):
    """Per unordered pair: Born radii 23, GB + Coulomb + LJ 40, chain rule 31
    multiply-adds or other operations (about 1.5 flops each); the GB energy's
    pair sum 20 and its adjoint 77.  Bytes: the state read and written once."""
    atoms = sum(n * w for n, w in _sizes(case))
    pairs = sum(w * n * (n - 1) / 2 for n, w in _sizes(case))
    kind = case["kind"]
    if kind == "energy":
        return dict(bytes=24.0 * atoms, flops=1.5 * pairs * (23 + 20))
    if kind == "grad":
        return dict(bytes=44.0 * atoms, flops=1.5 * pairs * (23 + 20 + 77))
    if kind == "mc":  # Born radii, and each site's atoms (about 9) against all atoms
        sites = case["walkers"] * len(_molecule(case["n"]).sites)
        return dict(bytes=56.0 * atoms, flops=1.5 * (pairs * 23 + sites * 9 * case["n"] * 20))
    if kind == "eval":
        return dict(bytes=96.0 * atoms, flops=1.5 * pairs * 94)
    return dict(bytes=120.0 * atoms * case["steps"], flops=1.5 * pairs * 94 * case["steps"])


# ------------------------------------------------------------------ exact
def _descreening(r, rt, s, rc):
    """The pairwise descreening integral (Hawkins, Cramer and Truhlar), with shells beyond rc left out."""
    U = torch.clamp(r + s, max=rc)
    L = torch.maximum(rt, (r - s).abs())
    h = 1 / L - 1 / U + (r - s * s / r) / 4 * (1 / U**2 - 1 / L**2) + torch.log(L / U) / (2 * r)
    top = torch.clamp(s - r, max=rc)
    inside = rt < top
    return torch.where(L < U, h, 0.0) + torch.where(inside, 2 * (1 / rt - 1 / torch.where(inside, top, 1.0)), 0.0)


class _Exact:
    """One conformation in 64 bits: Born radii, energies and gradients, rows of
    atoms against all atoms at a time."""

    def __init__(self, x, q, rho, screen, gb, lj=None, excl=None):
        self.x, self.q, self.rho = (t.detach().clone().requires_grad_(True) for t in (x, q, rho))
        self.screen, self.gb, self.lj, self.excl = screen, gb, lj, excl
        self.n = x.shape[0]
        self.rc = gb.rgbmax if gb.rgbmax > 0 else math.inf
        self.rows = [(a, min(self.n, a + max(1, 20_000_000 // self.n))) for a in range(0, self.n, max(1, 20_000_000 // self.n))]

    def r2(self, a, b):
        return sum((self.x[a:b, None, c] - self.x[None, :, c]) ** 2 for c in range(3))

    def other(self, a, b):
        """1 where the atoms differ."""
        m = torch.ones(b - a, self.n, dtype=torch.float64, device=self.x.device)
        i = torch.arange(a, b, device=self.x.device)
        m[i - a, i] = 0
        return m

    def psi(self, a, b):
        o = self.other(a, b)
        r = torch.sqrt(self.r2(a, b) + (1 - o))
        rt = self.rho - self.gb.offset
        return rt[a:b] / 2 * (o * _descreening(r, rt[a:b, None], (self.screen * rt)[None, :], self.rc)).sum(1)

    def radii(self, psi):
        g = self.gb
        th = torch.tanh(g.alpha * psi - g.beta * psi**2 + g.gamma * psi**3)
        return 1 / (1 / (self.rho - g.offset) - th / self.rho)

    def born(self):
        with torch.no_grad():
            return torch.cat([self.psi(a, b) for a, b in self.rows])

    def pair_energies(self, a, b, R):
        g = self.gb
        r2 = self.r2(a, b)
        RR = R[a:b, None] * R[None, :]
        f = torch.sqrt(r2 + RR * torch.exp(-r2 / (4 * RR)))
        tau = 1 / g.eps_in - (torch.exp(-g.kappa * f) if g.kappa else 1.0) / g.eps_out
        qq = self.q[a:b, None] * self.q[None, :]
        E = [-0.5 * COULOMB * (tau * qq / f).sum()]
        if self.lj is not None:
            o = self.other(a, b)
            r2 = r2 + (1 - o)
            ei, ej = self.excl
            k = (ei >= a) & (ei < b)
            o[ei[k] - a, ej[k]] = 0
            E.append(0.5 * COULOMB / g.eps_in * (o * qq / torch.sqrt(r2)).sum())
            sig, eps = self.lj
            sr6 = ((sig[a:b, None] + sig[None, :]) / 2) ** 6 / r2**3
            E.append(2.0 * (o * torch.sqrt(eps[a:b, None] * eps[None, :]) * (sr6 * sr6 - sr6)).sum())
        return E

    def solve(self, gradients=True, bonded=None):
        """(energies, radii, gradients of x, q and rho)."""
        psi = self.born().requires_grad_(True)
        R0 = self.radii(psi)
        R = R0.detach().requires_grad_(True)
        total = None
        for a, b in self.rows:
            with torch.set_grad_enabled(gradients):
                E = self.pair_energies(a, b, R)
            if gradients:
                sum(E).backward()
            E = torch.stack([e.detach() for e in E])
            total = E if total is None else total + E
        if bonded is not None:
            E = bonded(self.x)
            sum(E).backward()
            total = torch.cat([total, torch.stack([e.detach() for e in E])])
        if gradients:
            R0.backward(R.grad)  # dE/dpsi, and rho at fixed psi
            for a, b in self.rows:
                (self.psi(a, b) * psi.grad[a:b]).sum().backward()
        return total, R.detach(), (self.x.grad, self.q.grad, self.rho.grad)


def _bonded(m, dev):
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    bk, br, ak, at = t(m.bond_k), t(m.bond_r0), t(m.angle_k), t(m.angle_t0)
    b, a = torch.tensor(m.bonds, device=dev).long(), torch.tensor(m.angles, device=dev).long()

    def energies(x):
        r = (x[b[:, 0]] - x[b[:, 1]]).norm(dim=1)
        u, v = x[a[:, 0]] - x[a[:, 1]], x[a[:, 2]] - x[a[:, 1]]
        th = torch.acos((u * v).sum(1) / (u.norm(dim=1) * v.norm(dim=1)))
        return [(bk * (r - br) ** 2).sum(), (ak * (th - at) ** 2).sum()]

    return energies


def _exclusions(m, dev):
    """Ordered pairs one or two bonds apart."""
    nb = [set() for _ in range(m.n)]
    for i, j in m.bonds:
        nb[int(i)].add(int(j))
        nb[int(j)].add(int(i))
    p = {(i, k) for i in range(m.n) for j in nb[i] for k in (nb[j] | {j}) if k != i}
    e = torch.tensor(sorted(p), device=dev).long().reshape(-1, 2)
    return e[:, 0], e[:, 1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "mc":
        return None  # the outcomes of a random sweep: whole numbers and table values
    if kind in ("md", "md3d"):
        return None  # a trajectory: a long integration that plain torch would take minutes for
    st = prepare(case, seed) if kind in ("energy", "grad") else None
    dev = torch.device("cuda")
    gb = _gb(case)
    if kind in ("energy", "grad"):
        E, g = [], ([], [], [])
        for r in range(case["n_rep"]):
            t, _, grads = _Exact(st["x"][r].double(), st["q"][r].double(), st["rho"][r].double(),
                                 st["screen"].double(), gb).solve(kind == "grad")
            E.append(t[0])
            for k in range(3):
                g[k].append(grads[k])
        if kind == "energy":
            return torch.stack(E)
        return [torch.stack(E), *(torch.stack(v) for v in g)]
    m, W = _molecule(case["n"]), case["walkers"]
    x, _ = _conformations([m], _grid(W, 1), seed, 0.03)
    t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    q = m.q.copy()
    for s in m.sites:
        q[s.atoms] = s.q[s.init_state]
    E, F, R = [], [], []
    bonded, excl = _bonded(m, dev), _exclusions(m, dev)
    for xw in x.reshape(W, m.n, 3):
        e, r, (gx, _, _) = _Exact(t(xw), t(q), t(m.rho), t(m.screen), gb, (t(m.sigma), t(m.eps)), excl).solve(True, bonded)
        E.append(torch.cat([e, e.sum()[None]]))
        F.append(-gx)
        R.append(r)
    return [torch.stack(E), torch.cat(F), torch.cat(R)]
