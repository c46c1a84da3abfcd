"""Thread-block-cluster kernels: a CTA may touch another CTA's shared memory only
once that CTA has started, which a cluster barrier establishes.  Nothing else in a
kernel does, and a run need not show the lack of it, so the order is read off the
source; the sizes at which it matters most (CTAs without an atom, a few
instructions before the first store) run against the oracle."""
import os
import re

import numpy as np
import pytest

import oracle
from paper_1809_07726_gb300 import build, cphremd, synth


def _kernels():
    """(name, body) of every kernel that maps another CTA's shared memory."""
    out = []
    for f in sorted(os.listdir(build.CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\(", text):
            k = text.index("{", m.end())
            depth, e = 1, k + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[e], 0)
                e += 1
            if "map_shared_rank" in text[k:e]:
                out.append((m.group(1), text[k:e]))
    return out


def test_a_cluster_barrier_precedes_the_first_access_to_another_cta():
    kernels = _kernels()
    assert {"k_gsmall", "k_small"} <= {name for name, _ in kernels}
    for name, body in kernels:
        body = re.sub(r"auto sync = \[&\] \{.*?\};", "", body, flags=re.S)  # the wrapper's definition is no call
        barrier = re.search(r"(?<![\w.:])(?:cl\.)?sync\(\);", body)
        assert barrier and barrier.start() < body.index("map_shared_rank"), name


@pytest.mark.gpu
@pytest.mark.parametrize("n_rep", [1, 40])
@pytest.mark.parametrize("n", [2, 3, 7, 8, 9, 17])
def test_gb_energy_and_gradient_of_few_atoms(n, n_rep):
    """Fewer atoms than a cluster has CTAs, or one or two to a CTA; the
    repository's bars (energy 1e-6, gradients 1e-5 RMS relative)."""
    import torch
    build.build()
    s, x, q, rho = synth.config_c5(n_rep=n_rep, n=n, seed=30 + n)
    t = [torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in (x, q, rho)]
    scr = torch.tensor(s.screen, dtype=torch.float32, device="cuda:0")
    E = cphremd.gb_energy(*t, scr).cpu().numpy()
    g = [a.cpu().numpy().astype(np.float64) for a in
         cphremd.gb_energy_backward(*t, scr, torch.ones(n_rep, dtype=torch.float64, device="cuda:0"))]
    for r in {0, n_rep - 1}:
        Eo, *go = oracle.gb_grad(*(a[r].astype(np.float32).astype(np.float64) for a in (x, q, rho)),
                                 s.screen.astype(np.float32).astype(np.float64))
        assert abs(E[r] - Eo) <= 1e-6 * abs(Eo), (r, E[r], Eo)
        for a, o in zip(g, go):
            assert np.sqrt(((a[r] - o) ** 2).mean()) <= 1e-5 * np.sqrt((o ** 2).mean())
