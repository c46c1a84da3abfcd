"""The short FP64 functions against CUDA's (tests/device/fp64_functions.cu), over their
domains and at the edges of their tables' intervals."""
import os
import subprocess

import pytest

from paper_1809_07726_gb300 import build

pytestmark = pytest.mark.gpu

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device", "fp64_functions.cu")

# Derived from their steps, u = 2^-53 being half an ulp, CUDA's own function at most
# an ulp or two off (2u to 4u):
#   rcp64      y (1 + e + e^2): e^3 < 2^-57, one rounding                -> 2u + u
#   rsqrt64    e to 2u, halved; 5 e^3 / 16 < 2^-57; one rounding; CUDA 2u -> 5u
#   log64      of max(|log x|, 2^-7): the sum's rounding, r's and r^2 p's of
#              2^-7, the table's entry; CUDA 2u                            -> 6u
#   exp64      the table's entry, b r, the sum, r to 2^-58; CUDA 2u       -> 6u
#   tanh64     absolute: 2 e / (1 + e) <= 1 to e's 5u / 2, rcp64's 3u and the
#              sum's u; the result's u; CUDA 4u                            -> 12u
#   sincos64   absolute: t to 2u, the series' remainder 2u, its sum's u; CUDA 4u -> 9u
U = 2.0 ** -53
BOUNDS = {"rcp64": (1, 3 * U), "rsqrt64": (1, 5 * U), "log64": (1, 6 * U), "exp64": (1, 6 * U), "exp64_tab": (1, 6 * U),
          "tanh64": (0, 12 * U), "sin64": (0, 9 * U), "cos64": (0, 9 * U), "fix32": (0, 0.0)}


def test_errors_stay_within_their_bounds(tmp_path):
    exe = str(tmp_path / "fp64_functions")
    r = subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-cudart", "static", "-I", build.CSRC, SRC, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    got = {f[0]: (float(f[1]), float(f[2])) for f in (line.split() for line in out.stdout.splitlines())}
    assert set(got) == set(BOUNDS)
    for name, (which, bound) in BOUNDS.items():
        assert got[name][which] <= bound, (name, got[name], bound)
