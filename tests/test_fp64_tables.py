"""The tables of the short FP64 logarithm and exponential, recomputed: 1/c and -log of it
for the middles c of log64's intervals (1/256 wide from 0.6875 to 1, 1/128 from there to
1.375), and 2^(j/16)."""
import os
import re
from fractions import Fraction

import numpy as np

from paper_1809_07726_gb300 import build


def _numbers(name):
    text = open(os.path.join(build.CSRC, "cph_device.cuh")).read()
    body = re.search(name + r"\[\w+\] = \{(.*?)\};", text, re.S).group(1)
    return [float(v) for v in re.findall(r"-?\d+\.\d+(?:e-?\d+)?", body)]


def test_log_and_exp_tables():
    v = _numbers("kTab64Values")
    assert len(v) == 2 * 136
    logs, exps = np.array(v[:256]).reshape(128, 2), v[256:]
    edges = [Fraction(11, 16) + Fraction(j, 256) for j in range(80)] + [1 + Fraction(j, 128) for j in range(49)]
    for (inv, lg), a, b in zip(logs, edges, edges[1:]):
        assert inv == float(2 / (a + b))  # the nearest double
        want = -np.log(np.longdouble(inv))
        assert abs(np.longdouble(lg) - want) <= np.spacing(abs(lg))
    assert edges[-1] == Fraction(11, 8)
    want = [float(np.longdouble(2) ** (np.longdouble(j) / 16)) for j in range(16)]
    for got in (exps, _numbers("kExp2Tab")):
        assert len(got) == 16 and all(abs(g - w) <= np.spacing(w) for g, w in zip(got, want))
