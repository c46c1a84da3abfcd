"""The small-walker kernel's SHAKE, built for the host with its four lanes as
threads (tests/host/shake_small.cpp)."""
import os
import subprocess

import pytest

from paper_1809_07726_gb300 import build

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("shake") / "shake_small")
    r = subprocess.run(["g++", "-std=c++20", "-O1", "-ffp-contract=off", "-pthread", "-Wno-unknown-pragmas",
                        "-I", build.CSRC, os.path.join(HOST, "shake_small.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lambda *a: subprocess.run([exe, *map(str, a)], capture_output=True, text=True, check=True).stdout.split()


def test_a_clusters_lanes_hold_the_same_sum(program):
    """The lanes decide by it, each for its own component: one low bit of
    difference freezes a component of a constraint that the others still move."""
    assert program("sums", 3000) == ["0"]


@pytest.mark.parametrize("tol", [1e-8, 1e-10, 1e-12])
def test_constraints_settle_along_the_old_bonds(program, tol):
    """|d^2 - d0^2| <= 2 tol d0^2, and the arithmetic's own 1e-13 (pairs of floats:
    a few 2^-47); hydrogens move along their old bond vectors to the pairs' 2^-47 of
    displacements below 1 A."""
    unsettled, worst, off = program("shake", 600, tol)
    assert unsettled == "0" and float(worst) <= 2 * tol + 1e-13 and float(off) <= 1e-13
