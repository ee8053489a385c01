"""The representatives of a lattice's Fourier indices (csrc/pf_index.h), on the CPU: for all
shapes up to 7 x 7 x 7 and some long ones, in order, each j that is not above -j mod L."""
import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_00339_gb300", "csrc")


def test_representatives(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "pf_index_driver")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, os.path.join(ROOT, "tests", "pf_index_driver.cpp"), "-o", exe], check=True)
    shapes = list(itertools.product(range(1, 8), repeat=3)) + [(1, 1, 64), (64, 1, 1), (1, 64, 1), (33, 1, 2), (2, 17, 16)]
    out = subprocess.run([exe], input="\n".join("%d %d %d" % s for s in shapes), capture_output=True, text=True, check=True).stdout
    for (a, b, c), line in zip(shapes, out.split("\n")):
        got = [int(x) for x in line.split()]
        ref = [(i * b + j) * c + k for i in range(a) for j in range(b) for k in range(c)
               if (-i % a * b + -j % b) * c + -k % c >= (i * b + j) * c + k]
        assert got[0] == len(ref) and got[1:] == ref, (a, b, c)
