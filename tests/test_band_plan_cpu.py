"""The banded solves' shared memory (csrc/band_plan.h), on the CPU: over every block size
and reach that the preconditioner's rule admits, alone and together in one launch, each
piece of coefficients fits its stage, starts and ends on 16 bytes, the pieces cover all
rows, and two stages and the rows kept beside them fit a CTA's 227 KB."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_00339_gb300", "csrc")
ROOM = (232448 - 1024) // 8


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("band") / "band_plan_driver")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, os.path.join(ROOT, "tests", "band_plan_driver.cpp"), "-o", exe], check=True)
    return exe


def _admitted(L, D, m0):
    return 2.0 * L * D * D * m0 ** 3 <= 8e9


def _launches(driver, launches):
    text = "".join(f"{len(ts)}\n" + "".join(f"{m} {D} {L}\n" for m, D, L in ts) + f"{ROOM}\n" for ts in launches)
    out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for ts, line in zip(launches, out):
        v = [int(x) for x in line.split()]
        yield ts, v[0], v[1], [v[2 + 4 * i:6 + 4 * i] for i in range(len(ts))]


def _check(driver, launches):
    n = 0
    for ts, stage, rows, tasks in _launches(driver, launches):
        assert stage % 2 == 0 and 2 * stage + rows <= ROOM, ts
        for (m0, D, L), (rule, most, aligned, covered) in zip(ts, tasks):
            assert rule == _admitted(L, D, m0)
            assert most <= stage and aligned and covered == m0, (ts, m0, D, L, stage, most, covered)
            n += 1
    assert n == sum(len(ts) for ts in launches)


def _reaches(m0):
    """Every reach the rule admits: from one end at the shortest chain, from both where that is admitted."""
    for D in range(0, 1700):
        if not _admitted(D + 1, D, m0):
            return
        yield m0, D, D + 1
        if _admitted(2 * D + 2, D, m0):
            yield m0, D, 2 * D + 2


def test_every_admitted_task_alone(driver):
    _check(driver, [[t] for m0 in range(1, 33) for t in _reaches(m0)])


def test_the_longest_reaches_of_all_blocks_together(driver):
    last = [list(_reaches(m0))[-2:] for m0 in range(1, 33)]
    _check(driver, [[t for ts in last for t in ts]] + [a + b for a in last for b in last])
