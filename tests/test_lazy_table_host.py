"""The float64 solves' tables by lambda (mode factors, elimination pivots),
with a fake allocation on the host: built once per lambda, and a failed
allocation is not tried again by the solves that follow (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2104_05024_gb300", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("lazytable") / "lazy_table_host")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, os.path.join(HERE, "host", "lazy_table_host.cpp"),
                    "-o", exe], check=True)
    return exe


def requests(exe, have, keys):
    out = subprocess.run([exe, str(int(have)), *map(str, keys)], capture_output=True, text=True, check=True).stdout
    return [tuple(float(x) for x in line.split()) for line in out.splitlines()]


def test_one_allocation_and_one_build_per_change(harness):
    r = requests(harness, True, [60.0, 60.0, 0.0, 0.0, 60.0])
    assert [x[0] for x in r] == [1] * 5 and [x[1] for x in r] == [1] * 5
    assert [x[2] for x in r] == [1, 1, 2, 2, 3] and [x[3] for x in r] == [60.0, 60.0, 0.0, 0.0, 60.0]


def test_failed_allocation_is_remembered(harness):
    r = requests(harness, False, [60.0, 60.0, 0.0])
    assert [x[0] for x in r] == [0] * 3 and [x[1] for x in r] == [1] * 3 and r[-1][2] == 0
