"""The fixed point's stop test inside a solver launch, on host threads (no GPU): whenever another
block stores the status word, all threads of a block decide alike and all or none join its sums."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_15676_gb300", "csrc")


def test_a_block_decides_as_one(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("needs g++")
    exe = tmp_path / "fp_stop"
    subprocess.run([gxx, "-std=c++20", "-O1", "-pthread", "-I", CSRC, os.path.join(HERE, "fp_stop_host.cpp"), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split("\n")
    rows = [line.split() for line in out if line]
    assert len(rows) == 2 * 67
    for stop, n, yes, no, summed in rows:
        assert (int(yes), int(no)) == (0, 64), (stop, n, yes, no)   # the loop stops, whoever noticed
        assert int(summed) in (0, 64), (stop, n, summed)
