"""The fixed-point fp64 collision (csrc/fx64.cuh) on the CPU: host build of the
same arithmetic against a long-double evaluation of the scheme, on random nodes
of every compiled velocity set -- channel-like states, states of any amplitude
(the range checks must send what does not fit to the general form) and states
with single large populations."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_fixed_point_collision_within_bound(tmp_path):
    exe = str(tmp_path / "fx64_driver")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-Wno-unknown-pragmas",
                    "-I", os.path.join(ROOT, "paper_1510_08886_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx64", "fx64_driver.cpp")], check=True)
    r = subprocess.run([exe, "2000"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    # both forms were reached in the regimes that straddle the range
    rows = [line.split() for line in r.stdout.splitlines()]
    for row in rows:
        taken, left = int(row[7]), int(row[9])
        assert taken > 0 and (row[5] == "0:" or left > 0), row
