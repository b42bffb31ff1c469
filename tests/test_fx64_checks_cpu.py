"""Properties of the fixed-point fp64 collision (csrc/fx64.cuh) on the CPU that the
comparison of random nodes with a long-double evaluation does not show: each
program of tests/fx64 named here says in its first lines what it checks."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
@pytest.mark.parametrize("program", ["fx64_force", "fx64_rest", "fx64_rates", "fx64_range", "fx64_moments"])
def test_fixed_point_collision(program, tmp_path):
    exe = str(tmp_path / program)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wno-unknown-pragmas",
                    "-I", os.path.join(ROOT, "paper_1510_08886_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx64", program + ".cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
