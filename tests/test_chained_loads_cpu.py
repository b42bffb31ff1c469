"""Source check of the chained steps' loads (no GPU): a kernel launched with
programmatic serialisation starts while its predecessor writes the lattice, so
no function of the step kernels may take a lattice pointer (src, dst) as
__restrict__, which licenses loads through the read-only path."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_08886_gb300", "csrc")


def test_lattice_pointers_are_not_restrict():
    for name in ("lbm_kernels.cuh", "k_cluster.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        assert not re.findall(r"__restrict__\s+(?:src|dst|fin|fout)\b", text), name
