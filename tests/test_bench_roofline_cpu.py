"""The bench's roofline on the host: fraction of the HBM rate in every precision,
and counters taken from a profile only if its hash is that of the sources of the
profiled precision's kernel."""
import os

import bench


def test_fraction_is_of_the_memory_rate():
    r = bench.step_roofline(3300.0, 6600.0, "measured", None)
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["frac"] == 0.5


def test_source_hash_is_per_precision(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_1510_08886_gb300" / "csrc"
    os.makedirs(csrc)
    os.makedirs(tmp_path / "profiles")
    names = {"lbm_kernels.cuh", "lbm_internal.h"}.union(*bench.KERNEL_SOURCES.values())
    for fn in names:
        (csrc / fn).write_text(fn)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    for p in ("fp32", "fp64"):
        (tmp_path / "profiles" / f"stream_collide_{p}_D2V33_4096x512.md").write_text(
            f"kernel_source_sha256_16: {bench.kernel_source_hash(p)}\ndram_bytes_per_launch: 5e8\n")
    assert bench.ncu_traffic("fp32") == bench.ncu_traffic("fp64") == 5e8
    (csrc / "fx64.cuh").write_text("changed")
    assert bench.ncu_traffic("fp32") == 5e8 and bench.ncu_traffic("fp64") is None
    (csrc / "lbm_kernels.cuh").write_text("changed")
    assert bench.ncu_traffic("fp32") is None
    assert bench.ncu_traffic("fp16") is None          # no profile of it
