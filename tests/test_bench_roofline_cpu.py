"""The bench's roofline on the host: fraction of the HBM rate in every precision."""
import bench


def test_fraction_is_of_the_memory_rate():
    r = bench.step_roofline(3300.0, 6600.0, "measured", None)
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["frac"] == 0.5
