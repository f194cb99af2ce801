"""The bench's roofline holds what the timed kernel needs. CPU only."""
import pytest

import bench


def test_roofline_counts_what_the_timed_kernel_needs():
    """The nodes and leaves that another kernel counted do not enter the roofline of the timed one."""
    st = {"rays": 1000, "blended": 20_000, "nodes": 10**9, "leaves": 10**9}
    r = bench.roofline_of(st, 2.0, {"hbm_gbs": 5000.0})
    assert r["achieved"] == pytest.approx((208 * 20_000 + 16 * 1000) / 2e-3 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / 5000.0) and r["peak_source"] == "measured"
    assert r["bytes_per_ray"] == pytest.approx(208 * 20 + 16)
