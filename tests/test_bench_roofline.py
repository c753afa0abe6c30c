"""The benchmark's roofline entry: the kernel that was launched, and a share of
the copy bandwidth only where the step moves the bytes it is figured on."""
import pytest

import bench
from paper_2203_01462_gb300 import inputs as I


@pytest.mark.parametrize("make,blocked,kernel", [
    (I.cfg_2d_316, True, "k_rt2d "), (I.cfg_2d_316, False, "k_step2d "),
    (I.cfg_2d_inplane_paper, True, "k_rt2dp "), (I.cfg_2d_inplane_paper, False, "k_hp "),
    (I.cfg_3d_256, False, "k_h3d ")])
def test_share_of_bandwidth(make, blocked, kernel):
    r = bench.roofline(make(), blocked, 5000.0, 6800.0, "measured", 1e6)
    assert r["kernel"].startswith(kernel)
    if blocked:
        assert r["bound"] != "hbm" and r["frac"] is None and r["achieved"] is None and r["unblocked_equivalent"] == 5000.0
    else:
        assert r["bound"] == "hbm" and r["frac"] == 5000.0 / 6800.0
