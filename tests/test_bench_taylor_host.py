"""CPU checks of the Taylor workload's roofline fields: no share of the HBM rate for what the L2 keeps."""
import bench


def _line(by_masks, l2, n=16, K=3, traffic=5e8):
    info = {"r": 100, "K": K, "D": 455, "S": 26_000_000, "by_masks": by_masks}
    return bench.taylor_roofline(n, info, 12e-6, 6800.7, "measured", l2, traffic)


def test_masks_in_l2_have_no_hbm_share():
    r = _line(True, 126 << 20)
    assert r["bound"] == "l2" and r["frac"] is None and r["peak"] is None and r["traffic"] is None
    assert r["algorithmic_bytes_per_launch"] == 8 * 65536 * (1 + 16 + 120) + 16 * 65536
    assert r["hbm_bytes_per_evolution"] == 8 * 26_000_000 + 16 * 65536
    assert abs(r["achieved"] - r["algorithmic_bytes_per_launch"] / 12e-6 / 1e9) < 1e-6


def test_diagonals_beyond_l2_are_an_hbm_share():
    r = _line(False, 126 << 20)
    assert r["bound"] == "hbm" and r["kernel"] == "spmv_kernel"
    assert abs(r["frac"] - r["achieved"] / 6800.7) < 1e-12 and r["traffic"] == 5e8
    # masks that do not fit are read from HBM too; the profile of the other kernel says nothing of them
    r = _line(True, 64 << 20)
    assert r["bound"] == "hbm" and r["traffic"] is None
