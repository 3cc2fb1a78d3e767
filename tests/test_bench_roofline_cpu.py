"""What the bench line says of the COCG kernels, from made-up statistics: the HBM roofline is the
launched kernels' alone, the resident kernel has an entry of its own."""
import bench

PK = dict(hbm_gbs=6000.0, src="measured")


def stats(launched, resident):
    ks, kb, kl = [0.0] * 8, [0.0] * 8, [0] * 8
    if launched:
        ks[:5], kl[1], kl[3] = [0.1, 2.0, 0.3, 1.0, 0.1], 20, 20
        kb[1], kb[3] = 2.0 * 3000e9, 1.0 * 2500e9
        ks[6], kl[6] = 3.5, 20
    if resident:
        ks[7], kl[7], kb[7] = 4.0, 10, 4.0 * 500e9
    return ks, kb, kl


def test_resident_kernel_is_no_part_of_the_launched_roofline():
    alone, none = bench.cocg_roofline(*stats(True, False), -102, 0, 20.0, 4, 1000, PK)
    both, res = bench.cocg_roofline(*stats(True, True), -102, -7, 20.0, 4, 1000, PK)
    assert none is None
    assert both == alone and both["kernel"] == "k_dirmatvec_band"
    assert abs(both["achieved"] - 3000.0) < 1e-9 and abs(both["cocg_share"] - 2.0 / 3.5) < 1e-12
    assert res["kernel"] == "k_cocg_resident" and res["bound"] != "hbm"
    assert res["cocg_share"] == 4.0 / 20.0 and abs(res["global_gbs"] - 500.0) < 1e-9


def test_a_run_of_the_resident_kernel_alone():
    line, res = bench.cocg_roofline(*stats(False, True), -7, -7, 5.0, 8, 1000, PK)
    assert line["kernel"] == "k_cocg_resident" and line["bound"] == "FP64 pipe"
    assert line["cocg_share"] == res["cocg_share"] == 0.8 and line["traffic"] is None
    assert "launches over" not in bench.tilings(-7, -7) and "one kernel" in bench.tilings(-7, -7)
    assert "(last active systems)" in bench.tilings(-102, -7)
    assert "(<= 32 systems)" in bench.tilings(-102, 0)
