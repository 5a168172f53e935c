"""The roofline of the dominant kernel class: a rate that the kernel can be bound by.  The FP64 per-shift
update does its multiply-adds on the tensor cores, so their count is not measured against the
FP64 rate (figures of the random matrix with 256 shifts: 17 launches of 81.5 ms each)."""
import bench


def test_shift_update_is_measured_against_hbm():
    stats = [dict(name="shift_update", launches=17, ms=1386.4, alg_bytes=17 * 72.2e9, alg_flops=17 * 9.0e11),
             dict(name="seed_mvm", launches=936, ms=733.3, alg_bytes=1e12, alg_flops=1e12)]
    for prec in (0, 1):
        top, roof = bench.dominant_roofline(stats, prec, {"hbm_gbs": 6778.7})
        assert top["name"] == "shift_update" and roof["bound"] == "hbm" and 0.0 < roof["frac"] < 1.0
