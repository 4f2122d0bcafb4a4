"""How bench.py rates an iteration (no GPU): the streaming kernels by HBM bytes;
a solve held on the chip, which moves none of its own, by its arithmetic against
the FP32 FMA rate."""
import bench


class _Lib:
    PRECISIONS = {"fp64": 0, "fp32_refined": 1}

    @staticmethod
    def heat_probe_fma_rate(fp64, reps):
        return 1.2 if fp64 else 70.0


def test_an_iteration_on_the_chip_is_no_memory_rate():
    chip = {"ms_apply": 0.0133, "ms_update": 0.0, "bytes_apply": 0.0, "bytes_update": 0.0}
    assert bench.iteration_kernel(_Lib, chip, "fp32_refined", "stream") == "k_cg_res (one iteration)"
    r = bench.iteration_roofline(_Lib, chip, "k", 1030301, 6800.0, "measured")
    assert r["unit"] == "TFLOP/s" and r["peak"] == 70.0 and r["bound"] != "hbm"
    assert abs(r["achieved"] - bench.ITERATION_FLOPS_PER_NODE * 1030301 / 0.0133e-3 / 1e12) < 1e-9
    assert bench.apply_rate(chip) is None and bench.fraction(None, 6800.0) is None


def test_streaming_launches_are_rated_by_their_bytes():
    prof = {"ms_apply": 0.06, "ms_update": 0.05, "bytes_apply": 2.2e8, "bytes_update": 2.3e8}
    assert bench.iteration_kernel(_Lib, prof, "fp32_refined", "stream") == "stream"
    r = bench.iteration_roofline(_Lib, prof, "stream", 8120601, 6800.0, "measured")
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and abs(r["achieved"] - 2.2e8 / 0.06e-3 / 1e9) < 1e-6
    assert r["frac"] == r["achieved"] / 6800.0 and r["update_kernel"]["achieved"] > 0.0
