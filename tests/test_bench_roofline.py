"""The roofline that the benchmark reports of the tensor-core kernel."""
import bench


def test_split_roofline_is_of_the_tensor_pipe():
    """F_3 [80,40]: one MAC a symbol for two codewords, 40 flops a codeword.
    (Counted in POPCs the kernel read 1.19 of a unit it does not use.)"""
    r = bench.split_roofline(3, 80, 40, 268257056, 0.0899, 1909.5, "measured")
    assert r["bound"] == "tensor" and r["flops_per_codeword"] == 40
    assert abs(r["achieved"] - 268257056 * 40 / 0.0899e-3 / 1e12) < 1e-6
    assert 0 < r["frac"] < 1 and r["peak"] == 2 * 1909.5
    assert bench.split_roofline(7, 50, 25, 10 ** 9, 1.0, 1909.5, "measured")["flops_per_codeword"] == 75
    assert bench.split_roofline(5, 51, 24, 10 ** 9, 1.0, 1909.5, "measured")["flops_per_codeword"] == 81


def test_bf16_peak_has_a_figure():
    value, source = bench.bf16_peak()
    assert value > 1000 and source in ("measured", "fallback")
