"""bench.py's roofline of the FD product: each pipe's work against that pipe's rate."""
import bench


def test_only_fp64_work_over_the_fp64_peak():
    """Traces, sum factorisation and lifts grow with the order and run on the FP32 pipe: at the same
    time a product of any order shows the same FP64 rate, and a second of work at the peak shows 1."""
    r = [bench.fd_product_roofline(k, 1000, 2000, 0.01, 1.25, 152, 2070.0) for k in (1, 2, 3, 4)]
    assert len({x["flop"] for x in r}) == 1 and len({x["frac"] for x in r}) == 1
    assert all(a["two_float"]["fma"] < b["two_float"]["fma"] for a, b in zip(r, r[1:]))
    flops = r[0]["flop"]
    assert flops == 1000 * 58 + 2000 * 34
    full = bench.fd_product_roofline(3, 1000, 2000, flops / 1.25e12 * 1e3, 1.25, 152, 2070.0)
    assert abs(full["frac"] - 1.0) < 1e-12
