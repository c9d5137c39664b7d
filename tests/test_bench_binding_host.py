"""bench.py reports a kernel against the roof that bounds it: the FP64 contractions in block floating
point against the integer multiply-add pipe, everything else unchanged."""
from tests.test_bench_host import load_bench


def test_reported_fraction_is_of_the_binding_roof():
    b = load_bench()
    pk = {"hbm_gbs": 6794.5, "sm_max_mhz": 2070.0}
    ax = {"launches": 1, "ms": 0.41, "bytes": 1.133e9, "flops": 1.8623e9}
    r = b.binding(b.roofline("ax", 7, ax, pk, "measured"))
    peak = 152 * 12 * 2 * 2.07e9 / 1e12
    assert r["bound"] == "int" and abs(r["peak"] - peak) < 1e-3 and "int_pipe" not in r
    assert abs(r["frac"] - 1.8623e9 / 0.41e-3 / 1e12 / peak) < 1e-3 and r["frac"] < 1.0
    assert abs(r["hbm_frac"] - 1.133e9 / 0.41e-3 / 1e9 / 6794.5) < 1e-3
    assert abs(r["over_fp64_pipe_peak"] - 6 * r["frac"]) < 1e-2
    table = b.kernel_table({("ax", 7): ax}, 1, pk, "measured")
    assert table["ax p=7 f64"]["bound"] == "int" and table["ax p=7 f64"]["roof_frac"] == r["frac"]
    for kernel, variant, d in (("cheby_update", 0, {"launches": 10, "ms": 2.0, "bytes": 1e10, "flops": 1e8}),
                               ("fdm", 39, {"launches": 36, "ms": 5.4, "bytes": 36 * 2.4e8, "flops": 36 * 3.28e9})):
        r = b.roofline(kernel, variant, d, pk, "measured")
        assert b.binding(r) == r
