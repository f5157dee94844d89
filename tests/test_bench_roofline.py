"""The bench line's roofline: no share of a bound above 1 for the measured launch of the large
workload, and the bound of the kernel that ran."""
import bench


def test_share_of_the_bound_of_the_kernel_that_ran():
    n, P, D = 10_000_000, 1024, 4
    r = bench._eval_roofline((51, 3), D, P, n, 3.63e-3, 152, 2070.0, "measured")
    assert r["bound"] == "shared" and "eval_slice_kernel<4,3>" in r["kernel"]
    assert r["wavefronts_per_launch"] == 9766 * 1024 * 15 * 5  # tiles, trees, nodes, rows
    assert 0.6 < r["frac"] < 1.0
    r = bench._eval_roofline((0, 0), D, P, n, 10.22e-3, 152, 2070.0, "measured")
    assert r["bound"] == "alu" and "eval_kernel<2,4>" in r["kernel"]
    assert 0.4 < r["frac"] < 0.5
    assert abs(r["evals_per_s"] - P * n / 10.22e-3) < 1.0
