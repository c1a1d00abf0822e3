"""The operations and bytes behind the bench's fractions are those of the kernels that run, restated here by hand.

p = 2, per element: 4 for a coefficient row along x; 3 columns of 4 along y; 3 columns of 5 to values and
derivatives; 3 rows of 8 to T, T_x, T_y; 9 points of 9; 3 rows of 11 to the x sums; 3 columns of 8 to the y sums, of 7
to rows; 8 for a finished row.
"""
import bench


def test_quadrature_operations():
    assert bench.quadrature_ops(2, 0) == 4 + 3 * 4 + 3 * 5 + 3 * 8 + 9 * 9 + 3 * 11 + 3 * 8 + 3 * 7 + 8 == 222
    assert bench.quadrature_ops(1, 0) == 2 + 2 * 2 + 2 * 2 + 2 * 4 + 4 * 9 + 2 * 6 + 2 * 4 + 2 * 4 + 5 == 87
    assert bench.quadrature_ops(3, 0) == 9 + 4 * 9 + 4 * 15 + 4 * 23 + 16 * 9 + 4 * 31 + 4 * 21 + 4 * 14 + 15 == 620
    # two multiply-adds a point and rank; ranks run as 0, 2 or 4
    assert bench.quadrature_ops(2, 1) == bench.quadrature_ops(2, 2) == 222 + 9 * 4
    assert bench.quadrature_ops(2, 3) == bench.quadrature_ops(2, 4) == 222 + 9 * 8


def test_kernels_of_a_step():
    pr = bench.kernel_costs(2, 0, "pr")
    assert set(pr) == {"rhs_quadrature_1", "xsolve_1", "ysolve_1", "step_persistent"}
    assert pr["rhs_quadrature_1"] == {"bytes": 12, "flops": 444}
    assert pr["xsolve_1"] == {"bytes": 16, "flops": 36} and pr["ysolve_1"] == {"bytes": 24, "flops": 40}
    assert pr["step_persistent"] == {"bytes": 40, "flops": 76}
    assert bench.step_costs(2, 0, "pr") == {"bytes": 52, "flops": 520}
    assert bench.kernel_costs(2, 0, "pr", split=True)["ysolve_1"] == {"bytes": 12, "flops": 20}
    assert bench.step_costs(2, 0, "explicit") == {"bytes": 52, "flops": 520}
    assert bench.step_costs(2, 0, "strang")["bytes"] == 12 + 16 + 12 + 8 + 8 + 24
    # the names are those the library times
    with open(bench.ROOT + "/paper_2604_19370_gb300/csrc/wf_api.cu") as f:
        src = f.read()
    for scheme in ("pr", "strang", "explicit"):
        assert all(f'"{k}"' in src for k in bench.kernel_costs(2, 0, scheme))


def test_fractions_of_the_pipe_stay_below_one():
    # the default ensemble's quadrature, 0.23 ms on one GB300 (80 TFLOP/s): with the method's 690 flops its fraction read 0.64
    dofs, c = 256 * 258 * 258, bench.kernel_costs(2, 0, "pr")
    r = bench.roofline("rhs_quadrature_1", 0.23, dofs, c, 4, 6767.0, "measured", 80.0, "probe")
    assert r["bound"] == "alu" and 0.35 < r["frac"] < 0.5
