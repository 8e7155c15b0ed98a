"""The benchmark's rooflines count FP64 work against the FP64 rate only where it is done in FP64."""
import bench


def test_eos_counts_the_fp64_part_of_the_search():
    # 3 evaluations and 2.5 solves a particle and stage, one of the evaluations at the solution
    got = bench.eos_flops((3000.0, 2500.0, 10.0), 1000.0)
    assert got == 2000 * 164.0 + 1000 * 416.0 + 10 * 26.0
    assert bench.eos_flops((0.0, 0.0, 50.0), 0.0) == 50 * 26.0


def test_integer_passes_state_no_fraction_of_a_floating_point_rate():
    r = bench.alu_roof("density", 1e9, 1.0, 2, None, None, "k")
    assert r["frac"] is None and r["peak"] is None and r["achieved"] == 1e3
    assert bench.alu_roof("eos", 1e9, 1.0, 2, 2e3, "p", "k")["frac"] == 0.5
