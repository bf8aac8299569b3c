"""Which kernel the benchmark's roofline is about."""
import bench


def test_dominant_kernel_is_one_that_the_solve_launches():
    kt = {"primal_step": {"ms": 0.008}, "dual_step": {"ms": 0.011}, "persistent_attempt": {"ms": 0.0125}}
    assert bench.dominant_kernel(kt) == "persistent_attempt"
    kt["persistent_attempt"]["ms"] = 0.0  # the separate launches
    assert bench.dominant_kernel(kt) == "dual_step"
    kt["primal_step"]["ms"] = 0.02
    assert bench.dominant_kernel(kt) == "primal_step"
