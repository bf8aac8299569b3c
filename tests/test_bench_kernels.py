"""Which kernel the benchmark's roofline is about."""
import bench


def test_dominant_kernel_is_one_that_the_solve_launches():
    kt = {"primal_step": {"ms": 0.008}, "dual_step": {"ms": 0.011}, "persistent_attempt": {"ms": 0.0125}}
    assert bench.dominant_kernel(kt) == "persistent_attempt"
    kt["persistent_attempt"]["ms"] = 0.0  # the separate launches
    assert bench.dominant_kernel(kt) == "dual_step"
    kt["primal_step"]["ms"] = 0.02
    assert bench.dominant_kernel(kt) == "primal_step"


def test_the_timed_iterations_keep_their_name():
    """iters_per_solve is formed of the timed solves' iterations at the end of the run: no loop
    variable of a later section takes their name."""
    import ast
    import inspect
    import textwrap
    fn = ast.parse(textwrap.dedent(inspect.getsource(bench.run_gpu))).body[0]
    loops = {n.id for node in ast.walk(fn) if isinstance(node, ast.For)
             for n in ast.walk(node.target) if isinstance(n, ast.Name)}
    assert not loops & {"iters", "launches", "res", "ms"}, loops
