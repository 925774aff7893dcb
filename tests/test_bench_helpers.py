"""The benchmark's guard of its captured DRAM figure covers the files that hold
the pair pass, and its timed steps run as a user's (profiling off)."""
import ast
import os

import bench


def test_guard_hashes_the_pair_pass():
    csrc = os.path.join(bench.ROOT, "paper_2606_10019_gb300", "csrc")
    holds = {f for f in os.listdir(csrc) for t in [open(os.path.join(csrc, f)).read()]
             if "bool tile_pass(" in t or "void __launch_bounds__(PAIR_WARPS * 32, MODE" in t}
    assert holds and holds <= set(bench.PAIR_KERNEL_FILES)
    assert len(bench.pair_kernel_sha()) == 16


def test_timed_steps_run_without_profiling():
    tree = ast.parse(open(bench.__file__).read())
    fn = {f.name: f for f in tree.body if isinstance(f, ast.FunctionDef)}
    for name in ("run_gcvo", "lidar_tracking_block", "exact_hessian_block"):
        calls = [c.func.attr for c in ast.walk(fn[name]) if isinstance(c, ast.Call) and isinstance(c.func, ast.Attribute)]
        assert "gcvo_profile_enable" not in calls, name
