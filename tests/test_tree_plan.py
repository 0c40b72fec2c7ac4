"""The compile-time structure of the humanoid's tree kernel (order of its sums,
shared-memory slots, constants of the prismatic base), checked on the CPU by
the library's own host code (tests/host/tree_plan_check.cu)."""
import os
import subprocess
import tempfile

from tests.test_host_plans import ROOT, _nvcc


def test_tree_kernel_structure_matches_the_plan():
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "tree_plan_check")
        src = os.path.join(ROOT, "tests", "host", "tree_plan_check.cu")
        r = subprocess.run([_nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                            "--expt-relaxed-constexpr", "-O1", "-I",
                            os.path.join(ROOT, "include"), src, "-o", exe], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout[-3000:]
        assert "humanoid36: 0 problems" in r.stdout and "humanoid36_hull: 0 problems" in r.stdout
