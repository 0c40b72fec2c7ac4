"""The sine and cosine of the FP64 acceptance, whose small terms are evaluated
in FP32: their error against extended precision, on the CPU, by the library's
own source (tests/host/sincos_split_check.cu, with the bounds' derivation)."""
import os
import subprocess
import tempfile

from tests.test_host_plans import ROOT, _nvcc


def test_error_of_the_split_sine_and_cosine():
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "sincos_split_check")
        src = os.path.join(ROOT, "tests", "host", "sincos_split_check.cu")
        r = subprocess.run([_nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                            "--expt-relaxed-constexpr", "-O1", "-Xcompiler", "-ffp-contract=off", src, "-o", exe],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
