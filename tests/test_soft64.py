"""Fixed-point sums of float64 products (the integer-pipe part of the float64
stencil) stay within their derived error bound and decline every operand they
cannot hold.  Host code only; no GPU needed."""
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_sums_of_products():
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "soft_check")
        subprocess.check_call(["nvcc", "-std=c++17", "-O2", "-o", exe, os.path.join(HERE, "soft_check.cu")])
        out = subprocess.run([exe], capture_output=True, text=True, timeout=600)
        assert out.returncode == 0, out.stdout + out.stderr
        assert out.stdout.startswith("OK"), out.stdout
