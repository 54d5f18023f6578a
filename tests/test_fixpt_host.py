"""The two-word fixed-point sums of the complex128 gradients, compiled for the
host from the kernels' header (no GPU)."""
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))


def test_two_word_sums_of_equal_terms():
    with tempfile.TemporaryDirectory() as td:
        exe = os.path.join(td, "fixcheck")
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math",
                               os.path.join(HERE, "fixpt_host_check.cpp"), "-o", exe])
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
