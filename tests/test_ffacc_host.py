"""The error of the double-float sums of a full Hamiltonian pass, compiled for
the host from the kernels' header (no GPU)."""
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))


def test_sums_of_a_full_pass():
    with tempfile.TemporaryDirectory() as td:
        exe = os.path.join(td, "ffacc")
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math",
                               os.path.join(HERE, "ffacc_host_check.cpp"), "-o", exe])
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
