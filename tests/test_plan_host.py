"""The circuit planner's time, compiled for the host from the kernels' header
(no GPU)."""
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_planning_is_linear_in_the_gates():
    with tempfile.TemporaryDirectory() as td:
        exe = os.path.join(td, "plan")
        subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O2",
                               "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                               os.path.join(HERE, "plan_host_check.cu"), "-o", exe])
        out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
        assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
