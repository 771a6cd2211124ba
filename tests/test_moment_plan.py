"""The choice of the moments' forms and of the cell side (csrc/moments_plan.cuh), checked on the host."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plans_of_random_calls(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "moment_plan")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include"), "-o",
                    exe, os.path.join(ROOT, "tests", "c", "moment_plan.cu")], check=True)
    r = subprocess.run([exe, "1", "200000"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 10000
