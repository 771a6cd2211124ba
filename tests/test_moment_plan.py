"""Host checks of the moments' plan and tiling: the choice of the forms and of the cell side
(csrc/moments_plan.cuh), the staging of candidates under the tiling overrides (csrc/moments.cuh)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plans_of_random_calls(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "moment_plan")
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I" + os.path.join(ROOT, "include"), "-o",
                    exe, os.path.join(ROOT, "tests", "c", "moment_plan.cu")], check=True)
    r = subprocess.run([exe, "1", "200000"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 10000


@pytest.mark.parametrize("scr", [32, 256, 512])
def test_staged_candidates_can_be_indexed(tmp_path, scr):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-DMP3_MOM_SCR_F32=%d" % scr, "-DMP3_MOM_SCR_F32_WIDE=%d" % scr, "-I" + os.path.join(ROOT, "include"),
                    "-c", "-o", str(tmp_path / "staged_index.o"), os.path.join(ROOT, "tests", "c", "staged_index.cu")],
                   check=True)
