"""The plan of the one-site-per-thread kernel (csrc/lbks_plan.h), on the host: every site is
stored exactly once, every stretch of a longer lattice has c_max k halo sites on each cut
side, the pieces of a block do not overlap and fit it, and the tilings the cost model
chooses can hold their lattices."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_blocked_plans(tmp_path):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "vector_types.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path / "blocked_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "paper_1711_03540_gb300", "csrc"), "-I" + CUDA_INC,
                    os.path.join(ROOT, "tests", "blocked_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
