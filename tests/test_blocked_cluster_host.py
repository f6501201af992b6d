"""The cluster plan of the one-site-per-thread kernel (csrc/lbks_plan.h), on the host: one
step's values are moved as the kernel's threads move them, so that every site is held once,
every thread reads the value of the site its plane comes from, no column is written twice,
nothing lies outside a block's exchange area, and the chosen tilings hold their lattices."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_cluster_plans(tmp_path):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "vector_types.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path / "cluster_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "paper_1711_03540_gb300", "csrc"), "-I" + CUDA_INC,
                    os.path.join(ROOT, "tests", "cluster_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
