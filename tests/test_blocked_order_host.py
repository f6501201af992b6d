"""The one-site-per-thread kernel's tiling (csrc/lbks_plan.h, choose_blocked) of batches of more
than 128 lattices of which few are longer than a block: whatever the caller's order, the
chosen tiling holds every lattice (the longest one decides whether halos are needed) and is
the same."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_blocked_tiling_in_any_order(tmp_path):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "vector_types.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path / "blocked_order_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror",
                    "-I" + os.path.join(ROOT, "paper_1711_03540_gb300", "csrc"), "-I" + CUDA_INC,
                    os.path.join(ROOT, "tests", "blocked_order_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
