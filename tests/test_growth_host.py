"""The constructors' linear stability decision (csrc/lbks_growth.h) equals lb_ks_max_growth's
rate compared with the limit, and the rate reported above it that rate, over random spacings, time steps, relaxation times and
readings of both schemes, at the library's limit and just above and below the rate."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_decision_equals_the_rate(tmp_path):
    exe = str(tmp_path / "growth_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "growth_check.cpp"),
                    os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_params.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
