"""The fixed-point collision (csrc/lbks_fix64.cuh), on the host, at sites where the density
changes sign: populations that cancel to a sum of either sign, down to 2^-56 of their size.
Every result is the long double value to within 64 units of the last place at the
neighbours' density (an error of s^2, whose sign such a sum does not fix in two limbs, is
larger by nine orders of magnitude)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sums_that_cancel(tmp_path):
    exe = str(tmp_path / "fix64_cancel_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "fix64_cancel_check.cpp"),
                    os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_params.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
