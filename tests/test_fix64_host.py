"""The fixed-point collision of FP64 storage (csrc/lbks_fix64.cuh), on the host: the same
integer arithmetic the kernels run, compiled with g++.

On random sites of both schemes, over spacings, time steps, relaxation times, amplitudes
and departures from equilibrium, each result is within the bound that follows from the
grid (stated in the program) of the value in long double, and mass is kept within the
conversions' half ulps.  Lattices advanced 1500 steps end, over the settings, no further
from the long double run than with the FP64 arithmetic it stands in for.  Values it does not cover are refused."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_collision(tmp_path):
    exe = str(tmp_path / "fix64_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "fix64_check.cpp"),
                    os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_params.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
