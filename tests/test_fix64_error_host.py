"""The error of the FP64 collision (csrc/lbks_fix64.cuh) over long runs, on the host, against
long double: lattices advanced 200000 steps with the library's collision end, setting by
setting (three lattices pooled), no further from the exact run than with FP64 arithmetic.
The settings have small and large time steps on fine and coarse spacings, with and without a
mean, so that the moving planes lie 2 to 30 binades below g_0.  The mass of a lattice with a
mean is kept to its last place, and one collision's error in the smallest planes is no larger
than FP64 arithmetic's."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_error_over_long_runs(tmp_path):
    exe = str(tmp_path / "fix64_error_check")
    subprocess.run(["g++", "-O3", "-std=gnu++17", "-ffp-contract=off", "-pthread", "-I", os.path.join(ROOT, "include"),
                    "-o", exe, os.path.join(ROOT, "tests", "fix64_error_check.cpp"),
                    os.path.join(ROOT, "paper_1711_03540_gb300", "csrc", "lbks_params.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
