"""The fixed-point collision's input conversion (csrc/lbks_fix64.cuh, to_limbs), on the host: a
population 0 to 70 binades below its site's grid is cut to the grid with its last bit set
when any bit is lost, powers of two and values with a short mantissa included, and zero
stays zero, so that the conversion has no bias (a bias would drift the conserved mass)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_lost_bits_are_jammed_at_every_gap(tmp_path):
    exe = str(tmp_path / "fix64_jam_check")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "fix64_jam_check.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
