"""The fixed-point pull's arithmetic on the host, at the ends of its ranges (tests/fixed_point_pull.cpp):
every sum of pulls within 4 units of 2^-53 of the sum of the terms' magnitudes. A term carries the
positions' grid (2^-54), the residual's cut (2^-57), the series' (2^-58) and four products of 2^-60
or better, and the sum's components one rounding to double each, sqrt(3) 2^-54 together."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1404_2324_gb300", "csrc")


def test_pulls_at_the_ends_of_the_binades(tmp_path):
    exe = str(tmp_path / "pull")
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", f"-I{CSRC}", os.path.join(HERE, "fixed_point_pull.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True)
    pairs, worst = out.stdout.split()
    assert int(pairs) > 100000 and float(worst) <= 4.0, out.stderr
