"""The clock of the bounded waits in a launch of many steps (csrc/bounded_wait.h), on
the host: a wait gives up after the time it has waited, whatever else held the GPU in
between."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1312_3426_gb300", "csrc")


def test_a_wait_counts_its_own_time(tmp_path):
    exe = str(tmp_path / "bounded_wait")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", CSRC,
                    os.path.join(ROOT, "tests", "bounded_wait.cpp"), "-o", exe], check=True)
    slow, fast, hour, short, half = map(float, subprocess.run([exe], capture_output=True, text=True,
                                                              check=True).stdout.split())
    # at the first reading past the bound (the numbers have three decimals); a gap counts 10 ms
    digit = 1e-3
    assert 10000.0 < slow <= 10000.0 + 0.7 + digit and 10000.0 < fast <= 10000.0 + 0.04 + digit
    assert 3600e3 + 10000.0 - 10.0 < hour <= 3600e3 + 10000.0 - 10.0 + 2 * 0.7 + digit
    assert short == half == -1.0
