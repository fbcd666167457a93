"""Read-outs fault in the pages of their destination only where they are not there
yet (csrc/prefault.h), on the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1312_3426_gb300", "csrc")


def test_only_fresh_ranges_are_faulted_in(tmp_path):
    exe = str(tmp_path / "prefault")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-pthread", "-I", CSRC,
                    os.path.join(ROOT, "tests", "prefault.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    got = dict(zip(out[::2], map(int, out[1::2])))
    assert got == {"fresh": 0, "ends": 0, "contents": 1, "touched": 1, "middle": 0, "small": 1}
