"""The exact per-thread sums of the integer legs, compiled for the host."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_sums_hold_over_their_ranges(tmp_path):
    exe = str(tmp_path / "sums")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror",
                    os.path.join(HERE, "cpp", "sums_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
