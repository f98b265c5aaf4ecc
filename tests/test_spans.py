"""The overlap check of the batched solve, compiled for the host."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_spans_cross(tmp_path):
    exe = str(tmp_path / "spans")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror",
                    os.path.join(HERE, "cpp", "spans_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
