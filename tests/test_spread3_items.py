"""The work items of the volume spreading (csrc/spread3_items.cuh), on the CPU."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_items_cover_the_lists(tmp_path):
    from paper_2411_01955_gb300 import build
    exe = str(tmp_path / "check")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, "-I", build.CSRC, os.path.join(HERE, "spread3_items_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
