"""Failing CUDA calls under the library's host code, on the CPU: a stand-in for the CUDA
runtime makes one call fail and checks the copies (scenarios in host_fault_runs.py)."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    from paper_2411_01955_gb300 import build
    fake = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", fake], check=True)
    return fake, build.build()


def run(libs, scenario):
    r = subprocess.run([sys.executable, os.path.join(HERE, "host_fault_runs.py"), *libs, scenario],
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_net_scratch_holds_the_samples(libs):
    run(libs, "net_scratch_holds_the_samples")


@pytest.mark.parametrize("what", ["net", "learned"])
def test_scratch_after_failed_growth(libs, what):
    run(libs, what + "_scratch_after_failed_growth")


def test_next_call_after_oom(libs):
    run(libs, "next_call_after_oom")


def test_retile_fails_whole(libs):
    run(libs, "retile_fails_whole")
