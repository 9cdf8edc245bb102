"""Splits of doubles into BF16 planes (csrc/split.cuh) lose nothing to a rounding to FP32 first: the device
function compiled as host code (tests/native/split.cpp), without a GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_planes_of_a_double(tmp_path):
    exe = str(tmp_path / "split")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2012_06714_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "split.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
