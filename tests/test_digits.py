"""The integer arithmetic and the launch plans of the FP64 contractions (csrc/digits.cuh, csrc/plan64.cuh) as
host code (tests/native/digits.cpp), without a GPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_digit_products_and_plans(tmp_path):
    exe = str(tmp_path / "digits")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2012_06714_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "digits.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
