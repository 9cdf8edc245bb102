"""Memory that handles hold for speed (csrc/memory.cu) is never released under work in flight: the registry
compiled as host code against a fake CUDA runtime (tests/native/held_memory.cpp), without a GPU."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cuda_include():
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def test_unpinned_memory_has_no_work_in_flight(tmp_path):
    csrc = os.path.join(ROOT, "paper_2012_06714_gb300", "csrc")
    exe = str(tmp_path / "held_memory")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", csrc, "-I", cuda_include(), "-o", exe, "-x", "c++",
                    os.path.join(csrc, "memory.cu"), os.path.join(ROOT, "tests", "native", "held_memory.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
