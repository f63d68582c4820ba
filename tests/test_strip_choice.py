"""The strip width chosen for pairs of unequal length (csrc/ga_kx.cu), on the CPU
(tests/strip_choice_check.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_width_of_unequal_pairs(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = tmp_path / "strip_choice_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wall", "-I", os.path.join(cuda, "include"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "strip_choice_check.cpp")], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
