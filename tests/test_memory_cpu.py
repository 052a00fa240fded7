"""Result words of contexts over device resets, with the CUDA runtime's calls
faked on the CPU (no GPU): hsg_memory.cu itself, compiled for the host."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1006_2566_gb300", "csrc")


def test_result_words_over_resets():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    with tempfile.TemporaryDirectory() as tmp:
        exe = os.path.join(tmp, "memory_check")
        subprocess.run([nvcc, "-std=c++17", "-O2", "-cudart", "none", "-x", "c++", "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, "-o", exe, os.path.join(ROOT, "tests", "native", "memory_check.cpp"),
                        os.path.join(CSRC, "hsg_memory.cu")], check=True)
        r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout
