"""Device memory as the engine takes it (csrc/devmem.h), over an allocator of the
test's: a failed allocation leaves no error behind, cached blocks are given back
before a request fails, and the cache stays within its limit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_pool_over_a_small_allocator(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "devmem_driver")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2304_08356_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "devmem_driver.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
