"""The plans' device memory (csrc/device_memory.h) on a fake CUDA runtime, compiled for the host:
which freed memory the driver gets back at once, which small blocks are kept and for whom, the
bounds and the order of eviction, a full device, trimming, another device being current, and that a
plan's limit bounds the memory it really holds."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_on_a_fake_runtime(tmp_path):
    gxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "device_memory")
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-I", cuda, "-I",
                        os.path.join(ROOT, "paper_1504_05022_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "device_memory_host.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    assert r.stdout.count(": ok") == 12
