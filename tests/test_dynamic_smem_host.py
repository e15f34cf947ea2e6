"""Host threads that launch the same kernel for products of different widths: the kernel's limit of
dynamic shared memory, state of the device and not of the launch, is only ever raised."""
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1504_05022_gb300", "csrc")


def test_every_kernel_raises_its_limit_in_one_place():
    users = [os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*"))
             if "MaxDynamicSharedMemorySize" in open(f).read()]
    assert users == ["dynamic_smem.h"]


def test_limit_on_a_fake_runtime(tmp_path):
    gxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "dynamic_smem")
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-pthread", "-I", cuda, "-I", CSRC,
                        os.path.join(ROOT, "tests", "dynamic_smem_host.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr
