"""The handle's device memory on the host alone: csrc/wf_mem.cu compiled as C++
and run against the fake two-device CUDA runtime of mem_driver.cpp, which says
when a buffer is handed on while work queued on its device may still use it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_00503_gb300", "csrc")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("mem") / "mem_driver")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", include, "-I", CSRC, os.path.join(ROOT, "tests", "mem_driver.cpp"),
                    "-x", "c++", os.path.join(CSRC, "wf_mem.cu"), "-o", exe, "-lpthread"], check=True)
    return exe


@pytest.mark.parametrize("what", ["other_device", "failed_wait", "current_device", "trims", "refused"])
def test_memory_of_a_handle(driver, what):
    r = subprocess.run([driver, what], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
