"""The library's allocations (ms_blocks.cu) compiled for the host against fakes
of the CUDA calls: what freed contexts leave is bounded, every allocation gives it
back before it reports that the device is out of memory, nothing of it outlives a
device reset, and no call waits for the whole device (which would invalidate a
stream capture elsewhere in the process).
"""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_blocks_on_fake_cuda(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda.h")):
        inc = "/usr/local/cuda/include"
    csrc = os.path.join(ROOT, "paper_2007_14283_gb300", "csrc")
    exe = str(tmp_path / "blocks")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", inc, "-I", csrc, "-x", "c++",
                    os.path.join(csrc, "ms_blocks.cu"), os.path.join(ROOT, "tests", "native", "blocks_on_fakes.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
