"""The launch groups of the re-delivery fast path's full comparisons (csrc/cm_dedup_groups.h),
on the CPU: fragments that start at one address but differ in size are compared apart, each
copy over its own length."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_copies_are_compared_over_their_own_size(tmp_path):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc))) if nvcc else "/usr/local/cuda"
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "dedup_groups_check")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Wextra", "-Werror", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2607_01308_gb300", "csrc"), "-isystem",
                    os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "dedup_groups_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout
