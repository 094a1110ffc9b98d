"""A small CUDA library of a test's own, built where the test runs."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build(source, tmp_path):
    """Compile `source` (CUDA C++, the library's headers on the include path) and load it."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.fail("nvcc is needed to build this test's kernels")
    src, so = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text(source)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", os.path.join(ROOT, "paper_1008_0861_gb300", "csrc"), "-o", str(so), str(src)],
                   check=True)
    return ctypes.CDLL(str(so))
