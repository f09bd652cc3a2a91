"""Cell offsets of the largest grids (up to 2^31 - 1 cells, as the create call
accepts them), computed on the CPU with the code the kernels use."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc")
    inc = os.path.join(os.path.dirname(os.path.dirname(nvcc)) if nvcc else CUDA, "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("index")
    src = d / "index.cpp"
    src.write_text('#include "fvm_internal.h"\n'
                   'extern "C" int plane_above(int o, int nxy, int n) '
                   '{ return fvm::plane_above(o, nxy, n); }\n')
    so = str(d / "index.so")
    csrc = os.path.join(ROOT, "paper_2209_09671_gb300", "csrc")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-fwrapv", "-shared", "-fPIC", "-I", csrc, "-I", inc,
                        str(src), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


@pytest.mark.parametrize("nxy,nz", [(4 * 4, 4), (1024 * 1024, 2047), (1290 * 1290, 1290),
                                    (46340 * 11585, 4), (4 * 5, 107374182)])
def test_plane_above(lib, nxy, nz):
    n = nxy * nz
    assert n < 2 ** 31
    for k in (0, 1, nz // 2, nz - 3, nz - 2, nz - 1):
        for q in (0, 1, nxy // 2, nxy - 1):
            assert lib.plane_above(k * nxy + q, nxy, n) == (k + 1) % nz * nxy + q
