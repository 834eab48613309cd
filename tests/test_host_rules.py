"""Decisions that the library makes on the host, without a GPU: which arrays a kernel
may write to."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2011_08170_gb300", "csrc")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    inc = [d for d in (os.path.join(os.environ.get("CUDA_HOME", ""), "include"), "/usr/local/cuda/include")
           if os.path.exists(os.path.join(d, "cuda_runtime.h"))]
    cxx = shutil.which("g++")
    if not inc or cxx is None:
        pytest.skip("needs g++ and the CUDA headers (for the types the library's headers use)")
    out = str(tmp_path_factory.mktemp("rules") / "librules.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", inc[0],
                    os.path.join(os.path.dirname(__file__), "host_rules_shim.cpp"), "-o", out],
                   check=True, capture_output=True)
    return C.CDLL(out)


UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3  # cudaMemoryType


@pytest.mark.parametrize("kind,device,current,want", [
    (DEVICE, 0, 0, True), (DEVICE, 1, 0, False), (DEVICE, 0, 1, False), (DEVICE, 3, 3, True),
    (MANAGED, 0, 0, True), (MANAGED, 1, 0, True), (HOST, 0, 0, False), (UNREGISTERED, 0, 0, False)])
def test_kernels_write_only_where_they_reach(rules, kind, device, current, want):
    # a read-out's kernel stores to arrays on its own GPU; another GPU's take a copy
    assert bool(rules.shim_kernel_reaches(kind, device, current)) == want
