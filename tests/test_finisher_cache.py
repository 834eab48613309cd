"""The cache of the host finisher's work arrays on the CPU: what a context of a size
takes from it, and that its bound covers all that the arrays hold."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2011_08170_gb300", "csrc")


@pytest.fixture
def cache(tmp_path):
    inc = "/usr/local/cuda/include"
    cxx = shutil.which("g++")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")) or cxx is None:
        pytest.skip("needs g++ and the CUDA headers (for the types the library's headers use)")
    out = str(tmp_path / "libcache.so")  # a library, and with it an empty cache, of each test's own
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", CSRC, "-I", inc,
                    os.path.join(os.path.dirname(__file__), "finisher_cache_shim.cpp"), "-o", out],
                   check=True, capture_output=True)
    L = C.CDLL(out)
    L.shim_take.restype = C.c_void_p
    for f in (L.shim_free, L.shim_nodes):
        f.argtypes = [C.c_void_p]
    L.shim_search.argtypes = [C.c_void_p, C.c_int64]
    for f in (L.shim_nodes, L.shim_cached_search_bytes, L.shim_cache_max):
        f.restype = C.c_int64
    return L


@pytest.mark.parametrize("held,n,taken", [(1_600_000, 1000, False), (1_600_000, 799_999, False),
                                          (1_600_000, 800_000, True), (1_600_000, 1_600_000, True),
                                          (1_600_000, 1_600_001, False), (16_384, 4, True), (16_385, 4, False)])
def test_a_context_takes_arrays_of_its_size(cache, held, n, taken):
    w = cache.shim_take(held)
    cache.shim_free(w)
    assert (cache.shim_nodes(cache.shim_take(n)) == held) == taken


def test_the_bound_covers_heaps_and_lists(cache):
    items = 4_000_000  # 80 MB of heap and list
    works = [cache.shim_take(1000) for _ in range(8)]
    for w in works:
        cache.shim_search(w, items)
    for w in works:
        cache.shim_free(w)
    assert 0 < cache.shim_cached_search_bytes() <= cache.shim_cache_max()


def test_copies_without_threads(tmp_path):
    # an exception out of a C entry point would end the caller's process
    inc, cxx = "/usr/local/cuda/include", shutil.which("g++")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")) or cxx is None or (os.cpu_count() or 1) < 2:
        pytest.skip("needs g++, the CUDA headers and a second core")
    exe = str(tmp_path / "copy")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, "-I", inc,
                    os.path.join(os.path.dirname(__file__), "host_copy_main.cpp"), os.path.join(CSRC, "finisher.cpp"),
                    "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "copied\n", (r.returncode, r.stderr)


def test_what_is_freed_last_is_kept(cache):
    # a block near the bound (2.9 M nodes, 255 MB) makes room for others
    cache.shim_free(cache.shim_take(2_900_000))
    sizes = [400_000, 150_000, 50_000]
    for n in sizes:
        cache.shim_free(cache.shim_take(n))
    assert [cache.shim_nodes(cache.shim_take(n - 1)) for n in sizes] == sizes
    many = [cache.shim_take(20_000 + 100 * i) for i in range(70)]  # more than 64: the first six go
    for w in many:
        cache.shim_free(w)
    assert cache.shim_nodes(cache.shim_take(20_000)) == 20_600
