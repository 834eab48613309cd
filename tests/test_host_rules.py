"""Decisions that the library makes on the host, without a GPU: which arrays a kernel
may write to, what a work array says of itself after an allocation failed, how many
block pairs a culled scan lists, and which graphs are not tried on tiles."""
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


OK, HELD, COVERS = 1, 2, 4


@pytest.mark.parametrize("had,need,room,blocks,want", [
    (0, 10, 15, 1, OK | HELD | COVERS),   # the first block
    (20, 10, 15, 0, OK | HELD | COVERS),  # large enough
    (5, 10, 15, 1, OK | HELD | COVERS),   # replaced
    (5, 10, 15, 0, 0),                    # no memory: nothing held, and none claimed
    (0, 10, 15, 0, 0)])
def test_a_failed_allocation_claims_no_room(rules, had, need, room, blocks, want):
    # a capacity noted before the allocation had the next call write through a null pointer
    rules.shim_grow.argtypes = [C.c_longlong] * 3 + [C.c_int]
    assert rules.shim_grow(had, need, room, blocks) == want


OLD = 8


@pytest.mark.parametrize("had,need,room,blocks,want", [
    (0, 10, 15, 1, OK | HELD | COVERS), (20, 10, 15, 0, OK | HELD | COVERS | OLD), (5, 10, 15, 1, OK | HELD | COVERS),
    (5, 10, 15, 0, HELD | OLD),  # no memory: the graph keeps its arrays
    (0, 10, 15, 0, 0)])
def test_a_failed_merge_leaves_the_graph_its_arrays(rules, had, need, room, blocks, want):
    # given back first, the renumbered graph was gone and the next sweep read through null
    rules.shim_regrow.argtypes = [C.c_longlong] * 3 + [C.c_int]
    assert rules.shim_regrow(had, need, room, blocks) == want


def test_no_capacity_is_noted_before_its_allocation():
    # the sources: a member's capacity is assigned from its size only after the block is there
    import re
    for name in ("api.cu", "batch.cu", "cuts.cu"):
        src = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"(\w+->(\w+)_cap) = (?!0;)[^;]*;\s*CK\(c, dalloc\(&\w+->d_\w+, \1\)\)", src):
            raise AssertionError(f"{name}: {m.group(0)}")


@pytest.mark.parametrize("listed", [0, 1, 4096, 1 << 20, (1 << 31) - 2])
def test_a_listed_scan_gets_room(rules, listed):
    rules.shim_price_list_room.argtypes, rules.shim_price_list_room.restype = [C.c_ulonglong], C.c_longlong
    assert listed <= rules.shim_price_list_room(listed) < 1 << 31


@pytest.mark.parametrize("listed", [(1 << 31) - 1, 1 << 31, (1 << 32) - 1, 1 << 32, (1 << 32) + 5, 8_590_000_128])
def test_a_list_past_the_handed_out_numbers_is_refused(rules, listed):
    # 2^24 points make 131,072 blocks, 8.6e9 pairs of them: clamped to 2^31 - 1 the
    # scan and its list never met, and past 2^32 a 32-bit count wrapped
    rules.shim_price_list_room.argtypes, rules.shim_price_list_room.restype = [C.c_ulonglong], C.c_longlong
    assert rules.shim_price_list_room(listed) == 0


SMEM = 232_448 - 128  # a CTA's shared memory


@pytest.mark.parametrize("n,degree,half,want", [
    (1000, 12, False, True), (200_000, 14, False, True), (301_568, 40, False, True),  # 1,984 rows a tile: registers
    (301_569, 60, False, False), (550_000, 12, False, True), (600_000, 13, False, False), (700_000, 7, False, True),
    (1_300_000, 3, False, False), (2_000_000, 12, False, False), (1 << 24, 3, False, False),
    (200_000, 12, True, True), (301_568, 60, True, False)])
def test_what_no_tile_can_hold_is_not_tried(rules, n, degree, half, want):
    rules.shim_ring_can_fit.argtypes = [C.c_longlong] * 4 + [C.c_int]
    tiles = 304 if half else 152
    assert bool(rules.shim_ring_can_fit(n, n * degree, tiles, SMEM // 2 if half else SMEM, half)) == want
