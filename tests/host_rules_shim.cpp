// C entry points to decisions of the library that are made on the host, for CPU
// tests (tests/test_host_rules.py builds this file with g++).
#include <cstdlib>

#include "ctx_internal.h"

// the library's allocator, with a budget of blocks
static int g_blocks = 0;
namespace f2m {
cudaError_t dev_malloc(void** p, size_t bytes) {
  if (g_blocks-- <= 0) return cudaErrorMemoryAllocation;
  *p = std::malloc(bytes);
  return cudaSuccess;
}
void dev_free(void* p) { std::free(p); }
void dev_free_synced(void* p) { std::free(p); }
}  // namespace f2m

extern "C" int shim_kernel_reaches(int type, int device, int current) {
  return f2m::kernel_reaches((cudaMemoryType)type, device, current);
}

// dgrow on an array that holds `had` items (0: none), with `blocks` blocks left:
// bit 0 success, bit 1 a block is held, bit 2 the capacity covers `need`
extern "C" int shim_grow(long long had, long long need, long long room, int blocks) {
  int* p = nullptr;
  int64_t cap = 0;
  g_blocks = 1;
  if (had) f2m::dalloc(&p, had);
  cap = had;
  g_blocks = blocks;
  const bool ok = f2m::dgrow(&p, &cap, need, room) == cudaSuccess;
  const int r = ok | (p != nullptr) << 1 | (cap >= need) << 2;
  std::free(p);
  return r;
}

// dev_regrow: bit 0 success, bit 1 a block is held, bit 2 the capacity covers `need`,
// bit 3 the block is the old one
extern "C" int shim_regrow(long long had, long long need, long long room, int blocks) {
  int* p = nullptr;
  int64_t cap = 0;
  g_blocks = 1;
  if (had) f2m::dev_regrow(&p, &cap, had, had);
  const int* old = p;
  g_blocks = blocks;
  const bool ok = f2m::dev_regrow(&p, &cap, need, room) == cudaSuccess;
  const int r = ok | (p != nullptr) << 1 | (cap >= need) << 2 | (had && p == old) << 3;
  std::free(p);
  return r;
}

extern "C" long long shim_price_list_room(unsigned long long listed) { return f2m::price_list_room(listed); }

extern "C" int shim_ring_can_fit(long long n, long long nnz, long long tiles, long long smem, int half) {
  return f2m::ring_can_fit(n, nnz, tiles, smem, half != 0);
}
