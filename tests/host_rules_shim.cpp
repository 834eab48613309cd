// C entry points to decisions of the library that are made on the host, for CPU
// tests (tests/test_host_rules.py builds this file with g++).
#include "f2m_internal.h"

extern "C" int shim_kernel_reaches(int type, int device, int current) {
  return f2m::kernel_reaches((cudaMemoryType)type, device, current);
}
