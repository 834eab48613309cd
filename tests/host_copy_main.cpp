// host_copy of the library where no thread can be made (pthread_create fails, as at a
// limit on processes): the copies are made all the same, by the caller.
#include <pthread.h>

#include <cerrno>
#include <cstdio>
#include <vector>

#include "f2m_internal.h"

extern "C" int pthread_create(pthread_t*, const pthread_attr_t*, void* (*)(void*), void*) { return EAGAIN; }

int main() {
  std::vector<unsigned> src(8 << 20), dst(src.size(), 0);  // 32 MB: enough for the workers
  for (size_t i = 0; i < src.size(); ++i) src[i] = (unsigned)(i * 2654435761u);
  const size_t half = src.size() / 2 + 3;
  f2m::host_copy({{dst.data(), src.data(), half * 4},
                  {dst.data() + half, src.data() + half, (src.size() - half) * 4}});
  if (dst != src) return 1;
  std::puts("copied");
}
