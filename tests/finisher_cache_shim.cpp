// C entry points to the cache of the host finisher's work arrays, for CPU tests.
// The sizes are private to finisher.cpp, so that file is part of this one.
#include "finisher.cpp"

using namespace f2m;

extern "C" {
void* shim_take(int32_t n) { return finisher_work_take(n); }
void shim_free(void* w) { finisher_work_free(static_cast<FinisherWork*>(w)); }
int64_t shim_nodes(void* w) { return (int64_t)static_cast<FinisherWork*>(w)->pi.size() / 2; }
// as a search of `items` pushes leaves its worker
void shim_search(void* w, int64_t items) {
  auto* f = static_cast<FinisherWork*>(w);
  f->workers.resize(1);
  f->workers[0].heap.reserve((size_t)items);
  f->workers[0].order.reserve((size_t)items);
}
// bytes of heap and list capacity that the cache holds beside the node arrays
int64_t shim_cached_search_bytes() {
  int64_t b = 0;
  for (const FinisherWork* w : g_work_free)
    for (const Searcher& s : w->workers) b += (int64_t)(s.heap.capacity() * 16 + s.order.capacity() * 4);
  return b;
}
int64_t shim_cache_max() { return (int64_t)kWorkCacheMax; }
}
