// The renumbering along a Morton (Z-order) curve and the candidate CSR in that
// order.  A contiguous node range is then a compact patch of the plane, and most
// neighbours of its nodes lie inside it: the GDP tiles, the batch kernels, the
// finisher's blocks and the pricing scan's blocks are such ranges.  Jacobi sweeps
// do not depend on node order, so the renumbering changes no value.
#include <climits>
#include <vector>

#include "f2m_device.cuh"
#include "f2m_internal.h"

namespace f2m {

#define F2M_GRID_STRIDE(i, count) \
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (count); \
       i += (long long)gridDim.x * blockDim.x)

static inline int grid_for(long long items, int threads) {
  long long b = (items + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 8192) b = 8192;
  return (int)b;
}

// ---- spatial renumbering ---------------------------------------------------------

// key = segment * 2^40 + Morton code (bit b of x at position 2b, bit b of y at
// 2b+1; x, y < 2^20), so nodes stay grouped by segment (instance) and follow a
// Morton curve inside each
__global__ void morton_kernel(const int2* __restrict__ xy, int32_t n, const int32_t* __restrict__ seg_off,
                              int32_t nseg, uint64_t* key, int32_t* idx) {
  F2M_GRID_STRIDE(v, n) {
    const unsigned x = (unsigned)xy[v].x, y = (unsigned)xy[v].y;
    uint64_t code = 0;
#pragma unroll
    for (int b = 0; b < 20; ++b)
      code |= ((uint64_t)((x >> b) & 1u) << (2 * b)) | ((uint64_t)((y >> b) & 1u) << (2 * b + 1));
    int lo = 0, hi = nseg - 1;  // segment of v: last s with seg_off[s] <= v
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (seg_off[mid] <= v) lo = mid; else hi = mid - 1;
    }
    key[v] = ((uint64_t)lo << 40) | code;
    idx[v] = (int32_t)v;
  }
}

__global__ void invert_perm_kernel(const int32_t* __restrict__ perm, int32_t n, int32_t* inv) {
  F2M_GRID_STRIDE(i, n) inv[perm[i]] = (int32_t)i;
}

__global__ void internal_degree_kernel(const int32_t* __restrict__ rp, const int32_t* __restrict__ perm,
                                       int32_t n, int32_t* ideg) {
  F2M_GRID_STRIDE(i, n) {
    const int v = perm[i];
    ideg[i] = rp[v + 1] - rp[v];
  }
}

// 13 -> 11 us at 100,000 points with eight lanes a row
__global__ void internal_rows_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec,
                                     const int32_t* __restrict__ perm, const int32_t* __restrict__ inv,
                                     const int32_t* __restrict__ irp, int32_t n, int2* __restrict__ iec) {
  F2M_ROWS(i, sub, n) {
    const int v = perm[i];
    const int a = rp[v], cnt = rp[v + 1] - a, o = irp[i];
    for (int k = sub; k < cnt; k += kRowLanes) {
      const int2 q = ec[a + k];
      iec[o + k] = make_int2(inv[q.x], q.y);
    }
  }
}

__global__ void gather_perm_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ perm,
                                   int32_t n, int32_t* __restrict__ dst) {
  F2M_GRID_STRIDE(i, n) dst[i] = src[perm[i]];
}

__global__ void scatter_perm_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ perm,
                                    int32_t n, int32_t* __restrict__ dst) {
  F2M_GRID_STRIDE(i, n) dst[perm[i]] = src[i];
}

#define PCK(x)                             \
  do {                                     \
    cudaError_t e_ = (x);                  \
    if (e_ != cudaSuccess) return e_;      \
  } while (0)

template <typename T>
static cudaError_t grow(T** p, int64_t* cap, int64_t need) {
  return dev_regrow(p, cap, need, need + (need >> 3) + 64);
}

void plan_free(GdpPlan& p) {
  void* ptrs[] = {p.perm, p.inv, p.irp, p.iec, p.ilam[0], p.ilam[1], p.keys, p.keys2, p.idx, p.sort_tmp, p.scan_tmp};
  for (void* q : ptrs)
    if (q) dev_free(q);
  p = GdpPlan();
}

cudaError_t plan_renumber(const int2* xy, int32_t n, const std::vector<int32_t>& seg_off, GdpPlan& p,
                          cudaStream_t st) {
  int64_t cap = 0;
  const int32_t nseg = (int32_t)seg_off.size() - 1;
  int32_t* d_seg = nullptr;  // not read for one segment
  if (nseg > 1) {
    PCK(dev_malloc((void**)&d_seg, sizeof(int32_t) * seg_off.size()));
    cudaError_t e0 = cudaMemcpyAsync(d_seg, seg_off.data(), sizeof(int32_t) * seg_off.size(),
                                     cudaMemcpyHostToDevice, st);
    if (e0 != cudaSuccess) { dev_free(d_seg); return e0; }
  }
  int end_bit = 40;
  while ((1LL << (end_bit - 40)) < nseg) ++end_bit;
  PCK(grow(&p.perm, &cap, n)); cap = 0;
  PCK(grow(&p.inv, &cap, n)); cap = 0;
  PCK(grow(&p.keys, &cap, n)); cap = 0;
  PCK(grow(&p.keys2, &cap, n)); cap = 0;
  PCK(grow(&p.idx, &cap, n));
  morton_kernel<<<grid_for(n, 256), 256, 0, st>>>(xy, n, d_seg, nseg, p.keys, p.idx);
  count_launch();
  cudaError_t e1 = cudaGetLastError();
  if (d_seg) {
    if (e1 == cudaSuccess) e1 = cudaStreamSynchronize(st);
    dev_free(d_seg);
  }
  PCK(e1);
  size_t bytes = 0;
  PCK(sort_pairs_u64(nullptr, bytes, p.keys, p.keys2, p.idx, p.perm, n, end_bit, st));
  PCK(dev_malloc(&p.sort_tmp, bytes > 0 ? bytes : 1));
  PCK(sort_pairs_u64(p.sort_tmp, bytes, p.keys, p.keys2, p.idx, p.perm, n, end_bit, st));
  count_launch();
  invert_perm_kernel<<<grid_for(n, 256), 256, 0, st>>>(p.perm, n, p.inv);
  count_launch();
  PCK(cudaGetLastError());
  p.n = n;
  return cudaSuccess;
}

cudaError_t gather_perm(const int32_t* src, const int32_t* perm, int32_t n, int32_t* dst,
                        cudaStream_t st) {
  gather_perm_kernel<<<grid_for(n, 256), 256, 0, st>>>(src, perm, n, dst);
  count_launch();
  return cudaGetLastError();
}

cudaError_t scatter_perm(const int32_t* src, const int32_t* perm, int32_t n, int32_t* dst,
                         cudaStream_t st) {
  scatter_perm_kernel<<<grid_for(n, 256), 256, 0, st>>>(src, perm, n, dst);
  count_launch();
  return cudaGetLastError();
}

cudaError_t plan_room(int32_t n, int64_t nnz, GdpPlan& p) {
  PCK(grow(&p.irp, &p.irp_cap, (int64_t)n + 1));
  PCK(grow(&p.iec, &p.iec_cap, nnz));
  PCK(grow(&p.ilam[0], &p.ilam_cap[0], n));
  PCK(grow(&p.ilam[1], &p.ilam_cap[1], n));
  PCK(grow(&p.scan_tmp, &p.scan_cap, (int64_t)scan_scratch_ints(n) + 1));
  return cudaSuccess;
}

cudaError_t plan_merge(const int2* xy, const int32_t* rp, const int2* ec_in, const int2* pairs, int64_t npairs,
                       int32_t n, int64_t nnz, MergeBuffers& mb, int2* ec_out, GdpPlan& p, cudaStream_t st) {
  PCK(plan_room(n, nnz, p));
  PCK(launch_merge_new(xy, rp, ec_in, pairs, npairs, n, mb, p.perm, p.inv, p.scan_tmp, ec_out, p.irp, p.iec, st));
  p.version += 1;
  p.n = n;
  p.nnz = nnz;
  return cudaSuccess;
}

cudaError_t plan_build(const int32_t* rp, const int2* ec, int32_t n, int64_t nnz, GdpPlan& p, cudaStream_t st) {
  p.version += 1;
  PCK(plan_room(n, nnz, p));
  // internal CSR: rows in renumbered order, columns renumbered
  int32_t* ideg = p.ilam[1];  // free until the phase starts
  internal_degree_kernel<<<grid_for(n, 256), 256, 0, st>>>(rp, p.perm, n, ideg);
  count_launch();
  PCK(cudaGetLastError());
  PCK(launch_scan(ideg, p.irp, n, p.scan_tmp, st));
  internal_rows_kernel<<<grid_for((long long)n * kRowLanes, 256), 256, 0, st>>>(rp, ec, p.perm, p.inv, p.irp, n, p.iec);
  count_launch();
  PCK(cudaGetLastError());
  p.n = n;
  p.nnz = nnz;
  return cudaSuccess;
}

}  // namespace f2m
