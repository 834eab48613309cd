// Candidate-graph kernels: input validation, the cost table, and the union of
// the CSR with the pairs found by pricing (rows kept sorted and unique, so the
// result does not depend on the order in which pairs were appended).
#include <climits>

#include "f2m_device.cuh"
#include "f2m_internal.h"

namespace f2m {

static inline int grid_for(long long items, int threads) {
  long long b = (items + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 8192) b = 8192;
  return (int)b;
}

#define F2M_GRID_STRIDE(i, count) \
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (count); \
       i += (long long)gridDim.x * blockDim.x)

__device__ __forceinline__ void flag(CheckCtl* ctl, int bit, long long where) {
  atomicOr(&ctl->flags, bit);
  atomicMin(&ctl->first_bad, (int)(where < INT_MAX ? where : INT_MAX));
}

// pass 1: row offsets monotone and in [0, nnz], coordinates in range; nnz = rp[n]
// goes to the host with the verdict
__global__ void check_rowptr_kernel(const int2* xy, const int32_t* rp, int32_t n, CheckCtl* ctl) {
  const int32_t nnz = rp[n];
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl[1].flags = nnz;
  F2M_GRID_STRIDE(v, n) {
    const int a = rp[v], b = rp[v + 1];
    if (a < 0 || b < a || b > nnz || (v == 0 && a != 0))
      flag(ctl, kBadRowPtr, v);
    const int2 p = xy[v];
    if (p.x < 0 || p.y < 0 || p.x >= kCoordLimit || p.y >= kCoordLimit) flag(ctl, kBadCoord, v);
  }
}

// coordinates only (for calls that take points without a graph)
__global__ void check_points_kernel(const int2* xy, int32_t n, CheckCtl* ctl) {
  F2M_GRID_STRIDE(v, n) {
    const int2 p = xy[v];
    if (p.x < 0 || p.y < 0 || p.x >= kCoordLimit || p.y >= kCoordLimit) flag(ctl, kBadCoord, v);
  }
}

// pass 2 (row offsets valid): columns, order, self-loops, degree, symmetry.
// Eight lanes a row (see F2M_ROWS), each with a search of its own in flight:
// 28 -> 21 us at 100,000 points and 10 neighbours, 16 -> 6 at 1,000.
__global__ void check_rows_kernel(const int32_t* rp, const int32_t* col, int32_t n, CheckCtl* ctl) {
  F2M_ROWS(v, sub, n) {
    const int a = rp[v], b = rp[v + 1];
    if (b - a < 3 && sub == 0) flag(ctl, kLowDegree, v);
    for (int e = a + sub; e < b; e += kRowLanes) {
      const int c = col[e];
      if (c < 0 || c >= n) { flag(ctl, kBadCol, v); continue; }
      if (c == v) flag(ctl, kSelfLoop, v);
      int p = e - 1;  // the last entry before this one that names a node
      while (p >= a && (col[p] < 0 || col[p] >= n)) --p;
      if (p >= a && c <= col[p]) flag(ctl, kUnsorted, v);
      // reverse entry (c -> v) must exist; row c is searched only if sorted
      int lo = rp[c], hi = rp[c + 1] - 1, found = 0;
      while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int cm = col[mid];
        if (cm == v) { found = 1; break; }
        if (cm < v) lo = mid + 1; else hi = mid - 1;
      }
      if (!found) {
        // unsorted rows make binary search unreliable; fall back to a scan
        for (int f = rp[c]; f < rp[c + 1] && !found; ++f) found = (col[f] == v);
        if (!found) flag(ctl, kAsymmetric, v);
      }
    }
  }
}

cudaError_t launch_check_points(const int2* xy, int32_t n, CheckCtl* ctl, cudaStream_t st) {
  check_points_kernel<<<grid_for(n, 256), 256, 0, st>>>(xy, n, ctl);
  count_launch();
  return cudaGetLastError();
}

// degree requirements: 1 <= b_v and b_v + 1 <= deg(v) (the (b_v+1)-th value of
// the row must exist, Section 3)
__global__ void check_degrees_kernel(const int32_t* rp, const int32_t* bdeg, int32_t n, CheckCtl* ctl,
                                     unsigned long long* bmax) {
  F2M_GRID_STRIDE(v, n) {
    const int bv = bdeg[v];
    if (bv < 1 || (long long)bv + 1 > (long long)rp[v + 1] - rp[v]) flag(ctl, kBadDegreeReq, v);
    else atomicMax(bmax, (unsigned long long)bv);
  }
}

cudaError_t launch_check_degrees(const int32_t* rp, const int32_t* bdeg, int32_t n, CheckCtl* ctl,
                                 unsigned long long* bmax, cudaStream_t st) {
  check_degrees_kernel<<<grid_for(n, 256), 256, 0, st>>>(rp, bdeg, n, ctl, bmax);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_check(const int2* xy, const int32_t* rp, const int32_t* col, int32_t n, CheckCtl* ctl,
                         cudaStream_t st) {
  // two passes; the host reads ctl between them (pass 2 trusts the row offsets)
  if (col == nullptr) {
    check_rowptr_kernel<<<grid_for(n, 256), 256, 0, st>>>(xy, rp, n, ctl);
    count_launch();
  } else {
    check_rows_kernel<<<grid_for((long long)n * kRowLanes, 256), 256, 0, st>>>(rp, col, n, ctl);
    count_launch();
  }
  return cudaGetLastError();
}

// ec[e] = {col[e], c(v, col[e])}: 25 -> 12 us at 100,000 points (a thread per entry
// searched the row offsets for its row)
__global__ void build_ec_kernel(const int2* __restrict__ xy, const int32_t* __restrict__ rp,
                                const int32_t* __restrict__ col, int32_t n, int2* __restrict__ ec) {
  F2M_ROWS(v, sub, n) {
    const int2 pv = xy[v];
    for (int e = rp[v] + sub, b = rp[v + 1]; e < b; e += kRowLanes) {
      const int c = col[e];
      ec[e] = make_int2(c, exact_cost(pv, xy[c]));
    }
  }
}

cudaError_t launch_build_ec(const int2* xy, const int32_t* rp, const int32_t* col, int32_t n,
                            int2* ec, cudaStream_t st) {
  build_ec_kernel<<<grid_for((long long)n * kRowLanes, 256), 256, 0, st>>>(xy, rp, col, n, ec);
  count_launch();
  return cudaGetLastError();
}

// ---- exclusive scan of int32 (m+1 outputs, out[m] = total) -------------------
//
// Two launches: the sum of each tile, then each tile's scan, whose block adds up
// the sums before it by itself (at most 4,096 of them for 2^24 items; the second
// read of the items comes from L2).  One launch when one tile holds all.  A warp
// takes 256 consecutive items, 32 at a time.  Three launches (tile scans, a scan
// of the sums, a pass that added them) took 17 us at 100,000 items and 11 us at
// 1,000, the addition alone 10: now 8 and 3.

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;  // per lane
constexpr int kScanBlock = kScanThreads * kScanItems;

size_t scan_scratch_ints(int32_t m) { return (size_t)(((long long)m + kScanBlock - 1) / kScanBlock) + 1; }

template <typename In>
__device__ __forceinline__ void scan_sum(const In& in, int32_t m, int32_t* __restrict__ sums) {
  __shared__ int s_warp[33];
  const long long base = (long long)blockIdx.x * kScanBlock;
  int sum = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const long long i = base + k * kScanThreads + threadIdx.x;
    if (i < m) sum += in(i);
  }
  int total;
  block_exclusive_scan(sum, s_warp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

template <typename In>
__device__ __forceinline__ void scan_tile(const In& in, int32_t* __restrict__ out, int32_t m,
                                          const int32_t* __restrict__ sums) {
  __shared__ int s_warp[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0;
  if (blockIdx.x) {
    int before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += sums[b];
    block_exclusive_scan(before, s_warp, carry);
  }
  const long long base = (long long)blockIdx.x * kScanBlock + warp * 32 * kScanItems + lane;
  int v[kScanItems], run = 0;  // v: sums of this warp's items up to and with this one
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) v[k] = base + k * 32 < m ? in(base + k * 32) : 0;
  int own[kScanItems];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    own[k] = v[k];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v[k], o);
      if (lane >= o) v[k] += y;
    }
    v[k] += run;
    run = __shfl_sync(0xffffffffu, v[k], 31);
  }
  int total;
  const int warp_base = __shfl_sync(0xffffffffu, block_exclusive_scan(lane == 0 ? run : 0, s_warp, total), 0);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (base + k * 32 < m) out[base + k * 32] = carry + warp_base + v[k] - own[k];
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[m] = carry + total;
}

struct ScanArray {
  const int32_t* p;
  __device__ __forceinline__ int operator()(long long i) const { return p[i]; }
};

__global__ void __launch_bounds__(kScanThreads)
scan_sums_kernel(const int32_t* in, int32_t m, int32_t* sums) {
  scan_sum(ScanArray{in}, m, sums);
}

__global__ void __launch_bounds__(kScanThreads)
scan_tiles_kernel(const int32_t* in, int32_t* out, int32_t m, const int32_t* sums) {
  scan_tile(ScanArray{in}, out, m, sums);
}

cudaError_t launch_scan(const int32_t* in, int32_t* out, int32_t m, int32_t* block_sums,
                        cudaStream_t st) {
  const int nb = (int)(((long long)m + kScanBlock - 1) / kScanBlock);
  if (nb == 0) return cudaMemsetAsync(out, 0, sizeof(int32_t), st);
  if (nb > 1) {
    scan_sums_kernel<<<nb, kScanThreads, 0, st>>>(in, m, block_sums);
    count_launch();
  }
  scan_tiles_kernel<<<nb, kScanThreads, 0, st>>>(in, out, m, block_sums);
  count_launch();
  return cudaGetLastError();
}

// ---- merge: CSR u pairs ---------------------------------------------------------

__global__ void merge_degree_kernel(const int32_t* __restrict__ rp, int32_t n, int32_t* deg) {
  F2M_GRID_STRIDE(v, n) deg[v] = rp[v + 1] - rp[v];
}

__global__ void merge_count_kernel(const int2* __restrict__ pairs, long long npairs, int32_t n,
                                   int32_t* deg, CheckCtl* ctl) {
  F2M_GRID_STRIDE(k, npairs) {
    const int2 p = pairs[k];
    if (p.x < 0 || p.y < 0 || p.x >= n || p.y >= n || p.x == p.y) {
      flag(ctl, kBadPair, k);
      continue;
    }
    atomicAdd(&deg[p.x], 1);
    atomicAdd(&deg[p.y], 1);
  }
}

cudaError_t launch_merge_count(const int32_t* rp, const int2* pairs, int64_t npairs, int32_t n,
                               MergeBuffers& mb, cudaStream_t st) {
  merge_degree_kernel<<<grid_for(n, 256), 256, 0, st>>>(rp, n, mb.deg);
  count_launch();
  if (npairs > 0) {
    merge_count_kernel<<<grid_for(npairs, 256), 256, 0, st>>>(pairs, npairs, n, mb.deg, mb.ctl);
    count_launch();
  }
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  return launch_scan(mb.deg, mb.tmp_rp, n, mb.block_sums, st);
}

// Rows are strictly increasing (checked when the graph is created, and kept
// so by every merge), so a row that no pair touches comes out of the merge as
// it went in: only the touched rows (those that gained room in tmp_rp) are
// copied, sorted and deduplicated in tmp_col; the others keep their entries.
__device__ __forceinline__ bool merge_touched(const int32_t* rp, const int32_t* tmp_rp, int v) {
  return tmp_rp[v + 1] - tmp_rp[v] != rp[v + 1] - rp[v];
}

// copy a touched row's old entries to the front of its new row; deg becomes
// the append cursor
__global__ void merge_copy_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec,
                                  int32_t n, const int32_t* __restrict__ tmp_rp, int32_t* tmp_col,
                                  int32_t* cursor) {
  F2M_GRID_STRIDE(v, n) {
    if (!merge_touched(rp, tmp_rp, (int)v)) continue;
    const int a = rp[v], b = rp[v + 1], o = tmp_rp[v];
    for (int e = a; e < b; ++e) tmp_col[o + (e - a)] = ec[e].x;
    cursor[v] = o + (b - a);
  }
}

__global__ void merge_scatter_kernel(const int2* __restrict__ pairs, long long npairs, int32_t n,
                                     int32_t* tmp_col, int32_t* cursor) {
  F2M_GRID_STRIDE(k, npairs) {
    const int2 p = pairs[k];
    if (p.x < 0 || p.y < 0 || p.x >= n || p.y >= n || p.x == p.y) continue;
    tmp_col[atomicAdd(&cursor[p.x], 1)] = p.y;
    tmp_col[atomicAdd(&cursor[p.y], 1)] = p.x;
  }
}

cudaError_t launch_merge_fill(const int32_t* rp, const int2* ec, const int2* pairs, int64_t npairs,
                              int32_t n, MergeBuffers& mb, cudaStream_t st) {
  merge_copy_kernel<<<grid_for(n, 256), 256, 0, st>>>(rp, ec, n, mb.tmp_rp, mb.tmp_col, mb.deg);
  count_launch();
  if (npairs > 0) {
    merge_scatter_kernel<<<grid_for(npairs, 256), 256, 0, st>>>(pairs, npairs, n, mb.tmp_col,
                                                                mb.deg);
    count_launch();
  }
  return cudaGetLastError();
}

// sort each touched row (insertion sort: rows are short) and count distinct
// columns; an untouched row keeps its length
__global__ void merge_sort_rows_kernel(const int32_t* __restrict__ rp, const int32_t* __restrict__ tmp_rp,
                                       int32_t* tmp_col, int32_t n, int32_t* uniq) {
  F2M_GRID_STRIDE(v, n) {
    const int a = tmp_rp[v], b = tmp_rp[v + 1];
    if (!merge_touched(rp, tmp_rp, (int)v)) {
      uniq[v] = b - a;
      continue;
    }
    for (int i = a + 1; i < b; ++i) {
      const int x = tmp_col[i];
      int j = i - 1;
      while (j >= a && tmp_col[j] > x) { tmp_col[j + 1] = tmp_col[j]; --j; }
      tmp_col[j + 1] = x;
    }
    int u = 0;
    for (int i = a; i < b; ++i) u += (i == a || tmp_col[i] != tmp_col[i - 1]);
    uniq[v] = u;
  }
}

// the merged rows into ec_out (another array than ec_in): an untouched row's
// entries as they were (its costs are the exact costs of its points), a
// touched row's distinct columns with their exact costs, each lane's entry after
// the distinct ones before it.  19.5 -> 9.8 us at 100,000 points, 15.8 -> 5.7 at
// 1,000 (where one lane's walk over a touched row was the kernel).
__global__ void merge_compact_kernel(const int2* __restrict__ xy, const int32_t* __restrict__ rp,
                                     const int2* __restrict__ ec_in, const int32_t* __restrict__ tmp_rp,
                                     const int32_t* __restrict__ tmp_col, int32_t n,
                                     const int32_t* __restrict__ new_rp, int2* __restrict__ ec_out) {
  F2M_ROWS(v, sub, n) {
    int o = new_rp[v];
    if (!merge_touched(rp, tmp_rp, (int)v)) {
      const int a = rp[v], cnt = rp[v + 1] - a;
      for (int k = sub; k < cnt; k += kRowLanes) ec_out[o + k] = ec_in[a + k];
      continue;
    }
    const int first = threadIdx.x & 31 & ~(kRowLanes - 1);
    const unsigned group = ((1u << kRowLanes) - 1u) << first;
    const int a = tmp_rp[v], b = tmp_rp[v + 1];
    const int2 pv = xy[v];
    for (int base = a; base < b; base += kRowLanes) {
      const int i = base + sub;
      const int c = i < b ? tmp_col[i] : 0;
      const bool keep = i < b && (i == a || tmp_col[i - 1] != c);
      const unsigned kept = __ballot_sync(group, keep) >> first;
      if (keep) ec_out[o + __popc(kept & ((1u << sub) - 1u))] = make_int2(c, exact_cost(pv, xy[c]));
      o += __popc(kept & ((1u << kRowLanes) - 1u));
    }
  }
}

cudaError_t launch_merge_finish(const int2* xy, const int32_t* rp, const int2* ec_in, int32_t n,
                                MergeBuffers& mb, int2* ec_out, cudaStream_t st) {
  merge_sort_rows_kernel<<<grid_for(n, 128), 128, 0, st>>>(rp, mb.tmp_rp, mb.tmp_col, n, mb.deg);
  count_launch();
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  err = launch_scan(mb.deg, mb.new_rp, n, mb.block_sums, st);
  if (err != cudaSuccess) return err;
  merge_compact_kernel<<<grid_for((long long)n * kRowLanes, 256), 256, 0, st>>>(xy, rp, ec_in, mb.tmp_rp, mb.tmp_col, n, mb.new_rp,
                                                         ec_out);
  count_launch();
  return cudaGetLastError();
}

// ---- merge of pairs that are distinct and outside the CSR --------------------------
//
// What a pricing scan finds.  No entry goes away, so the merged size is known
// beforehand and nothing has to be read back: the added columns are counted per
// row, the row lengths scanned in caller and in renumbered order by the same two
// launches, the added columns scattered behind their rows' places, and each row
// written to both edge arrays at once, every entry to the number of smaller ones
// (the old entries are in order).  Seven operations on the stream against fifteen
// with a wait in their middle: 97 -> 40 us at 30,000 points, 104 -> 50 at 100,000,
// 99 -> 28 at 1,000 (with the renumbered graph).

__global__ void merge_extra_kernel(const int2* __restrict__ pairs, long long npairs, int32_t* extra) {
  F2M_GRID_STRIDE(k, npairs) {
    const int2 p = pairs[k];
    atomicAdd(&extra[p.x], 1);
    atomicAdd(&extra[p.y], 1);
  }
}

struct MergedRow {  // entries of row i after the merge: in caller order, or (perm) in renumbered order
  const int32_t *rp, *extra, *perm;
  __device__ __forceinline__ int operator()(long long i) const {
    const int v = perm ? perm[i] : (int)i;
    return rp[v + 1] - rp[v] + extra[v];
  }
};

__global__ void __launch_bounds__(kScanThreads)
merge_sums_kernel(const int32_t* rp, const int32_t* extra, const int32_t* perm, int32_t n, int32_t* sums,
                  int32_t* isums) {
  const bool in = blockIdx.y;
  scan_sum(MergedRow{rp, extra, in ? perm : nullptr}, n, in ? isums : sums);
}

__global__ void __launch_bounds__(kScanThreads)
merge_tiles_kernel(const int32_t* rp, const int32_t* extra, const int32_t* perm, int32_t n, int32_t* new_rp,
                   int32_t* irp, const int32_t* sums, const int32_t* isums) {
  const bool in = blockIdx.y;
  scan_tile(MergedRow{rp, extra, in ? perm : nullptr}, in ? irp : new_rp, n, in ? isums : sums);
}

// extra counts down to zero
__global__ void merge_place_kernel(const int2* __restrict__ pairs, long long npairs, const int32_t* __restrict__ rp,
                                   const int32_t* __restrict__ new_rp, int32_t* extra, int32_t* __restrict__ tmp_col) {
  F2M_GRID_STRIDE(k, npairs) {
    const int2 p = pairs[k];
    tmp_col[new_rp[p.x] + rp[p.x + 1] - rp[p.x] + atomicSub(&extra[p.x], 1) - 1] = p.y;
    tmp_col[new_rp[p.y] + rp[p.y + 1] - rp[p.y] + atomicSub(&extra[p.y], 1) - 1] = p.x;
  }
}

__global__ void merge_rows_kernel(const int2* __restrict__ xy, const int32_t* __restrict__ rp,
                                  const int2* __restrict__ ec_in, const int32_t* __restrict__ new_rp,
                                  const int32_t* __restrict__ tmp_col, const int32_t* __restrict__ inv,
                                  const int32_t* __restrict__ irp, int32_t n, int2* __restrict__ ec_out,
                                  int2* __restrict__ iec) {
  F2M_ROWS(v, sub, n) {
    const int a = rp[v], m = rp[v + 1] - a, o = new_rp[v], x = new_rp[v + 1] - o - m, io = irp[inv[v]];
    const int32_t* added = tmp_col + o + m;
    for (int k = sub; k < m; k += kRowLanes) {
      const int2 q = ec_in[a + k];
      int r = k;
      for (int j = 0; j < x; ++j) r += added[j] < q.x;
      ec_out[o + r] = q;
      iec[io + r] = make_int2(inv[q.x], q.y);
    }
    for (int j = sub; j < x; j += kRowLanes) {
      const int c = added[j];
      int r = 0;
      for (int i = 0; i < x; ++i) r += added[i] < c;
      for (int i = 0; i < m; ++i) r += ec_in[a + i].x < c;
      const int cost = exact_cost(xy[v], xy[c]);
      ec_out[o + r] = make_int2(c, cost);
      iec[io + r] = make_int2(inv[c], cost);
    }
  }
}

cudaError_t launch_merge_new(const int2* xy, const int32_t* rp, const int2* ec_in, const int2* pairs, int64_t npairs,
                             int32_t n, MergeBuffers& mb, const int32_t* perm, const int32_t* inv, int32_t* isums,
                             int2* ec_out, int32_t* irp, int2* iec, cudaStream_t st) {
  cudaError_t err = cudaMemsetAsync(mb.deg, 0, sizeof(int32_t) * n, st);
  if (err != cudaSuccess) return err;
  const int nb = (int)(((long long)n + kScanBlock - 1) / kScanBlock);
  merge_extra_kernel<<<grid_for(npairs, 256), 256, 0, st>>>(pairs, npairs, mb.deg);
  if (nb > 1)
    merge_sums_kernel<<<dim3(nb, 2), kScanThreads, 0, st>>>(rp, mb.deg, perm, n, mb.block_sums, isums);
  merge_tiles_kernel<<<dim3(nb, 2), kScanThreads, 0, st>>>(rp, mb.deg, perm, n, mb.new_rp, irp, mb.block_sums, isums);
  merge_place_kernel<<<grid_for(npairs, 256), 256, 0, st>>>(pairs, npairs, rp, mb.new_rp, mb.deg, mb.tmp_col);
  merge_rows_kernel<<<grid_for((long long)n * kRowLanes, 256), 256, 0, st>>>(xy, rp, ec_in, mb.new_rp, mb.tmp_col, inv,
                                                                             irp, n, ec_out, iec);
  count_launches(nb > 1 ? 5 : 4);
  return cudaGetLastError();
}

__global__ void split_ec_kernel(const int2* __restrict__ ec, long long nnz, int32_t* col,
                                int32_t* cost) {
  F2M_GRID_STRIDE(e, nnz) {
    const int2 q = ec[e];
    if (col) col[e] = q.x;
    if (cost) cost[e] = q.y;
  }
}

cudaError_t launch_split_ec(const int2* ec, int64_t nnz, int32_t* col, int32_t* cost,
                            cudaStream_t st) {
  if (nnz == 0) return cudaSuccess;
  split_ec_kernel<<<grid_for(nnz, 256), 256, 0, st>>>(ec, nnz, col, cost);
  count_launch();
  return cudaGetLastError();
}

}  // namespace f2m
