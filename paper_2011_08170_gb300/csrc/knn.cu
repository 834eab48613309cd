// Exact k nearest neighbours on a uniform cell grid: the candidate graph of
// Section 5.3 (each node keeps its top-N nearest neighbours) and the features of
// the learned warm start (distances to the 16 nearest neighbours).
//
// Points are bucketed into square cells of side 2^shift (row-major over a 2^g x
// 2^g grid covering [0, 2^20)^2) by a counting sort, so the points of a run of
// cells in one grid row are contiguous.  One thread per point (in cell order, so
// a warp's queries are neighbours) scans a square of cells around its own, keeps
// the k best (d^2, index) in registers, ordered by exact d^2 then index, and
// stops once the k-th kept d^2 is below the squared distance to the nearest cell
// not yet scanned.  The result is the exact k-NN list with ties broken by the
// smaller index, whatever the order of the points inside a cell.
//
// Bound: instruction issue, in the insertions and the set-up of a row's run, which
// a warp repeats for its slowest lane.  So (i) the first square is sized by the
// density around the point (the count of the 5 x 5 cells around it) to hold about
// 2k + 4 points, and where it was too small the k-th distance found says what the
// next one has to cover; (ii) rows are taken from the point outwards, and with a
// full list only the cells within its last distance are read; (iii) an entry is
// one word, d^2 above the index, kept sorted by min and max without branches (where 41
// + the index bits pass 64, points too far for the rest are left out, and where a
// point has fewer than k others nearer, all queries run again with 128 bits: 8.4 M
// uniform points, k = 8, 36 ms with 128 bits, below 3 without).  Rings of cells of 2 points each, with
// 64-bit compares of pairs, took 152 us at 100,000 uniform points, k = 10, and 520
// us at 200,000 clustered ones, k = 16: now 46 and 246,
// the latter with the features of the points.  Not faster: offsets
// and points fetched a step ahead (twice the instructions in the set-up: 435 against
// 296 us), one flat loop over a point's runs (the same), cells along the Z curve
// with a coarser level per point (627: a level is four times too coarse near the
// edge of a cluster).
#include <climits>
#include <cstdint>
#include <vector>

#include <cub/cub.cuh>

#include "ctx_internal.h"
#include "f2m_device.cuh"
#include "f2m_internal.h"

namespace f2m {

namespace {

struct KnnGrid {
  int shift, gbits;
};

__device__ __forceinline__ int knn_cell(int2 p, KnnGrid g) {
  return ((p.y >> g.shift) << g.gbits) | (p.x >> g.shift);
}

// the place of each point in its cell
__global__ void knn_count_kernel(const int2* __restrict__ xy, int32_t n, KnnGrid g, int32_t* __restrict__ count,
                                 int32_t* __restrict__ place) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) place[i] = atomicAdd(count + knn_cell(xy[i], g), 1);
}

// {x, y, index} in cell order
__global__ void knn_place_kernel(const int2* __restrict__ xy, int32_t n, KnnGrid g,
                                 const int32_t* __restrict__ start, const int32_t* __restrict__ place,
                                 int4* __restrict__ pts) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 p = xy[i];
  pts[start[knn_cell(p, g)] + place[i]] = make_int4(p.x, p.y, i, 0);
}

// v = hi + lo with hi the float nearest to it: does a value within 2^-38 of it
// round to another float?
__device__ __forceinline__ bool near_tie(float hi, float lo) {
  const float h = __int_as_float(__float_as_int(hi) & 0x7f800000) * 0x1p-24f;  // half an ulp
  const bool pow2 = (__float_as_int(hi) & 0x007fffff) == 0 && lo < 0.f;         // a quarter below a power of 2
  return fabsf(lo) > (pow2 ? 0.5f * h : h) - h * 0x1p-14f;
}

// feat = sorted 16-NN distances / s, s = max(1, their mean), in 64 bits rounded to
// float.  Computed as pairs of floats (good to 2^-43) unless one of the row's
// values lies within 2^-38 of the middle of two floats, where the 64-bit formula
// decides: the results are the 64-bit ones bit for bit.  The 64-bit square roots
// and quotients had bound a kernel of their own, 121 us at 200,000 points, and 42 in
// pairs of floats; here the list is in registers, and neither it nor its distances
// are written (38 MB) and read again.
__device__ __forceinline__ void write_features(const long long (&d2)[kFeatures], float* __restrict__ feat,
                                               float* __restrict__ scale) {
  float hi[kFeatures], lo[kFeatures], sh = 0.f, sl = 0.f;
#pragma unroll
  for (int j = 0; j < kFeatures; ++j) {
    const long long d = d2[j];
    const float a = (float)d, b = (float)(d - (long long)a);  // d = a + b
    const float y = sqrtf(a);
    // sqrt(d) = y + (d - y^2) / 2y less a term of (d - y^2)^2 / 8y^3
    const float e = d ? (fmaf(-y, y, a) + b) * (0.5f / y) : 0.f;
    hi[j] = y + e;
    lo[j] = e - (hi[j] - y);
    const float t = sh + hi[j], u = t - sh;
    const float c = (sh - (t - u)) + (hi[j] - u) + (sl + lo[j]);
    sh = t + c;
    sl = c - (sh - t);
  }
  sh *= 1.f / kFeatures;
  sl *= 1.f / kFeatures;
  if (sh < 1.f || (sh == 1.f && sl < 0.f)) {
    sh = 1.f;
    sl = 0.f;
  }
  bool tie = near_tie(sh, sl);
  const float inv = 1.f / sh;
#pragma unroll
  for (int j = 0; j < kFeatures; ++j) {
    const float q0 = hi[j] * inv;
    const float q1 = (fmaf(-q0, sh, hi[j]) + fmaf(-q0, sl, lo[j])) * inv;
    hi[j] = q0 + q1;
    lo[j] = q1 - (hi[j] - q0);
    tie |= near_tie(hi[j], lo[j]);
  }
  if (tie) {
    double sum = 0.0;
#pragma unroll
    for (int j = 0; j < kFeatures; ++j) sum += sqrt((double)d2[j]);
    const double s = fmax(1.0, sum / kFeatures);
#pragma unroll
    for (int j = 0; j < kFeatures; ++j) hi[j] = (float)(sqrt((double)d2[j]) / s);
    sh = (float)s;
  }
  // the caller's array may begin at any float
  if ((reinterpret_cast<uintptr_t>(feat) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < kFeatures; j += 4)
      *reinterpret_cast<float4*>(feat + j) = make_float4(hi[j], hi[j + 1], hi[j + 2], hi[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < kFeatures; ++j) feat[j] = hi[j];
  }
  *scale = sh;
}

// FEAT: the features of each point (k = 16) instead of its list.  CUT: entries hold d^2
// below 2^(64 - ibits); *far is set where a list has none for its place k.
template <int K, typename Key, bool FEAT, bool CUT>
__global__ void __launch_bounds__(128)
knn_query_kernel(const int4* __restrict__ pts, const int32_t* __restrict__ start, int32_t n, int32_t k, KnnGrid g,
                 int ibits, int32_t* __restrict__ nbr, long long* __restrict__ d2out, float* __restrict__ feat,
                 float* __restrict__ scale, int32_t* __restrict__ far) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int4 me = pts[t];
  const int x = me.x, y = me.y, gdim = 1 << g.gbits;
  const int cx = x >> g.shift, cy = y >> g.shift;
  const Key none = ~(Key)0;
  Key best[K];
#pragma unroll
  for (int p = 0; p < K; ++p) best[p] = none;
  // points in the 5 x 5 cells around this one
  int near = 0;
#pragma unroll
  for (int d = -2; d <= 2; ++d) {
    const int gy = cy + d;
    if (gy >= 0 && gy < gdim)
      near += start[(gy << g.gbits) + min(cx + 2, gdim - 1) + 1] - start[(gy << g.gbits) + max(cx - 2, 0)];
  }
  // half side of the first square; a thin count says little: start at 8 then
  const float want = (float)(2 * k + 4);
  int r = near < 4 ? 8 : min(64, (int)(2.5f * sqrtf(want / (float)near) + 0.5f));
  int done = -1;  // half side of the square scanned so far
  for (;;) {
    const int xa = max(cx - r, 0), xb = min(cx + r, gdim - 1);
    // rows cy, cy - 1, cy + 1, cy - 2, ...; in a row that the scanned square crosses
    // the parts left and right of it
    for (int step = 0; step <= 2 * r; ++step) {
      const int gy = (step & 1) ? cy - (step + 1) / 2 : cy + step / 2;
      if (gy < 0 || gy >= gdim) continue;
      int fa = xa, fb = xb;
      // with a full list only what lies within its last distance
      const Key last = best[K - 1];
      if (last != none) {
        const int dy = gy == cy ? 0 : gy < cy ? y - ((gy + 1) << g.shift) + 1 : (gy << g.shift) - y;
        const long long rest = (long long)(last >> ibits) - (long long)dy * dy;
        if (rest < 0) continue;
        const int h = (int)(sqrtf((float)rest) * 1.000001f) + 1;
        fa = max(fa, (x - h) >> g.shift);
        fb = min(fb, (x + h) >> g.shift);
      }
      const bool crossed = gy >= cy - done && gy <= cy + done;
      for (int part = 0; part < (crossed ? 2 : 1); ++part) {
        const int ga = part ? max(fa, cx + done + 1) : fa, gb = crossed && !part ? min(fb, cx - done - 1) : fb;
        if (ga > gb) continue;
        const int b = start[(gy << g.gbits) + gb + 1];
        for (int a = start[(gy << g.gbits) + ga]; a < b; ++a) {
          const int4 q = pts[a];
          const int dx = q.x - x, dy = q.y - y;
          const unsigned long long dd = (unsigned long long)((long long)dx * dx + (long long)dy * dy);
          if (CUT && dd >> (64 - ibits)) continue;
          Key key = ((Key)dd << ibits) | (Key)(unsigned)q.z;
          if (a != t && key < best[K - 1]) {
#pragma unroll
            for (int p = 0; p < K; ++p) {
              const Key lo = key < best[p] ? key : best[p];
              key = key < best[p] ? best[p] : key;
              best[p] = lo;
            }
          }
        }
      }
    }
    done = r;
    // smallest distance from (x, y) to a cell outside the scanned square
    const int x0 = cx - r, x1 = cx + r, y0 = cy - r, y1 = cy + r;
    long long bnd = LLONG_MAX;
    if (x0 > 0) bnd = min(bnd, (long long)x - ((long long)x0 << g.shift) + 1);
    if (y0 > 0) bnd = min(bnd, (long long)y - ((long long)y0 << g.shift) + 1);
    if (x1 < gdim - 1) bnd = min(bnd, ((long long)(x1 + 1) << g.shift) - x);
    if (y1 < gdim - 1) bnd = min(bnd, ((long long)(y1 + 1) << g.shift) - y);
    if (bnd == LLONG_MAX) break;  // the whole grid has been scanned
    Key kth = best[K - 1];
#pragma unroll
    for (int p = 0; p < K - 1; ++p) kth = p == k - 1 ? best[p] : kth;
    if (kth == none) {
      if (CUT && (unsigned long long)(bnd * bnd) >> (64 - ibits)) break;  // the others are too far
      r = 2 * r + 1;
      continue;
    }
    const long long d2 = (long long)(kth >> ibits);
    if (d2 < bnd * bnd) break;
    // a square of this half side covers the k-th distance (checked again after it)
    r = max(r + 1, (int)(sqrtf((float)d2) * 1.000001f / (float)(1 << g.shift)) + 1);
  }
  if (CUT) {
    Key kth = best[K - 1];
#pragma unroll
    for (int p = 0; p < K - 1; ++p) kth = p == k - 1 ? best[p] : kth;
    if (kth == none) *far = 1;
  }
  if (FEAT) {
    long long d2[kFeatures];
#pragma unroll
    for (int p = 0; p < kFeatures; ++p) d2[p] = (long long)(best[p < K ? p : 0] >> ibits);
    write_features(d2, feat + (size_t)me.z * kFeatures, scale + me.z);
    return;
  }
  const unsigned long long imask = (1ull << ibits) - 1;
#pragma unroll
  for (int p = 0; p < K; ++p) {
    if (p < k) {
      nbr[(size_t)me.z * k + p] = (int32_t)((unsigned long long)best[p] & imask);
      if (d2out) d2out[(size_t)me.z * k + p] = (long long)(best[p] >> ibits);
    }
  }
}

// ---- symmetrised CSR ----------------------------------------------------------------
//
// Row u holds u's own k neighbours and the nodes that list u without being listed
// by it.  Three passes and a scan instead of a sort of all 2nk pairs (280 us of
// radix passes, duplicates and searches at 100,000 points and k = 10): now 52 us.

constexpr int kKnnHub = 1024;  // longest row that is ordered by counting; longer ones: by sorting all pairs

__global__ void knn_fill_kernel(int32_t* p, int32_t n, int32_t v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// slot[e] of entry e = (u -> w): its place in row w, or -1 where w lists u itself.
// deg starts at k.
__global__ void knn_slot_kernel(const int32_t* __restrict__ nbr, int32_t n, int32_t k, int32_t* __restrict__ deg,
                                int32_t* __restrict__ slot, int32_t* __restrict__ hub) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= (long long)n * k) return;
  const int u = (int)(e / k), w = nbr[e];
  const int32_t* row = nbr + (size_t)w * k;
  bool both = false;
  for (int p = 0; p < k; ++p) both |= row[p] == u;
  int s = -1;
  if (!both) {
    s = atomicAdd(deg + w, 1);
    if (s >= kKnnHub) *hub = 1;
  }
  slot[e] = s;
}

__global__ void knn_extra_kernel(const int32_t* __restrict__ nbr, const int32_t* __restrict__ slot,
                                 const int32_t* __restrict__ row_ptr, int32_t n, int32_t k,
                                 int32_t* __restrict__ extra) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= (long long)n * k) return;
  const int s = slot[e];
  if (s >= 0) extra[row_ptr[nbr[e]] + s] = (int)(e / k);
}

// each entry goes to the number of smaller ones in its row (they are distinct)
__global__ void knn_order_kernel(const int32_t* __restrict__ nbr, const int32_t* __restrict__ extra,
                                 const int32_t* __restrict__ row_ptr, int32_t n, int32_t k,
                                 int32_t* __restrict__ col, int32_t* __restrict__ nnz) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *nnz = row_ptr[n];
  F2M_ROWS(u, sub, n) {
    const int a = row_ptr[u], m = row_ptr[u + 1] - a;
    if (m > kKnnHub) continue;
    const int32_t* own = nbr + (size_t)u * k;
    for (int i = sub; i < m; i += kRowLanes) {
      const int c = i < k ? own[i] : extra[a + i];
      int before = 0;
      for (int j = 0; j < k; ++j) before += own[j] < c;
      for (int j = k; j < m; ++j) before += extra[a + j] < c;
      col[a + before] = c;
    }
  }
}

// the same CSR by sorting: both directions of every k-NN entry as keys (u << 32 | w)
__global__ void knn_pair_keys_kernel(const int32_t* __restrict__ nbr, int32_t n, int32_t k,
                                     uint64_t* __restrict__ keys) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long m = (long long)n * k;
  if (e >= m) return;
  const uint64_t u = (uint64_t)(e / k), w = (uint64_t)(uint32_t)nbr[e];
  keys[2 * e] = (u << 32) | w;
  keys[2 * e + 1] = (w << 32) | u;
}

__global__ void knn_csr_cols_kernel(const uint64_t* __restrict__ ukeys, int nnz, int32_t* __restrict__ col) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e < nnz) col[e] = (int32_t)(uint32_t)(ukeys[e] & 0xffffffffu);
}

inline unsigned blocks_for(long long items, int threads) {
  return (unsigned)((items + threads - 1) / threads);
}

// the device blocks of one call: back to the cache at its end, after a wait for
// the device unless the call has waited for its stream
struct KnnScope {
  std::vector<void*> blocks;
  bool synced = false;
  template <typename T>
  cudaError_t get(T** p, int64_t count) {
    const cudaError_t e = dalloc(p, count);
    if (e == cudaSuccess) blocks.push_back(*p);
    return e;
  }
  ~KnnScope() {
    for (void* p : blocks)
      if (synced) dev_free_synced(p); else dev_free(p);
  }
};

// grid: the smallest g with 4^g >= n, up to 2^22 cells (a quarter of a point to one
// a cell when the points fill the square).  Four times as many cells cost uniform
// points 20 % in rows, a quarter as many cost clusters 50 % in points.
KnnGrid knn_grid(int32_t n) {
  int g = 1;
  while (g < 11 && (1LL << (2 * g)) < n) ++g;
  return KnnGrid{20 - g, g};
}

template <int K, typename Key, bool FEAT = false, bool CUT = false>
void knn_query(const int4* pts, const int32_t* start, int32_t n, int32_t k, KnnGrid g, int ibits, int32_t* nbr,
               long long* d2, float* feat, float* scale, int32_t* far, cudaStream_t st) {
  knn_query_kernel<K, Key, FEAT, CUT><<<blocks_for(n, 128), 128, 0, st>>>(pts, start, n, k, g, ibits, nbr, d2, feat,
                                                                         scale, far);
  count_launch();
}

cudaError_t knn_enqueue(KnnScope& w, const int2* d_xy, int32_t n, int32_t k, int32_t* d_nbr, long long* d_d2,
                        float* feat, float* scale, cudaStream_t st) {
  if (k < 1 || k > kKnnMax || n <= k) return cudaErrorInvalidValue;
  const KnnGrid g = knn_grid(n);
  const int ncell = 1 << (2 * g.gbits);
  int ibits = 1;
  while ((1LL << ibits) < n) ++ibits;
  int32_t *count = nullptr, *start = nullptr, *place = nullptr, *scan = nullptr;
  int4* pts = nullptr;
  cudaError_t e = w.get(&count, ncell);
  if (e == cudaSuccess) e = w.get(&start, (int64_t)ncell + 1);
  if (e == cudaSuccess) e = w.get(&place, n);
  if (e == cudaSuccess) e = w.get(&scan, (int64_t)scan_scratch_ints(ncell));
  if (e == cudaSuccess) e = w.get(&pts, n);
  if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof(int32_t) * ncell, st);
  if (e != cudaSuccess) return e;
  knn_count_kernel<<<blocks_for(n, 256), 256, 0, st>>>(d_xy, n, g, count, place);
  count_launch();
  e = launch_scan(count, start, ncell, scan, st);
  if (e != cudaSuccess) return e;
  knn_place_kernel<<<blocks_for(n, 256), 256, 0, st>>>(d_xy, n, g, start, place, pts);
  count_launch();
  using u64 = unsigned long long;
  using u128 = unsigned __int128;
  const bool wide = ibits > 64 - 41;  // d^2 < 2^41
  int32_t* far = nullptr;
#define F2M_KNN(...) knn_query<__VA_ARGS__>(pts, start, n, k, g, ibits, d_nbr, d_d2, feat, scale, far, st)
  if (wide) {
    e = w.get(&far, 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(far, 0, sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
    if (feat) F2M_KNN(kFeatures, u64, true, true);
    else if (k <= 8) F2M_KNN(8, u64, false, true);
    else if (k <= 16) F2M_KNN(16, u64, false, true);
    else F2M_KNN(32, u64, false, true);
    e = cudaGetLastError();
    int32_t h = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, far, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || !h) return e;
    if (feat) F2M_KNN(kFeatures, u128, true);
    else F2M_KNN(32, u128);
  } else if (feat) F2M_KNN(kFeatures, u64, true);
  else if (k <= 8) F2M_KNN(8, u64);
  else if (k <= 10) F2M_KNN(10, u64);
  else if (k <= 12) F2M_KNN(12, u64);
  else if (k <= 16) F2M_KNN(16, u64);
  else F2M_KNN(32, u64);
#undef F2M_KNN
  return cudaGetLastError();
}

}  // namespace

cudaError_t knn_device(const int2* d_xy, int32_t n, int32_t k, int32_t* d_nbr, long long* d_d2,
                       cudaStream_t st) {
  KnnScope w;
  cudaError_t e = knn_enqueue(w, d_xy, n, k, d_nbr, d_d2, nullptr, nullptr, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  w.synced = e == cudaSuccess;
  return e;
}

cudaError_t knn_csr_device(const int2* d_xy, int32_t n, int32_t k, int32_t* d_row_ptr, int32_t* d_col,
                           int64_t* nnz_out, cudaStream_t st) {
  const long long m = 2LL * n * k, half = (long long)n * k;
  if (m >= INT_MAX) return cudaErrorInvalidValue;
  KnnScope w;
  int32_t *nbr = nullptr, *slot = nullptr, *extra = nullptr, *deg = nullptr, *scan = nullptr, *ctl = nullptr;
  cudaError_t e = w.get(&nbr, half);
  if (e == cudaSuccess) e = w.get(&slot, half);
  if (e == cudaSuccess) e = w.get(&extra, m);
  if (e == cudaSuccess) e = w.get(&deg, n);
  if (e == cudaSuccess) e = w.get(&scan, (int64_t)scan_scratch_ints(n));
  if (e == cudaSuccess) e = w.get(&ctl, 2);  // {entries, a row is longer than kKnnHub}
  if (e == cudaSuccess) e = cudaMemsetAsync(ctl, 0, 2 * sizeof(int32_t), st);
  if (e == cudaSuccess) e = knn_enqueue(w, d_xy, n, k, nbr, nullptr, nullptr, nullptr, st);
  if (e != cudaSuccess) return e;
  knn_fill_kernel<<<blocks_for(n, 256), 256, 0, st>>>(deg, n, k);
  knn_slot_kernel<<<blocks_for(half, 256), 256, 0, st>>>(nbr, n, k, deg, slot, ctl + 1);
  count_launches(2);
  e = launch_scan(deg, d_row_ptr, n, scan, st);
  if (e != cudaSuccess) return e;
  knn_extra_kernel<<<blocks_for(half, 256), 256, 0, st>>>(nbr, slot, d_row_ptr, n, k, extra);
  const long long ob = ((long long)n * kRowLanes + 255) / 256;
  knn_order_kernel<<<(unsigned)(ob < 16384 ? ob : 16384), 256, 0, st>>>(nbr, extra, d_row_ptr, n, k, d_col, ctl);
  count_launches(2);
  e = cudaGetLastError();
  int32_t h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, ctl, sizeof h, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  *nnz_out = h[0];
  if (h[1]) {  // the row offsets stand; the columns in order
    uint64_t *keys = nullptr, *skeys = nullptr;
    int* d_nnz = nullptr;
    void* tmp = nullptr;
    size_t sort_bytes = 0, uniq_bytes = 0;
    e = cub::DeviceRadixSort::SortKeys(nullptr, sort_bytes, (const uint64_t*)nullptr, (uint64_t*)nullptr, (int)m, 0,
                                       64, st);
    if (e == cudaSuccess)
      e = cub::DeviceSelect::Unique(nullptr, uniq_bytes, (const uint64_t*)nullptr, (uint64_t*)nullptr, (int*)nullptr,
                                    (int)m, st);
    size_t tmp_bytes = sort_bytes > uniq_bytes ? sort_bytes : uniq_bytes;
    if (e == cudaSuccess) e = w.get(&keys, m);
    if (e == cudaSuccess) e = w.get(&skeys, m);
    if (e == cudaSuccess) e = w.get(&d_nnz, 1);
    if (e == cudaSuccess) e = w.get((char**)&tmp, (int64_t)tmp_bytes);
    if (e != cudaSuccess) return e;
    knn_pair_keys_kernel<<<blocks_for(half, 256), 256, 0, st>>>(nbr, n, k, keys);
    count_launch();
    size_t b = tmp_bytes;
    e = cub::DeviceRadixSort::SortKeys(tmp, b, keys, skeys, (int)m, 0, 64, st);
    b = tmp_bytes;
    if (e == cudaSuccess) e = cub::DeviceSelect::Unique(tmp, b, skeys, keys, d_nnz, (int)m, st);
    if (e != cudaSuccess) return e;
    knn_csr_cols_kernel<<<blocks_for(h[0], 256), 256, 0, st>>>(keys, h[0], d_col);
    count_launch();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  w.synced = e == cudaSuccess;
  return e;
}

cudaError_t features_device(const int2* d_xy, int32_t n, float* d_feat, float* d_scale,
                            cudaStream_t st) {
  KnnScope w;
  cudaError_t e = knn_enqueue(w, d_xy, n, kFeatures, nullptr, nullptr, d_feat, d_scale, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  w.synced = e == cudaSuccess;
  return e;
}

}  // namespace f2m
