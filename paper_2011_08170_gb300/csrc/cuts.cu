// Subtour-elimination cuts: GDP over node and cut duals.
//
// The paper's Discussion names the F2M LP plus subtour elimination constraints
// as the next relaxation for the method.  The LP:
//   minimise c x  subject to  x(delta(v)) = 2 for every node v      (Section 4)
//                             x(delta(S)) >= 2 for every cut S of a family
//                             0 <= x <= 1,
// Section 2's LP3 with equalities (1) and inequalities (2).  Every constraint
// has binary coefficients and right side 2 (Eq. 8), so Section 3's gradient
// applies to each: the 2nd and 3rd smallest modified values over its support.
// Inequality duals stay >= 0 (Eq. 5).  The modified objective (Eq. 4) of an
// edge uv is
//   z_uv = c_uv 2^F - lambda_u - lambda_v - sum of mu_S over the cuts S that
//          hold exactly one of u, v.
// One Jacobi sweep (Section 5.1's parallel update, extended to the cut duals)
// reads only the previous lambda and mu:
//   lambda_v += trunc((z(2) + z(3)) / 2^shift) over delta(v),
//   mu_S = max(0, mu_S + trunc((z(2) + z(3)) / 2^(shift + 2))) over delta(S),
// the cut step a quarter of the node step: an edge's z moves with both end
// duals and with up to two cut duals per layer at once, and nested cuts of
// different layers move nearly the same edges (a full node-sized step made
// the duals diverge after a few layers);
//   bound2 = 4 sum lambda + 4 sum mu + sum over directed entries of min(0, z).
//
// Cut family: up to kMaxCutLayers layers; layer l labels every node with -1
// (no cut of the layer) or a cut index s in [0, ncuts_l); the nodes labelled s
// form the cut set.  Cuts of one layer are disjoint.  Separation makes one
// layer from the connected components of the support of x.
//
// Device layout.  Caller order: comp [L][n] int32 labels, mask [nnz] uint8 (bit
// l: the entry's two ends differ in layer l's label) for the bound, rule (7) and
// pricing.  Renumbered order, for the GDP kernel: cid [L][n] the cut that holds
// a node (or -1), the mask again, cut lists cut_ptr [M+1] / items ({entry, row} of
// the entries whose row lies in the cut and whose column does not: each crossing
// edge once per cut); mu [2][M] (Jacobi double buffer).
//
// Kernel: one persistent cooperative launch per phase, one block per SM, one
// device-wide barrier a sweep.  A block takes an equal share of the rows (4 lanes
// each) and the cuts whose lists begin in its share of all lists (a warp each, the
// whole block for a list above 1,024 entries), and computes z for both from
// tables it builds once per phase in shared memory: its entries, and the distinct
// nodes and cuts that they read (one bit each, the rank of a bit is its place),
// whose lambda and mu it fetches once a sweep.  A block whose tables do not fit
// reads global memory through L1 instead.
//
// Bound, at 20,000 points with 10 neighbours and two layers (sweep of 6.8 us):
// issue and shared-memory latency of the 57 row groups and cuts of a block (3.5
// us), the fetch of some 1,200 values (1 us), the barrier and the slack of the
// fullest block (2.3 us).  With one gather per entry, end and crossed cut from L2
// (two million a sweep, all past L1) the same sweep took 19 to 24 us; through L1
// with no tables 8 to 11 us.  Per sweep before and now with one layer: 3,000 points
// 16.6 and 5.4 us, 40,000 points 30 and 9.7, 100,000 points (no tables) 41 and 30.
// z is kept in 32 bits in a sweep whose values allow it (checked with the fetch),
// else in 64: the 64-bit compares had been half of the instructions.  768 threads:
// 512 take 10 % longer, and with 1,024 the 64 registers a thread spill (9 us).
#include <algorithm>
#include <chrono>
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/f2m.h"
#include "ctx_internal.h"
#include "f2m_device.cuh"
#include "f2m_internal.h"

namespace f2m {

struct CutArgs {
  const int32_t* comp;  // [L][n]
  int32_t n, L;
  int32_t off[kMaxCutLayers + 1];  // first cut index of each layer
};

struct CutState {
  int32_t L = 0;
  std::vector<int32_t> ncuts;  // per layer
  std::vector<int32_t> off;    // [L + 1]
  int64_t M = 0;               // cuts in all layers
  int32_t* d_comp = nullptr;   // [kMaxCutLayers][n]
  int32_t* d_mu[2] = {nullptr, nullptr};
  int64_t mu_cap = 0;
  int cur = 0;                 // d_mu[cur] holds mu
  uint8_t* d_mask = nullptr;
  int64_t mask_cap = 0;
  int32_t* d_cnt = nullptr;    // per cut: count, then fill cursor
  int32_t* d_ptr = nullptr;    // [M + 1]
  int32_t* d_scan = nullptr;   // scan scratch
  int64_t ptr_cap = 0;
  int2* d_items = nullptr;     // {entry, row}, renumbered order
  int64_t item_cap = 0;
  int32_t* d_cid = nullptr;    // [L][n] renumbered order
  int64_t cid_cap = 0;
  uint8_t* d_imask = nullptr;  // [nnz] mask in the renumbered order
  int64_t imask_cap = 0;
  int64_t built_version = -1;  // graph version the mask and lists were built for
  int32_t built_L = -1;
  // separation and pricing scratch
  int32_t* d_lab = nullptr;    // [n] component label (smallest node)
  int32_t* d_cross = nullptr;  // [n] crossing entries per root
  int32_t* d_flag = nullptr;   // [n + 1] flags, then ranks
  int32_t* d_rank = nullptr;   // [n + 1]
  int32_t* d_small = nullptr;  // [4] small device counters
  int32_t* d_lamp = nullptr;   // [n] lambda + the duals of the cuts holding the node
  int32_t* d_keep = nullptr;   // [pair_cap + 1]
  int32_t* d_kpos = nullptr;   // [pair_cap + 1]
  int2* d_pairs2 = nullptr;
  int64_t pair_cap = 0;
  int32_t* d_pscan = nullptr;
  int64_t pscan_cap = 0;
};

void cut_state_free(CutState* s) {
  if (!s) return;
  dfree(s->d_comp); dfree(s->d_mu[0]); dfree(s->d_mu[1]); dfree(s->d_mask); dfree(s->d_cnt);
  dfree(s->d_ptr); dfree(s->d_scan); dfree(s->d_items); dfree(s->d_lab); dfree(s->d_cross);
  dfree(s->d_flag); dfree(s->d_rank); dfree(s->d_small); dfree(s->d_lamp); dfree(s->d_keep);
  dfree(s->d_kpos); dfree(s->d_pairs2); dfree(s->d_pscan); dfree(s->d_cid); dfree(s->d_imask);
  delete s;
}

int64_t cut_count(const f2m_ctx* c) { return c->cuts ? c->cuts->M : 0; }

namespace {

constexpr long long kInfZ = LLONG_MAX / 4;
constexpr int kLongCut = 1024;  // crossing entries above which a block's cut warps take a cut together

__device__ __forceinline__ void top3_ins_ll(long long z, long long& a, long long& b, long long& c) {
  if (z < c) {
    if (z < b) {
      c = b;
      if (z < a) { b = a; a = z; } else { b = z; }
    } else {
      c = z;
    }
  }
}

__device__ __forceinline__ long long step_ll(long long z2, long long z3, int shift) {
  const long long s = z2 + z3;
  return s >= 0 ? (s >> shift) : -((-s) >> shift);  // truncation toward zero
}

__device__ __forceinline__ long long ld_cg_i(const int32_t* p) { return (long long)__ldcg(p); }

// sum of the duals of the cuts that entry (u, v) crosses; bit l of m set when
// the ends differ in layer l's label
__device__ __forceinline__ long long cut_term(const CutArgs& a, const int32_t* mu, unsigned m, int u, int v) {
  long long t = 0;
  for (int l = 0; l < a.L; ++l) {
    if (!((m >> l) & 1u)) continue;
    const int cu = __ldg(a.comp + (long long)l * a.n + u), cv = __ldg(a.comp + (long long)l * a.n + v);
    if (cu >= 0) t += ld_cg_i(mu + a.off[l] + cu);
    if (cv >= 0) t += ld_cg_i(mu + a.off[l] + cv);
  }
  return t;
}

__device__ __forceinline__ long long entry_z(const CutArgs& a, const int32_t* lam, const int32_t* mu,
                                             unsigned m, int u, int2 q, int F) {
  long long z = ((long long)q.y << F) - ld_cg_i(lam + u) - ld_cg_i(lam + q.x);
  if (m) z -= cut_term(a, mu, m, u, q.x);
  return z;
}

// mask[e] for every directed entry
__global__ void cut_mask_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec, CutArgs a,
                                uint8_t* __restrict__ mask) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < a.n;
       v += (long long)gridDim.x * blockDim.x) {
    for (int e = rp[v]; e < rp[v + 1]; ++e) {
      const int w = ec[e].x;
      unsigned m = 0;
      for (int l = 0; l < a.L; ++l)
        if (a.comp[(long long)l * a.n + v] != a.comp[(long long)l * a.n + w]) m |= 1u << l;
      mask[e] = (uint8_t)m;
    }
  }
}

// cid[l][i] = the cut of layer l that holds internal node i, or -1
__global__ void cut_cid_kernel(CutArgs a, const int32_t* __restrict__ perm, int32_t* __restrict__ cid) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.n;
       i += (long long)gridDim.x * blockDim.x)
    for (int l = 0; l < a.L; ++l) {
      const int s = a.comp[(long long)l * a.n + perm[i]];
      cid[(long long)l * a.n + i] = s >= 0 ? a.off[l] + s : -1;
    }
}

// per cut: crossing entries whose row lies in the cut (counts, with the entries'
// masks, or the list filled at the cursors)
template <bool FILL>
__global__ void cut_list_kernel(const int32_t* __restrict__ irp, const int2* __restrict__ iec,
                                const int32_t* __restrict__ cid, int32_t n, int32_t L, uint8_t* __restrict__ mask,
                                int32_t* cnt, const int32_t* __restrict__ ptr, int2* items) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    for (int e = irp[v]; e < irp[v + 1]; ++e) {
      unsigned m = 0;
      if (FILL) {
        m = mask[e];
      } else {
        const int w = iec[e].x;
        for (int l = 0; l < L; ++l)
          if (cid[(long long)l * n + v] != cid[(long long)l * n + w]) m |= 1u << l;
        mask[e] = (uint8_t)m;
      }
      for (; m; m &= m - 1) {
        const int id = cid[(long long)(__ffs(m) - 1) * n + v];
        if (id < 0) continue;
        const int k = atomicAdd(cnt + id, 1);
        if (FILL) items[ptr[id] + k] = make_int2(e, (int)v);
      }
    }
  }
}

// labels of layer l in [-1, ncuts): else flag
__global__ void cut_label_check_kernel(const int32_t* __restrict__ comp, int32_t n, int32_t ncuts,
                                       int32_t* flag) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const int s = comp[v];
    if (s < -1 || s >= ncuts) atomicMin(flag, (int)v);
  }
}

// cuts with fewer than 3 crossing edges: smallest such cut index into flag
__global__ void cut_short_kernel(const int32_t* __restrict__ cnt, int32_t M, int32_t* flag) {
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < M;
       s += (long long)gridDim.x * blockDim.x)
    if (cnt[s] < 3) atomicMin(flag, (int)s);
}

struct CutGdp {
  const int32_t* irp;
  const int2* iec;
  const int32_t* perm;
  const int32_t* cid;
  const uint8_t* mask;
  const int32_t* cut_ptr;
  const int2* items;
  const int32_t* lam_in;   // caller order
  int32_t* lam_out;
  int32_t* lam[2];         // renumbered
  int32_t* mu[2];
  GdpCtl* ctl;
  long long* trace_b2;
  unsigned long long* trace_ch;
  long long trace_cap, max_sweeps, budget;
  int32_t n, L, M, F, shift;
};

constexpr int kCutThreads = 768;
constexpr int kCutGroup = 4;        // lanes of a row
constexpr int kCutSmem = 208 << 10; // a block's tables

template <typename Z>
__device__ __forceinline__ void cut_top3(Z z, Z& a, Z& b, Z& c) {  // no branches: the lanes of a warp disagree
  c = min(c, max(b, z));
  b = min(b, max(a, z));
  a = min(a, z);
}

// top-3 of the lanes of an aligned group of W
template <int W, typename Z>
__device__ __forceinline__ void cut_top3_group(unsigned gmask, Z& a, Z& b, Z& c) {
#pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const Z a1 = __shfl_xor_sync(gmask, a, o), b1 = __shfl_xor_sync(gmask, b, o), c1 = __shfl_xor_sync(gmask, c, o);
    // the third of the union: see top3_join
    const Z m = max(a, a1), q = min(b, b1);
    a = min(a, a1);
    c = min(max(m, q), min(c, c1));
    b = min(m, q);
  }
}

// Entries k, k + step, ... below end of a row or (not ROW) a cut into the top-3 and
// b2, from the tables in shared memory: tab {u, v, cost, 16 * (first pair) +
// pairs}, nodes by their place in val (the sweep's lambdas and mus), a pair {cut
// of u, cut of v} for each layer in which the ends differ; val[zero] is 0.
template <bool ROW, typename Z>
__device__ __forceinline__ void cut_scan_in(const CutGdp& A, const int4* tab, const int2* pairs, const int* val,
                                            int k, int end, int step, int lu, Z& a, Z& b, Z& c,
                                            long long& b2) {
#pragma unroll 2
  for (; k < end; k += step) {
    const int4 it = tab[k];
    Z z = (Z)it.z * (Z)(1 << A.F) - (Z)val[it.y] - (Z)(ROW ? lu : val[it.x]);
    const int2* q = pairs + ((unsigned)it.w >> 4);
    const int np = it.w & 15;
    for (int l = 0; l < np; ++l) z -= (Z)(val[q[l].x] + val[q[l].y]);  // two duals, each below 2^29
    if (ROW && z < 0) b2 += z;
    cut_top3(z, a, b, c);
  }
}

// The same from global memory.  Four at a time with every load unconditional (a
// dual that is not there reads cut 0 and counts as 0): loads inside branches wait
// for one another.  lambda and mu come through L1, which the acquire of the
// sweep's barrier has emptied of the sweep before: a block reads the same few
// nodes many times, and with every gather from L2 its rate bound the sweep.
template <bool ROW>
__device__ __forceinline__ void cut_scan_out(const CutGdp& A, int u, int k, int end, int step, const int32_t* lam,
                                             const int32_t* mu, long long lu, long long& a, long long& b, long long& c,
                                             long long& b2) {
  constexpr int U = 4;
  for (; k < end; k += U * step) {
    int4 it[U];
    long long z[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int e = k + j * step;
      it[j] = make_int4(0, 0, 0, 0);
      if (e >= end) continue;
      const int2 w = ROW ? make_int2(e, u) : __ldg(A.items + e);
      const int2 q = __ldg(A.iec + w.x);
      it[j] = make_int4(w.y, q.x, q.y, __ldg(A.mask + w.x));
    }
#pragma unroll
    for (int j = 0; j < U; ++j)
      z[j] = ((long long)it[j].z << A.F) - lam[it[j].y] - (ROW ? lu : (long long)lam[it[j].x]);
    for (int l = 0; l < A.L; ++l) {
      const int32_t* row = A.cid + (long long)l * A.n;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        int x = -1, y = -1;
        if ((unsigned)it[j].w >> l & 1u) {
          x = __ldg(row + it[j].x);
          y = __ldg(row + it[j].y);
        }
        const int mx = mu[max(x, 0)], my = mu[max(y, 0)];
        z[j] -= (x >= 0 ? mx : 0) + (y >= 0 ? my : 0);
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (k + j * step >= end) z[j] = kInfZ;
      if (ROW && z[j] < 0) b2 += z[j];
      cut_top3(z[j], a, b, c);
    }
  }
}

// exclusive sum of v over the block's threads; the total in *total
__device__ __forceinline__ int cut_block_scan(int v, int* total) {
  __shared__ int s_w[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  int before = 0, all = 0;
  for (int w = 0; w < (int)blockDim.x / 32; ++w) {
    if (w < warp) before += s_w[w];
    all += s_w[w];
  }
  *total = all;
  return before + x - v;
}

__global__ void __launch_bounds__(kCutThreads, 1) cut_gdp_kernel(const __grid_constant__ CutGdp A) {
  constexpr int G = kCutGroup, RW = 32 / G, NW = kCutThreads / 32;
  extern __shared__ int4 s_dyn[];
  __shared__ long long s_t3[NW * 3];
  __shared__ unsigned s_ch, s_pairs;
  __shared__ int s_ovf, s_stop, s_cut[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = lane & (G - 1);
  const unsigned gmask = ((1u << G) - 1u) << (lane & ~(G - 1));
  const int n = A.n, L = A.L, M = A.M, nb = gridDim.x, blk = blockIdx.x;
  const int v0 = (int)((long long)n * blk / nb), v1 = (int)((long long)n * (blk + 1) / nb), nr = v1 - v0;
  for (int i = v0 + tid; i < v1; i += kCutThreads) A.lam[0][i] = A.lam_in[__ldg(A.perm + i)];
  // the block's cuts: those whose list begins in its share of all lists
  if (tid < 2) {
    const long long T = __ldg(A.cut_ptr + M);
    int lo = 0, hi = M;
    if (blk + tid == nb) lo = M;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((long long)__ldg(A.cut_ptr + mid) * nb >= T * (blk + tid)) hi = mid; else lo = mid + 1;
    }
    s_cut[tid] = lo;
  }
  if (tid == 0) { s_ch = 0; s_ovf = 0; s_pairs = 0; }
  __syncthreads();
  const int s0 = s_cut[0], nc = s_cut[1] - s0;
  const int e0 = __ldg(A.irp + v0), ne = __ldg(A.irp + v1) - e0;
  const int k0 = __ldg(A.cut_ptr + s0), nk = __ldg(A.cut_ptr + s0 + nc) - k0;
  // Tables of the block in shared memory: the offsets of its rows and cuts, the
  // entries of both, the nodes and cuts they read (found with one bit each; a
  // place is the rank of the bit) with their values, and the pairs.  One that
  // does not fit leaves the block on global memory.
  const int wn = (n + 31) / 32, nw = wn + (M + 31) / 32;  // words: nodes, then cuts
  const int offs = (nr + 1 + nc + 1 + 3) & ~3;
  const long long fixed = 16LL * ne + 16LL * nk + 4LL * offs + 8LL * nw;
  bool in = fixed + 16 <= kCutSmem;
  int4* rtab = s_dyn;
  int4* ktab = rtab + (in ? ne : 0);
  int32_t* s_rp = reinterpret_cast<int32_t*>(ktab + (in ? nk : 0));
  int32_t* s_cp = s_rp + nr + 1;
  unsigned* bits = reinterpret_cast<unsigned*>(s_rp + (in ? offs : 0));
  int32_t* rank = reinterpret_cast<int32_t*>(bits + (in ? nw : 0));
  int32_t* need = rank + (in ? nw : 0);  // bit of each place, its value behind
  int32_t* val = need;
  int2* pairs = nullptr;
  int nneed = 0;
  auto entry = [&](auto&& f) {  // f(place in the tables, entry, row)
    for (int i = tid / G; i < nr; i += kCutThreads / G)
      for (int e = __ldg(A.irp + v0 + i) + sub, end = __ldg(A.irp + v0 + i + 1); e < end; e += G) f(e - e0, e, v0 + i);
    for (int k = tid; k < nk; k += kCutThreads) {
      const int2 w = __ldg(A.items + k0 + k);
      f(ne + k, w.x, w.y);
    }
  };
  auto mark = [&](int b) { atomicOr(bits + (b >> 5), 1u << (b & 31)); };
  auto place = [&](int b) { return rank[b >> 5] + __popc(bits[b >> 5] & ((1u << (b & 31)) - 1u)); };
  if (in) {
    for (int i = tid; i < nw; i += kCutThreads) bits[i] = 0;
    for (int i = tid; i <= nr; i += kCutThreads) s_rp[i] = __ldg(A.irp + v0 + i) - e0;
    for (int i = tid; i <= nc; i += kCutThreads) s_cp[i] = __ldg(A.cut_ptr + s0 + i) - k0;
    __syncthreads();
    for (int i = v0 + tid; i < v1; i += kCutThreads) mark(i);
    for (int i = s0 + tid; i < s0 + nc; i += kCutThreads) mark(wn * 32 + i);
    entry([&](int, int e, int u) {
      const int v = __ldg(A.iec + e).x;
      unsigned m = __ldg(A.mask + e);
      mark(u);
      mark(v);
      if (m) atomicAdd(&s_pairs, __popc(m));
      for (; m; m &= m - 1) {
        const int32_t* row = A.cid + (long long)(__ffs(m) - 1) * n;
        const int x = __ldg(row + u), y = __ldg(row + v);
        if (x >= 0) mark(wn * 32 + x);
        if (y >= 0) mark(wn * 32 + y);
      }
    });
    __syncthreads();
    const int per = (nw + kCutThreads - 1) / kCutThreads, w0 = min(nw, tid * per), w1 = min(nw, w0 + per);
    int mine = 0;
    for (int w = w0; w < w1; ++w) mine += __popc(bits[w]);
    int r = cut_block_scan(mine, &nneed);
    const long long npairs = s_pairs;
    in = fixed + 8LL * (nneed + 2) + 8LL * npairs + 16 <= kCutSmem;
    if (in) {
      val = need + nneed + 1;
      pairs = reinterpret_cast<int2*>(need + ((2 * nneed + 3) & ~1));
      pairs = reinterpret_cast<int2*>((reinterpret_cast<uintptr_t>(pairs) + 7) & ~(uintptr_t)7);
      for (int w = w0; w < w1; ++w) {
        rank[w] = r;
        for (unsigned m = bits[w]; m; m &= m - 1) need[r++] = w * 32 + __ffs(m) - 1;
      }
      if (tid == 0) val[nneed] = 0;
      __syncthreads();
      if (tid == 0) s_pairs = 0;
      __syncthreads();
      entry([&](int at, int e, int u) {
        const int2 q = __ldg(A.iec + e);
        unsigned m = __ldg(A.mask + e), w = 0;
        if (m) {
          unsigned p = atomicAdd(&s_pairs, __popc(m));
          w = p << 4 | __popc(m);
          for (; m; m &= m - 1) {
            const int32_t* row = A.cid + (long long)(__ffs(m) - 1) * n;
            const int x = __ldg(row + u), y = __ldg(row + q.x);
            pairs[p++] = make_int2(x >= 0 ? place(wn * 32 + x) : nneed, y >= 0 ? place(wn * 32 + y) : nneed);
          }
        }
        rtab[at] = make_int4(place(u), place(q.x), q.y, (int)w);
      });
    }
  }
  const int32_t* rp = in ? s_rp : A.irp + v0;
  const int32_t* cp = in ? s_cp : A.cut_ptr + s0;
  const int own = in ? place(v0 < n ? v0 : 0) : 0, own_cut = in && nc ? place(wn * 32 + s0) : 0;
  // z fits 32 bits while the values stay below lim: a cost times 2^F is below 2^29
  // whatever the points
  static_assert(2LL * kCoordLimit * kCoordLimit << 2 * kMaxFracBits < 1LL << 58, "costs in units 2^-F");
  const int lim = ((1 << 30) - 1 + (1 << 29)) / (2 + 2 * L);
  bool any_long = false;
  __syncthreads();  // the tables are complete
  for (int i = tid; i < nc; i += kCutThreads) any_long |= cp[i + 1] - cp[i] > kLongCut;
  any_long = __syncthreads_or(any_long);
  int par = 0;  // the buffers that hold the result
  bool ok = grid_barrier_counted(&A.ctl->bar_count, gridDim.x, A.budget);
  if (!ok && tid == 0) atomicOr(&A.ctl->status, kGdpTimeout);
  for (long long t = 0; ok && t < A.max_sweeps; ++t) {
    const int p = (int)(t & 1), sl = (int)(t % 3);
    const int32_t *lam = A.lam[p], *mu = A.mu[p];
    long long b2 = 0;
    unsigned ch = 0;
    int ovf = 0;
    bool narrow = false;
    if (in) {
      bool big = false;
      for (int i = tid; i < nneed; i += kCutThreads) {
        const int w = need[i], x = w < wn * 32 ? __ldcg(lam + w) : __ldcg(mu + w - wn * 32);
        big |= x >= lim || x <= -lim;
        val[i] = x;
      }
      narrow = !__syncthreads_or(big);
    }
    auto new_lambda = [&](int i, long long lv, long long b, long long c) {
      const long long d = step_ll(b, c, A.shift), nl = lv + d;
      ovf |= (nl >= kLamLimit || nl <= -kLamLimit);
      __stcg(A.lam[p ^ 1] + v0 + i, (int32_t)nl);
      ch += (d != 0);
      b2 += 4LL * lv;
    };
    auto new_mu = [&](int s, long long b, long long c) {
      const long long m = in ? val[own_cut + s] : mu[s0 + s];
      const long long nm = max(0LL, m + step_ll(b, c, A.shift + 2));
      ovf |= (nm >= kLamLimit);
      __stcg(A.mu[p ^ 1] + s0 + s, (int32_t)nm);
      ch += (nm != m);
      b2 += 4 * m;
    };
    // entries [k, end) of cut s at this stride: the top-3 of the warp
    auto cut_scan = [&](int k, int end, int step, long long& a, long long& b, long long& c) {
      a = b = c = kInfZ;
      if (narrow) {
        int a1 = INT_MAX, b1 = INT_MAX, c1 = INT_MAX;
        cut_scan_in<false>(A, ktab, pairs, val, k, end, step, 0, a1, b1, c1, b2);
        cut_top3_group<32>(0xffffffffu, a1, b1, c1);
        if (a1 != INT_MAX) a = a1;
        if (b1 != INT_MAX) b = b1;
        if (c1 != INT_MAX) c = c1;
        return;
      }
      if (in)
        cut_scan_in<false>(A, ktab, pairs, val, k, end, step, 0, a, b, c, b2);
      else
        cut_scan_out<false>(A, 0, k, end, step, lam, mu, 0, a, b, c, b2);
      cut_top3_group<32>(0xffffffffu, a, b, c);
    };
    // A warp takes one cut or eight rows at a time, cuts first (they are the
    // longer ones).
    const int jobs = (nr + RW - 1) / RW;
    for (int job = warp; job < nc + jobs; job += NW) {
      if (job < nc) {
        // cut duals: Section 3's gradient over delta(S), projected onto mu >= 0
        const int k = cp[job], end = cp[job + 1];
        if (end - k > kLongCut) continue;
        long long a, b, c;
        cut_scan(k + lane, end, 32, a, b, c);
        if (lane == 0) new_mu(job, b, c);
        continue;
      }
      // node duals: Section 3's gradient over delta(v)
      const int i = (job - nc) * RW + lane / G;
      const bool has = i < nr;
      const int k = has ? rp[i] + sub : 0, end = has ? rp[i + 1] : 0;
      if (narrow) {
        const int lv = has ? val[own + i] : 0;
        int a = INT_MAX, b = INT_MAX, c = INT_MAX;
        cut_scan_in<true>(A, rtab, pairs, val, k, end, G, lv, a, b, c, b2);
        cut_top3_group<G>(gmask, a, b, c);
        if (sub == 0 && has) new_lambda(i, lv, b == INT_MAX ? kInfZ : b, c == INT_MAX ? kInfZ : c);
      } else {
        const int lv = !has ? 0 : in ? val[own + i] : lam[v0 + i];
        long long a = kInfZ, b = kInfZ, c = kInfZ;
        if (in)
          cut_scan_in<true>(A, rtab, pairs, val, k, end, G, lv, a, b, c, b2);
        else
          cut_scan_out<true>(A, v0 + i, k, end, G, lam, mu, lv, a, b, c, b2);
        cut_top3_group<G>(gmask, a, b, c);
        if (sub == 0 && has) new_lambda(i, lv, b, c);
      }
    }
    // long cuts: all warps on one, their top-3s merged in shared memory
    for (int s = 0; any_long && s < nc; ++s) {
      const int k = cp[s], end = cp[s + 1];
      if (end - k <= kLongCut) continue;
      long long a, b, c;
      cut_scan(k + tid, end, kCutThreads, a, b, c);
      if (lane == 0) { s_t3[3 * warp] = a; s_t3[3 * warp + 1] = b; s_t3[3 * warp + 2] = c; }
      __syncthreads();
      if (warp == 0) {
        a = lane < NW ? s_t3[3 * lane] : kInfZ;
        b = lane < NW ? s_t3[3 * lane + 1] : kInfZ;
        c = lane < NW ? s_t3[3 * lane + 2] : kInfZ;
        cut_top3_group<32>(0xffffffffu, a, b, c);
        if (lane == 0) new_mu(s, b, c);
      }
      __syncthreads();
    }
    if (t < A.trace_cap) {
      b2 = warp_sum_ll(b2);
      if (lane == 0 && b2) atomicAdd(reinterpret_cast<unsigned long long*>(&A.ctl->slot_b2[sl]), (unsigned long long)b2);
    }
    ch = warp_sum_u(ch);
    ovf = __any_sync(0xffffffffu, ovf);
    if (lane == 0 && ch) atomicAdd(&s_ch, ch);
    if (lane == 0 && ovf) s_ovf = 1;
    __syncthreads();
    // The sweep's barrier carries its totals: arrivals in bits 0-15, blocks that
    // overflowed in bits 16-31, changed duals above.  Its word is the sweep's
    // own (of three), so that nobody adds to it before everyone has read it.
    if (tid == 0) {
      unsigned long long* word = &A.ctl->slot_ch[sl];
      unsigned long long x = 1ull | (s_ovf ? 1ull << 16 : 0ull) | (unsigned long long)s_ch << 32;
      s_ch = 0;
      s_ovf = 0;
      asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(x) : "memory");
      const long long c0 = clock64();
      int stop = 0;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(word) : "memory");
        if ((x & 0xffff) == (unsigned)nb) break;
        if (clock64() - c0 > A.budget) { stop = 3; break; }
      }
      const unsigned chg = (unsigned)(x >> 32);
      if (stop == 3) {
        atomicOr(&A.ctl->status, kGdpTimeout);
      } else {
        const bool over = ((x >> 16) & 0xffff) != 0;
        stop = over ? 2 : chg == 0;
        if (blk == 0) {
          volatile GdpCtl* vc = A.ctl;
          if (t < A.trace_cap) {
            A.trace_b2[t] = vc->slot_b2[sl];
            A.trace_ch[t] = chg;
          }
          const int r = (int)((t + 2) % 3);  // read by everyone before this barrier
          vc->slot_b2[r] = 0;
          vc->slot_ch[r] = 0;
          vc->sweeps = t + 1;
          vc->fixed_point = (chg == 0);
          if (over) atomicOr(&A.ctl->status, kGdpOverflow);
        }
      }
      s_stop = stop;
    }
    __syncthreads();
    const int stop = s_stop;
    // an overflowing sweep is not kept: the result stays in its input
    if (stop < 2) par = p ^ 1;
    if (stop) break;
  }
  for (int i = v0 + tid; i < v1; i += kCutThreads) A.lam_out[__ldg(A.perm + i)] = __ldcg(A.lam[par] + i);
}

// bound2 at (lam, mu) with fb bits, and (x2 != NULL) rule (7) with the cut terms
__global__ void cut_bound_extract_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec,
                                         const uint8_t* __restrict__ mask, CutArgs ca,
                                         const int32_t* __restrict__ lam, const int32_t* __restrict__ mu,
                                         int32_t M, int32_t fb, uint8_t* x2, long long* b2_out,
                                         unsigned long long* bad) {
  long long b2 = 0;
  unsigned nb = 0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < ca.n; v += stride) {
    int s = 0;
    for (int e = rp[v]; e < rp[v + 1]; ++e) {
      const long long z = entry_z(ca, lam, mu, mask[e], (int)v, ec[e], fb);
      if (z < 0) b2 += z;
      const int x = z < 0 ? 2 : (z == 0 ? 1 : 0);
      if (x2) x2[e] = (uint8_t)x;
      s += x;
    }
    b2 += 4LL * lam[v];
    nb += (s != 4);
  }
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < M; q += stride) b2 += 4LL * mu[q];
  b2 = warp_sum_ll(b2);
  nb = warp_sum_u(nb);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(reinterpret_cast<unsigned long long*>(b2_out), (unsigned long long)b2);
    if (nb) atomicAdd(bad, (unsigned long long)nb);
  }
}

// ---- separation: connected components of the support {e : x2_e > 0} -------

__global__ void cc_init_kernel(int32_t* lab, int32_t n) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x)
    lab[v] = (int32_t)v;
}

// hook the larger of two roots under the smaller along every support entry
__global__ void cc_hook_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec,
                               const uint8_t* __restrict__ x2, int32_t n, int32_t* lab, int32_t* changed) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    for (int e = rp[v]; e < rp[v + 1]; ++e) {
      if (!x2[e]) continue;
      const int a = __ldcg(lab + v), b = __ldcg(lab + ec[e].x);
      if (a == b) continue;
      const int hi = a > b ? a : b, lo = a > b ? b : a;
      if (atomicMin(lab + hi, lo) > lo) *changed = 1;
    }
  }
}

// pointer jumping to the root
__global__ void cc_compress_kernel(int32_t* lab, int32_t n, int32_t* changed) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int r = __ldcg(lab + v);
    int rr = __ldcg(lab + r);
    if (rr == r) continue;
    while (rr != r) {
      r = rr;
      rr = __ldcg(lab + r);
    }
    lab[v] = r;
    *changed = 1;
  }
}

// crossing candidate entries per component (by root), and the root flags
__global__ void cc_cross_kernel(const int32_t* __restrict__ rp, const int2* __restrict__ ec,
                                const int32_t* __restrict__ lab, int32_t n, int32_t* cross, int32_t* root) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const int a = lab[v];
    int k = 0;
    for (int e = rp[v]; e < rp[v + 1]; ++e) k += (lab[ec[e].x] != a);
    if (k) atomicAdd(cross + a, k);
    root[v] = (a == (int)v);
  }
}

// which components become cuts: all if m >= 3, the one without node 0 if m = 2;
// only those with at least 3 crossing candidate edges
__global__ void cc_keep_kernel(const int32_t* __restrict__ lab, const int32_t* __restrict__ cross,
                               int32_t n, int32_t m, int32_t* keep) {
  const int r0 = lab[0];
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const bool is_root = lab[v] == (int)v;
    const bool take = m >= 3 || (m == 2 && (int)v != r0);
    keep[v] = (is_root && take && cross[v] >= 3) ? 1 : 0;
  }
}

__global__ void cc_label_kernel(const int32_t* __restrict__ lab, const int32_t* __restrict__ keep,
                                const int32_t* __restrict__ rank, int32_t n, int32_t* comp) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const int r = lab[v];
    comp[v] = keep[r] ? rank[r] : -1;
  }
}

// ---- pricing with cuts -----------------------------------------------------

// lamp_v = lambda_v + the duals of the cuts holding v: z_uv >= c 2^fb - lamp_u -
// lamp_v, so the plain scan with lamp finds a superset of the pairs
__global__ void cut_lamp_kernel(CutArgs ca, const int32_t* __restrict__ lam, const int32_t* __restrict__ mu,
                                int32_t* lamp, int32_t* overflow) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < ca.n;
       v += (long long)gridDim.x * blockDim.x) {
    long long x = lam[v];
    for (int l = 0; l < ca.L; ++l) {
      const int s = ca.comp[(long long)l * ca.n + v];
      if (s >= 0) x += mu[ca.off[l] + s];
    }
    if (x >= INT_MAX || x <= INT_MIN) {
      atomicOr(overflow, 1);
      x = 0;
    }
    lamp[v] = (int32_t)x;
  }
}

// exact z with the cut terms for every pair of the superset: keep flags
__global__ void cut_pair_keep_kernel(const int2* __restrict__ pairs, long long np, const int2* __restrict__ xy,
                                     CutArgs ca, const int32_t* __restrict__ lam, const int32_t* __restrict__ mu,
                                     int32_t fb, int32_t* keep) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < np;
       k += (long long)gridDim.x * blockDim.x) {
    const int2 p = pairs[k];
    long long t = 0;
    for (int l = 0; l < ca.L; ++l) {
      const int cu = ca.comp[(long long)l * ca.n + p.x], cv = ca.comp[(long long)l * ca.n + p.y];
      if (cu != cv) {
        if (cu >= 0) t += mu[ca.off[l] + cu];
        if (cv >= 0) t += mu[ca.off[l] + cv];
      }
    }
    const long long z = ((long long)exact_cost(xy[p.x], xy[p.y]) << fb) - lam[p.x] - lam[p.y] - t;
    keep[k] = z < 0;
  }
}

__global__ void cut_pair_compact_kernel(const int2* __restrict__ pairs, long long np,
                                        const int32_t* __restrict__ keep, const int32_t* __restrict__ pos,
                                        int2* out) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < np;
       k += (long long)gridDim.x * blockDim.x)
    if (keep[k]) out[pos[k]] = pairs[k];
}

int grid_of(long long items, int threads) {
  long long b = (items + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return (int)b;
}

CutArgs cut_args(const f2m_ctx* c) {
  CutArgs a{};
  a.comp = c->cuts->d_comp;
  a.n = c->n;
  a.L = c->cuts->L;
  for (int l = 0; l <= c->cuts->L; ++l) a.off[l] = c->cuts->off[l];
  return a;
}

template <typename T>
cudaError_t grow(T** p, int64_t* cap, int64_t need) {
  return dgrow(p, cap, need, need + need / 4 + 16);
}

}  // namespace

// Mask and cut lists for the graph held now (rebuilt after a merge or a new layer).
f2m_status cut_lists(f2m_ctx* c) {
  CutState* S = c->cuts;
  if (S->built_version == c->plan.version && S->built_L == S->L) return F2M_OK;
  const CutArgs a = cut_args(c);
  CK(c, grow(&S->d_mask, &S->mask_cap, c->nnz));
  cut_mask_kernel<<<grid_of(c->n, 256), 256, 0, c->st>>>(c->d_rp, c->d_ec, a, S->d_mask);
  count_launch();
  if (S->ptr_cap < S->M + 1) {
    dfree(S->d_cnt);
    dfree(S->d_ptr);
    dfree(S->d_scan);
    S->ptr_cap = 0;
    const int64_t room = S->M + 1 + 1024;
    CK(c, dalloc(&S->d_cnt, room));
    CK(c, dalloc(&S->d_ptr, room));
    CK(c, dalloc(&S->d_scan, (int64_t)scan_scratch_ints((int32_t)room)));
    S->ptr_cap = room;
  }
  const int32_t n = c->n, L = S->L, M = (int32_t)S->M;
  const GdpPlan& P = c->plan;
  CK(c, grow(&S->d_cid, &S->cid_cap, (int64_t)L * n));
  CK(c, grow(&S->d_imask, &S->imask_cap, c->nnz));
  CK(c, grow(&S->d_items, &S->item_cap, L * c->nnz));  // an entry crosses a layer's cuts once per row
  cut_cid_kernel<<<grid_of(n, 256), 256, 0, c->st>>>(a, P.perm, S->d_cid);
  count_launch();
  for (int fill = 0; fill < 2; ++fill) {
    CK(c, cudaMemsetAsync(S->d_cnt, 0, sizeof(int32_t) * (M + 1), c->st));
    if (!fill)
      cut_list_kernel<false><<<grid_of(n, 256), 256, 0, c->st>>>(P.irp, P.iec, S->d_cid, n, L, S->d_imask, S->d_cnt,
                                                                 nullptr, nullptr);
    else
      cut_list_kernel<true><<<grid_of(n, 256), 256, 0, c->st>>>(P.irp, P.iec, S->d_cid, n, L, S->d_imask, S->d_cnt,
                                                                S->d_ptr, S->d_items);
    count_launch();
    CK(c, cudaGetLastError());
    if (!fill) CK(c, launch_scan(S->d_cnt, S->d_ptr, M, S->d_scan, c->st));
  }
  S->built_version = c->plan.version;
  S->built_L = S->L;
  return F2M_OK;
}

f2m_status cut_gdp_phase(f2m_ctx* c, int64_t max_sweeps, int64_t* sweeps, long long* tb,
                         unsigned long long* tc, int64_t tcap, double* ms) {
  CutState* S = c->cuts;
  c->lam_version += 1;
  f2m_status s = cut_lists(c);
  if (s != F2M_OK) return s;
  *sweeps = 0;
  if (max_sweeps <= 0) return F2M_ERR_NOT_CONVERGED;
  CK(c, cudaMemsetAsync(c->d_gdp, 0, sizeof(GdpCtl), c->st));
  cudaEvent_t e0 = c->ev0, e1 = c->ev1;
  CK(c, cudaEventRecord(e0, c->st));
  const GdpPlan& P = c->plan;
  CutGdp g{};
  g.irp = P.irp;
  g.iec = P.iec;
  g.perm = P.perm;
  g.cid = S->d_cid;
  g.mask = S->d_imask;
  g.cut_ptr = S->d_ptr;
  g.items = S->d_items;
  g.lam_in = c->d_lam[c->cur];
  g.lam_out = c->d_lam[c->cur ^ 1];
  g.lam[0] = P.ilam[0];
  g.lam[1] = P.ilam[1];
  g.mu[0] = S->d_mu[S->cur];
  g.mu[1] = S->d_mu[S->cur ^ 1];
  g.ctl = c->d_gdp;
  g.trace_b2 = tb;
  g.trace_ch = tc;
  g.trace_cap = tcap;
  g.max_sweeps = max_sweeps;
  g.budget = c->p.barrier_budget_cycles;
  g.n = c->n;
  g.L = S->L;
  g.M = (int32_t)S->M;
  g.F = c->p.frac_bits;
  g.shift = c->p.damping_shift;
  void* args[] = {(void*)&g};
  CK(c, cudaFuncSetAttribute((const void*)cut_gdp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCutSmem));
  CK(c, cudaLaunchCooperativeKernel((const void*)cut_gdp_kernel, dim3(c->num_sms), dim3(kCutThreads), args, kCutSmem, c->st));
  count_launch();
  CK(c, cudaEventRecord(e1, c->st));
  GdpCtl h{};
  CK(c, cudaMemcpyAsync(&h, c->d_gdp, sizeof(h), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  if (ms) {
    float t = 0.f;
    cudaEventElapsedTime(&t, e0, e1);
    *ms += t;
  }
  *sweeps = h.sweeps;
  // the state after the last sweep that was kept: an overflowing sweep is not
  const bool ovf = (h.status & kGdpOverflow) != 0;
  const long long used = ovf ? h.sweeps - 1 : h.sweeps;
  if (!(h.status & kGdpTimeout)) c->cur ^= 1;  // written from the buffer kept
  if (used & 1) S->cur ^= 1;
  c->gdp_kernel = F2M_GDP_KERNEL_CUTS;
  if (h.status & kGdpTimeout) return fail(c, F2M_ERR_TIMEOUT, "device-wide barrier wait exceeded its budget");
  if (ovf) return fail(c, F2M_ERR_OVERFLOW, "|lambda| or a cut dual reached 2^29");
  return h.fixed_point ? F2M_OK : F2M_ERR_NOT_CONVERGED;
}

// bound2 (and rule (7) into d_x2 when want_x) at the current duals with cuts
f2m_status cut_bound_extract(f2m_ctx* c, bool want_x, int64_t* b2, int64_t* bad) {
  CutState* S = c->cuts;
  f2m_status s = cut_lists(c);
  if (s != F2M_OK) return s;
  int32_t fb = 0;
  const int32_t* lam = cur_lambda(c, &fb);
  if (fb != c->p.frac_bits) return fail(c, F2M_ERR_INVALID_ARG, "cut duals are held at F bits");
  CK(c, cudaMemsetAsync(c->d_scalar, 0, sizeof(long long), c->st));
  CK(c, cudaMemsetAsync(c->d_bad, 0, sizeof(unsigned long long), c->st));
  cut_bound_extract_kernel<<<grid_of(c->n, 256), 256, 0, c->st>>>(
      c->d_rp, c->d_ec, S->d_mask, cut_args(c), lam, S->d_mu[S->cur], (int32_t)S->M, fb,
      want_x ? c->d_x2 : nullptr, c->d_scalar, c->d_bad);
  count_launch();
  long long h = 0;
  unsigned long long nb = 0;
  CK(c, cudaMemcpyAsync(&h, c->d_scalar, sizeof(h), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaMemcpyAsync(&nb, c->d_bad, sizeof(nb), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  if (b2) *b2 = h;
  if (bad) *bad = (int64_t)nb;
  return F2M_OK;
}

// pricing with cuts: the plain scan with lamp (a superset), then the exact test
f2m_status cut_price(f2m_ctx* c, double* ms) {
  CutState* S = c->cuts;
  int32_t fb = 0;
  const int32_t* lam = cur_lambda(c, &fb);
  if (fb != c->p.frac_bits) return fail(c, F2M_ERR_INVALID_ARG, "cut duals are held at F bits");
  const int64_t n1 = c->n + 1;
  if (!S->d_lamp) CK(c, dalloc(&S->d_lamp, c->n));
  if (!S->d_small) CK(c, dalloc(&S->d_small, 4));
  const CutArgs a = cut_args(c);
  CK(c, cudaMemsetAsync(S->d_small, 0, sizeof(int32_t), c->st));
  cut_lamp_kernel<<<grid_of(c->n, 256), 256, 0, c->st>>>(a, lam, S->d_mu[S->cur], S->d_lamp, S->d_small);
  count_launch();
  int32_t ovf = 0;
  CK(c, cudaMemcpyAsync(&ovf, S->d_small, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  if (ovf) return fail(c, F2M_ERR_OVERFLOW, "lambda plus cut duals exceeds 32 bits");
  f2m_status s = price_internal(c, ms, S->d_lamp);
  if (s != F2M_OK) return s;
  const int64_t np = c->npairs;
  if (np == 0) return F2M_OK;
  if (np > S->pair_cap) {
    dfree(S->d_keep);
    dfree(S->d_kpos);
    dfree(S->d_pairs2);
    dfree(S->d_pscan);
    S->pair_cap = 0;
    const int64_t room = np + np / 4 + 1024;
    if (room >= INT_MAX) return fail(c, F2M_ERR_INVALID_ARG, "too many pricing pairs");
    CK(c, dalloc(&S->d_keep, room + 1));
    CK(c, dalloc(&S->d_kpos, room + 1));
    CK(c, dalloc(&S->d_pairs2, room));
    CK(c, dalloc(&S->d_pscan, (int64_t)scan_scratch_ints((int32_t)room + 1)));
    S->pair_cap = room;
  }
  (void)n1;
  cut_pair_keep_kernel<<<grid_of(np, 256), 256, 0, c->st>>>(c->d_pairs, np, c->d_xy, a, lam, S->d_mu[S->cur], fb,
                                                            S->d_keep);
  count_launch();
  CK(c, launch_scan(S->d_keep, S->d_kpos, (int32_t)np, S->d_pscan, c->st));
  cut_pair_compact_kernel<<<grid_of(np, 256), 256, 0, c->st>>>(c->d_pairs, np, S->d_keep, S->d_kpos, S->d_pairs2);
  count_launch();
  int32_t kept = 0;
  CK(c, cudaMemcpyAsync(&kept, S->d_kpos + np, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  if (kept > 0)
    CK(c, cudaMemcpyAsync(c->d_pairs, S->d_pairs2, sizeof(int2) * kept, cudaMemcpyDeviceToDevice, c->st));
  c->npairs = kept;
  c->seg_pairs.assign(1, kept);
  return F2M_OK;
}

// components of the support of the x held now as one cut layer: comp [n] on
// the device (d_comp_out), number of cuts in *m_out
f2m_status cut_separate(f2m_ctx* c, int32_t* d_comp_out, int32_t* m_out) {
  if (!c->cuts) c->cuts = new CutState();
  CutState* S = c->cuts;
  const int32_t n = c->n;
  if (!S->d_lab) CK(c, dalloc(&S->d_lab, n));
  if (!S->d_cross) CK(c, dalloc(&S->d_cross, n));
  if (!S->d_flag) CK(c, dalloc(&S->d_flag, n + 1));
  if (!S->d_rank) CK(c, dalloc(&S->d_rank, n + 1));
  if (!S->d_small) CK(c, dalloc(&S->d_small, 4));
  if (S->ptr_cap < n + 1) {
    dfree(S->d_cnt);
    dfree(S->d_ptr);
    dfree(S->d_scan);
    S->ptr_cap = 0;
    S->built_version = -1;
    CK(c, dalloc(&S->d_cnt, n + 1));
    CK(c, dalloc(&S->d_ptr, n + 1));
    CK(c, dalloc(&S->d_scan, (int64_t)scan_scratch_ints(n + 1)));
    S->ptr_cap = n + 1;
  }
  const int g = grid_of(n, 256);
  cc_init_kernel<<<g, 256, 0, c->st>>>(S->d_lab, n);
  count_launch();
  // hooking and pointer jumping until no label moves (the labels end at the
  // smallest node of each component); bounded by n rounds
  for (int32_t round = 0;; ++round) {
    if (round > n) return fail(c, F2M_ERR_CUDA, "component labelling did not settle");
    CK(c, cudaMemsetAsync(S->d_small, 0, sizeof(int32_t), c->st));
    cc_hook_kernel<<<g, 256, 0, c->st>>>(c->d_rp, c->d_ec, c->d_x2, n, S->d_lab, S->d_small);
    cc_compress_kernel<<<g, 256, 0, c->st>>>(S->d_lab, n, S->d_small);
    count_launches(2);
    int32_t changed = 0;
    CK(c, cudaMemcpyAsync(&changed, S->d_small, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
    CK(c, cudaStreamSynchronize(c->st));
    if (!changed) break;
  }
  CK(c, cudaMemsetAsync(S->d_cross, 0, sizeof(int32_t) * n, c->st));
  cc_cross_kernel<<<g, 256, 0, c->st>>>(c->d_rp, c->d_ec, S->d_lab, n, S->d_cross, S->d_flag);
  count_launch();
  CK(c, launch_scan(S->d_flag, S->d_rank, n, S->d_scan, c->st));
  int32_t m = 0;
  CK(c, cudaMemcpyAsync(&m, S->d_rank + n, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  cc_keep_kernel<<<g, 256, 0, c->st>>>(S->d_lab, S->d_cross, n, m, S->d_flag);
  count_launch();
  CK(c, launch_scan(S->d_flag, S->d_rank, n, S->d_scan, c->st));
  cc_label_kernel<<<g, 256, 0, c->st>>>(S->d_lab, S->d_flag, S->d_rank, n, d_comp_out);
  count_launch();
  int32_t kept = 0;
  CK(c, cudaMemcpyAsync(&kept, S->d_rank + n, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  *m_out = m >= 2 ? kept : 0;
  if (m < 2) CK(c, cudaMemsetAsync(d_comp_out, 0xff, sizeof(int32_t) * n, c->st));
  return F2M_OK;
}

// appends a layer from device labels; checks them and the crossing counts
f2m_status cut_add_layer(f2m_ctx* c, const int32_t* d_labels, int32_t ncuts) {
  if (!c->cuts) c->cuts = new CutState();
  CutState* S = c->cuts;
  if (S->L >= kMaxCutLayers) return fail(c, F2M_ERR_INVALID_ARG, "at most 8 cut layers");
  if (ncuts < 1) return fail(c, F2M_ERR_INVALID_ARG, "a layer needs at least one cut");
  if (c->seg_off.size() != 2) return fail(c, F2M_ERR_INVALID_ARG, "cuts are for single-instance contexts");
  if (c->d_b) return fail(c, F2M_ERR_INVALID_ARG, "cuts need b_v = 2 (F2M)");
  const int32_t n = c->n;
  if (!S->d_comp) CK(c, dalloc(&S->d_comp, (int64_t)kMaxCutLayers * n));
  if (!S->d_small) CK(c, dalloc(&S->d_small, 4));
  int32_t* dst = S->d_comp + (int64_t)S->L * n;
  CK(c, cudaMemcpyAsync(dst, d_labels, sizeof(int32_t) * n, cudaMemcpyDefault, c->st));
  int32_t big = INT_MAX;
  CK(c, cudaMemcpyAsync(S->d_small, &big, sizeof(int32_t), cudaMemcpyHostToDevice, c->st));
  cut_label_check_kernel<<<grid_of(n, 256), 256, 0, c->st>>>(dst, n, ncuts, S->d_small);
  count_launch();
  int32_t badv = INT_MAX;
  CK(c, cudaMemcpyAsync(&badv, S->d_small, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  if (badv != INT_MAX)
    return fail(c, F2M_ERR_INVALID_ARG, "cut label outside [-1, ncuts) at node " + std::to_string(badv));
  const int64_t M0 = S->M;
  // the duals: old ones kept, the new layer's at 0 (both halves of the buffer)
  if (M0 + ncuts > S->mu_cap) {
    int32_t* nb[2] = {nullptr, nullptr};
    const int64_t cap = (M0 + ncuts) * 2 + 1024;
    CK(c, dalloc(&nb[0], cap));
    CK(c, dalloc(&nb[1], cap));
    if (M0 > 0) CK(c, cudaMemcpyAsync(nb[0], S->d_mu[S->cur], sizeof(int32_t) * M0, cudaMemcpyDeviceToDevice, c->st));
    CK(c, cudaStreamSynchronize(c->st));
    dfree(S->d_mu[0]);
    dfree(S->d_mu[1]);
    S->d_mu[0] = nb[0];
    S->d_mu[1] = nb[1];
    S->cur = 0;
    S->mu_cap = cap;
  }
  CK(c, cudaMemsetAsync(S->d_mu[S->cur] + M0, 0, sizeof(int32_t) * ncuts, c->st));
  S->L += 1;
  S->ncuts.push_back(ncuts);
  S->off.assign(1, 0);
  for (int32_t v : S->ncuts) S->off.push_back(S->off.back() + v);
  S->M = M0 + ncuts;
  S->built_L = -1;
  f2m_status s = cut_lists(c);
  if (s == F2M_OK) {
    CK(c, cudaMemcpyAsync(S->d_small, &big, sizeof(int32_t), cudaMemcpyHostToDevice, c->st));
    cut_short_kernel<<<grid_of(ncuts, 256), 256, 0, c->st>>>(S->d_cnt + M0, ncuts, S->d_small);
    count_launch();
    CK(c, cudaMemcpyAsync(&badv, S->d_small, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
    CK(c, cudaStreamSynchronize(c->st));
    if (badv != INT_MAX)
      s = fail(c, F2M_ERR_INVALID_ARG,
               "cut " + std::to_string(badv) + " of the new layer has fewer than 3 crossing candidate edges");
  }
  if (s != F2M_OK) {  // take the layer back
    S->L -= 1;
    S->ncuts.pop_back();
    S->off.pop_back();
    S->M = M0;
    S->built_L = -1;
  }
  return s;
}

}  // namespace f2m

using namespace f2m;

extern "C" f2m_status f2m_separate(f2m_ctx* c, int32_t* comp, int32_t* ncuts) {
  if (!c || !ncuts) return fail(c, F2M_ERR_INVALID_ARG, "NULL argument");
  if (c->seg_off.size() != 2) return fail(c, F2M_ERR_INVALID_ARG, "cuts are for single-instance contexts");
  int32_t* d = nullptr;
  CK(c, dalloc(&d, c->n));
  int32_t m = 0;
  f2m_status s = cut_separate(c, d, &m);
  if (s == F2M_OK && comp) {
    cudaError_t e = cudaMemcpyAsync(comp, d, sizeof(int32_t) * c->n, cudaMemcpyDefault, c->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->st);
    if (e != cudaSuccess) s = cuda_fail(c, e, "copy labels");
  }
  cudaStreamSynchronize(c->st);
  dfree(d);
  *ncuts = m;
  return s;
}

extern "C" f2m_status f2m_add_cut_layer(f2m_ctx* c, const int32_t* comp, int32_t ncuts) {
  if (!c || !comp) return fail(c, F2M_ERR_INVALID_ARG, "NULL argument");
  return cut_add_layer(c, comp, ncuts);
}

extern "C" f2m_status f2m_get_cut_duals(f2m_ctx* c, int32_t* mu, int64_t* count, int32_t* layers) {
  if (!c || !count) return fail(c, F2M_ERR_INVALID_ARG, "NULL argument");
  const int64_t cap = *count;
  *count = cut_count(c);
  if (layers) *layers = c->cuts ? c->cuts->L : 0;
  if (!mu || *count == 0) return F2M_OK;
  if (cap < *count) return fail(c, F2M_ERR_INVALID_ARG, "capacity below the number of cuts");
  CK(c, cudaMemcpyAsync(mu, c->cuts->d_mu[c->cuts->cur], sizeof(int32_t) * *count, cudaMemcpyDefault, c->st));
  CK(c, cudaStreamSynchronize(c->st));
  return F2M_OK;
}

// The subtour driver: GDP phases with pricing (as f2m_solve's first phase,
// without the finisher), then rounds of separation, a new layer and GDP over
// node and cut duals with pricing, each round ending with rule (7) for the
// next separation.
extern "C" f2m_status f2m_solve_subtour(f2m_ctx* c, int32_t rounds, f2m_subtour_info* info_out) {
  if (!c) return fail(c, F2M_ERR_INVALID_ARG, "NULL context");
  if (rounds < 0 || rounds > kMaxCutLayers) return fail(c, F2M_ERR_INVALID_ARG, "rounds must be in 0..8");
  if (c->seg_off.size() != 2 || c->d_b) return fail(c, F2M_ERR_INVALID_ARG, "single F2M instance only");
  const auto t0 = std::chrono::steady_clock::now();
  f2m_subtour_info info;
  std::memset(&info, 0, sizeof(info));
  info.frac_bits = c->p.frac_bits;
  f2m_status status = F2M_OK;
  int32_t* d_lab = nullptr;
  CK(c, dalloc(&d_lab, c->n));
  // one stage: GDP phases with pricing until a scan finds nothing
  auto stage = [&](int64_t* b2_out) -> f2m_status {
    for (int32_t k = 0;; ++k) {
      int64_t sw = 0;
      f2m_status s = gdp_phase(c, c->p.max_iters, &sw, false, 0, &info.ms_gdp);
      info.iterations += sw;
      info.phases += 1;
      if (s != F2M_OK && s != F2M_ERR_NOT_CONVERGED) return s;
      if (!c->p.pricing) break;
      if (info.pricing_rounds >= c->p.max_pricing_rounds) return fail(c, F2M_ERR_NOT_CONVERGED, "pricing rounds exhausted");
      s = cut_count(c) ? cut_price(c, &info.ms_pricing) : price_internal(c, &info.ms_pricing, nullptr);
      if (s != F2M_OK) return s;
      info.pricing_rounds += 1;
      if (c->npairs == 0) break;
      const int64_t found = c->npairs;
      s = merge_internal(c, c->d_pairs, c->npairs, &info.ms_merge, true);
      if (s != F2M_OK) return s;
      info.edges_added += found;
    }
    int64_t bad = 0;
    f2m_status s = cut_count(c) ? cut_bound_extract(c, true, b2_out, &bad) : extract_internal(c, &bad, nullptr);
    if (s != F2M_OK) return s;
    if (!cut_count(c)) s = bound_internal(c, b2_out);
    return s;
  };
  int64_t b2 = 0;
  status = stage(&b2);
  info.bound2_f2m = b2;
  info.bound2 = b2;
  for (int32_t r = 0; r < rounds && status == F2M_OK; ++r) {
    const auto s0 = std::chrono::steady_clock::now();
    int32_t m = 0;
    status = cut_separate(c, d_lab, &m);
    info.ms_separate += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - s0).count();
    if (status != F2M_OK || m == 0) break;
    status = cut_add_layer(c, d_lab, m);
    if (status != F2M_OK) break;
    info.rounds += 1;
    info.cuts += m;
    status = stage(&b2);
    info.bound2 = b2;
  }
  dfree(d_lab);
  info.layers = c->cuts ? c->cuts->L : 0;
  info.certified = status == F2M_OK && c->p.pricing ? 1 : 0;
  info.status = status;
  info.ms_total = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  if (info_out) *info_out = info;
  return status;
}
