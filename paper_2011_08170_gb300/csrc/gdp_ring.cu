// GDP phase, shared-memory tiles that hand lambda to their neighbours (the
// default path of f2m_gdp / f2m_solve and of batches).
//
// The sweep is the Jacobi step of Eq. 9 and Eq. 10 (Section 5.1), as in gdp.cu:
//   z_e = c_e * 2^F - lambda_v - lambda_u,  delta_v = trunc((z(2) + z(3)) / 2^shift),
// so every result is bit-identical to the streaming kernel and to the oracle.
// What differs is where the data lives and how often the CTAs meet:
//
//  * Nodes are renumbered along a Morton curve (plan.cu); a tile is a contiguous
//    node range of one instance, a compact patch of the plane, owned by a CTA
//    that keeps its rows and lambda in shared memory for the whole phase.
//  * Around its own nodes a tile holds K rings: R1 the outside nodes adjacent to
//    own ones, R2 those adjacent to R1, and so on, with the rows of R1 ...
//    R(K-1).  A round is K sweeps: sweep s computes own rows and those of R1 ...
//    R(K-1-s) (the rings redundantly: their owners compute the same integers),
//    so the tile needs other tiles' lambda once per K sweeps.
//  * That exchange is point to point.  The last sweep of a round stores each own
//    lambda as one word with the round's tag; a neighbour polls the words of its
//    rings until they carry the round it waits for.  There is no barrier and
//    no fence between the store and the load: the word is its own flag.  Two
//    buffers suffice: a tile that publishes round r + 1 has read round r from
//    every tile that reads it (K-step neighbourhood is symmetric), so those have
//    read its round r - 1, which the new words overwrite.
//  * The stop test needs the whole instance: a tile adds, per round, which of the
//    K sweeps changed one of its lambdas to the round's slot (one 64-bit atomic),
//    and before round r every tile waits for the complete slot of round r - 3
//    and draws the same conclusion from it.  Sweeps past a fixed point change
//    nothing, so the late stop costs three rounds and no result.
//  * An overflow in sweep t leaves the exact state (that sweep's input)
//    unmaterialised; the host runs the phase again for t sweeps.
//
// Entries sit sliced: 32 rows a slice, one lane a row, deep rows together, entries 2 q and 2 q + 1 of the 32 rows side by side so that a lane
// loads two at a time.  They stay in registers for the whole phase, one or two rows a
// thread; tiles too large for that keep them in shared memory, as {local index,
// cost * 2^F} (8 bytes) or, where that does not fit, cost << 13 | local index (4).
//
// Bound: at 150 own rows a tile and fewer the latency of a row (about 0.45 us a
// sweep) and of the exchange (about 1.1 us a round: a store and a polling load
// through L2); above that instruction issue and shared-memory wavefronts (a
// gather of 32 rows' lambda takes about 2.5).  Per sweep, 128-sweep phases, against
// the form before it (rows in shared memory walked one entry pair at a time, a
// device-wide barrier per two sweeps): 1,000 points 1.9 to 0.75 us, 20,000 2.03 to
// 0.95, 100,000 2.85 to 1.62, 200,000 clustered (k = 12) 4.2 to 2.9; the tiles'
// construction 170 to 30 us at 100,000.  What each part gave at 100,000 / 20,000:
// entries in registers 2.7 to 2.4 / 1.45 to 1.15; words of 4 bytes in slot order
// and sorted rings (8-byte words in arrival order cost as much as two sweeps'
// rows) 2.4 to 1.92 / 1.15 to 1.0; the stop test in a warp of its own 1.92 to
// 1.78 / 1.0 to 0.95; merging triples instead of inserting was worth 5 % of the
// instructions.
#include <climits>
#include <cstddef>

#include "f2m_device.cuh"
#include "f2m_internal.h"

namespace f2m {

namespace {

constexpr int kPlanThreads = 1024;
constexpr int kRegEntries = 16;             // register form: entries of a row in registers
constexpr int kRingLamBytes = 4 * kRingLocals;    // between its two lambda arrays
constexpr int kHash = 2 * kRingHalo;        // slots of the plan's table of outside nodes
constexpr int kShallow = 12;                // entries of most rows (k = 10 graphs: three in four)
constexpr int kPackIdx = 13;                // bits of a packed local index
constexpr int kMaxEntries = 49152;          // sliced entries of a tile: what 4 bytes each could hold in shared memory
constexpr int kDepthBits = 11;              // a slice's word: its first entry << kDepthBits | its depth
constexpr int kDepthMask = (1 << kDepthBits) - 1;
static_assert(kRingDepth <= kDepthMask - 1 && kMaxEntries < 1 << (31 - kDepthBits), "a slice's word");
static_assert(kRingDepth % 2 == 0 && kRingLong % 2 == 0 && kRingTail % 2 == 0, "a depth is even");
static_assert(kRingTail >= kRegEntries && kRingTail < kRingLong, "what a lane keeps");
constexpr uint32_t kPackPadCost = (1u << (32 - kPackIdx)) - 1;  // cost of a packed padding entry
// lambda of the padding slot in the packed form: with cost kPackPadCost its z
// is about 2^30 - lambda_v, above every real one (as the 8-byte padding's)
constexpr int kPackPadLam = -(1 << 30) + (1 << 27);
static_assert(kRingLocals <= (1 << kPackIdx), "local indices fit the packed form");

constexpr int kHashBits = 13;
static_assert(kHash == 1 << kHashBits, "table size");
__device__ __forceinline__ unsigned hash_slot(int c) { return ((unsigned)c * 2654435761u) >> (32 - kHashBits); }

// position of an outside node in the tile's ring list
__device__ __forceinline__ int hash_find(const int* keys, const uint16_t* vals, int c) {
  unsigned h = hash_slot(c);
  while (keys[h] != c) h = (h + 1) & (kHash - 1);
  return vals[h];
}

}  // namespace

// One CTA per tile: its node range (an equal share of its instance's nodes),
// the rings (each sorted by node), the slots, the slice table and the sliced
// entries.  A section (own rows, R1, ..., R(K-1)) starts a slice; its rows with
// more than 12 entries come first, by falling degree, then the others in node
// order, so that a slice's words are neighbours in the exchange and a reader's
// sorted ring finds several in a sector.  An own node's local index is its slot,
// a ring node's ownp + its position (ownp: own slots, whole slices).
__global__ void __launch_bounds__(kPlanThreads, 1)
ring_plan_kernel(const int32_t* __restrict__ irp, const int2* __restrict__ iec, const RingTile* __restrict__ list,
                 const int32_t* __restrict__ seg_off, int32_t tiles, int32_t K, int32_t F, int32_t ecap, int32_t maxdeg,
                 RingHdr* __restrict__ hdr, int32_t* __restrict__ halo, uint16_t* __restrict__ order,
                 uint32_t* __restrict__ slc, uint32_t* __restrict__ longs, int2* __restrict__ ent,
                 int32_t* __restrict__ pos, RingStats* stats, RingSeg* seg, RingLimit limit,
                 int32_t first) {
  extern __shared__ __align__(16) unsigned char smem[];
  int* keys = reinterpret_cast<int*>(smem);                         // [kHash] outside nodes
  int* ring = keys + kHash;                                         // [kRingHalo] in ring order
  int* fresh = ring + kRingHalo;                                    // [kRingHalo] as found
  uint16_t* vals = reinterpret_cast<uint16_t*>(fresh + kRingHalo);  // [kHash] position in ring
  uint16_t* at_key = vals + kHash;                                  // [kRingHalo] table slot of a found node
  uint16_t* deg = at_key + kRingHalo;                               // [kRingLocals] per row (own, then ring)
  uint16_t* ord = deg + kRingLocals;                                // [kRingSlots] row of a slot
  uint16_t* inv = ord + kRingSlots;                                 // [kRingLocals] slot of an own node
  __shared__ int s_cnt, s_bad, s_hist[64], s_maxcost, s_tail, s_long;
  __shared__ int s_sl[kRingSlices + 1];
  __shared__ int s_warp[33];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  RingTile tl{0, b, tiles};
  if (list) tl = list[b];
  const int n0 = seg_off[tl.seg], ns = seg_off[tl.seg + 1] - n0;
  for (int i = tid; i < kHash; i += kPlanThreads) keys[i] = -1;
  if (tid == 0) {
    s_cnt = 0;
    s_bad = 0;
    s_maxcost = 0;
    s_tail = 0;
    s_long = 0;
  }
  __syncthreads();
  const int lo = n0 + (int)((long long)ns * tl.j / tl.count), hi = n0 + (int)((long long)ns * (tl.j + 1) / tl.count);
  const int own = hi - lo, ownp = (own + 31) & ~31;
  // ring nodes that fit beside own slots and the two padding slots
  const int room = min(kRingHalo, kRingLocals - 2 - ownp);
  RingHdr h{};
  h.lo = lo;
  h.own = own;
  h.seg = tl.seg;
  h.count = tl.count;
  h.first = tl.j == 0;
  h.word0 = lo + 32 * (first + b);
  int bad = room < 32 ? kRingBadSize : 0;
  auto insert = [&](int c) {
    if (c >= lo && c < hi) return;
    unsigned s = hash_slot(c);
    for (;;) {
      const int k = atomicCAS(&keys[s], -1, c);
      if (k == c) return;
      if (k == -1) {
        const int p = atomicAdd(&s_cnt, 1);
        if (p < room) {
          fresh[p] = c;
          at_key[p] = (uint16_t)s;
        }
        return;
      }
      s = (s + 1) & (kHash - 1);
      if (*reinterpret_cast<volatile int*>(&s_cnt) > room) return;  // too many: the table may be full
    }
  };
  // rings, breadth first: 8 lanes a row
  int ring_end[kRingMax + 1];
  ring_end[0] = 0;
  if (!bad)
    for (int e = irp[lo] + tid; e < irp[hi]; e += kPlanThreads) insert(iec[e].x);
  __syncthreads();
#pragma unroll
  for (int k = 1; k <= kRingMax; ++k) {
    if (k > K) break;
    const int end = s_cnt, beg = ring_end[k - 1];
    if (end > room) bad = kRingBadSize;
    ring_end[k] = bad ? 0 : end;
    __syncthreads();
    if (!bad) {
      // rank by counting: a ring holds a few hundred nodes
      for (int i = beg + tid; i < end; i += kPlanThreads) {
        const int c = fresh[i];
        int rank = beg;
        for (int j = beg; j < end; ++j) rank += fresh[j] < c;
        ring[rank] = c;
        vals[at_key[i]] = (uint16_t)rank;
      }
      if (k < K)
        for (int i = beg + (tid >> 3); i < end; i += kPlanThreads / 8) {
          const int v = fresh[i];
          for (int e = irp[v] + (tid & 7); e < irp[v + 1]; e += 8) insert(iec[e].x);
        }
    }
    __syncthreads();
  }
  int HH = 0, rows = own;
#pragma unroll
  for (int k = 1; k <= kRingMax; ++k) {
    if (k == K) HH = ring_end[k];
    if (k == K - 1) rows = own + ring_end[k];
  }
  auto node_of = [&](int l) { return l < own ? lo + l : ring[l - own]; };
  if (!bad) {
    for (int l = tid; l < rows; l += kPlanThreads) {
      const int g = node_of(l), d = irp[g + 1] - irp[g];
      if (d > maxdeg) atomicOr(&s_bad, kRingBadSize);
      deg[l] = (uint16_t)min(d, maxdeg);
    }
    for (int h2 = tid; h2 < HH; h2 += kPlanThreads) halo[(size_t)b * kRingHalo + h2] = ring[h2];
  }
  __syncthreads();
  bad |= s_bad;
  int slots = 0;
  int sec_slice[kRingMax + 1];
#pragma unroll
  for (int k = 0; k < kRingMax; ++k) {
    sec_slice[k] = slots / 32;
    if (k >= K || bad) continue;
    const int a = k == 0 ? 0 : own + ring_end[k - 1], z = k == 0 ? own : own + ring_end[k];
    if (slots + (z - a) + 31 > kRingSlots) {
      bad = kRingBadSize;
      continue;
    }
    // deep rows: bins 0 (63 entries and more) ... 50 (13); the others in order
    if (tid < 64) s_hist[tid] = 0;
    __syncthreads();
    const int chunk = (z - a + kPlanThreads - 1) / kPlanThreads;
    const int l0 = min(z, a + tid * chunk), l1 = min(z, l0 + chunk);
    int flat = 0;
    for (int l = l0; l < l1; ++l) {
      if (deg[l] <= kShallow) ++flat;
      else atomicAdd(&s_hist[63 - min((int)deg[l], 63)], 1);
    }
    int nflat = 0;
    int f = block_exclusive_scan(flat, s_warp, nflat);  // a barrier: the bins are complete
    if (tid < 32) {  // exclusive sums of the bins
      int x0 = s_hist[2 * tid], x1 = s_hist[2 * tid + 1], s = x0 + x1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, s, o);
        if (tid >= o) s += y;
      }
      s_hist[2 * tid] = slots + s - x0 - x1;
      s_hist[2 * tid + 1] = slots + s - x1;
    }
    __syncthreads();
    f += slots + (z - a) - nflat;
    for (int l = l0; l < l1; ++l) {
      const int p = deg[l] <= kShallow ? f++ : atomicAdd(&s_hist[63 - min((int)deg[l], 63)], 1);
      ord[p] = (uint16_t)l;
      if (k == 0) inv[l] = (uint16_t)p;
    }
    const int end = slots + (z - a), pad = (end + 31) & ~31;
    for (int p = end + tid; p < pad; p += kPlanThreads) ord[p] = 0xFFFF;
    slots = pad;
    __syncthreads();
  }
  sec_slice[kRingMax] = slots / 32;
  const int nsl = bad ? 0 : slots / 32;
  // depth of a slice (even), offsets
  for (int s = warp; s < nsl; s += kPlanThreads / 32) {
    const int l = ord[s * 32 + lane];
    const int dl = l == 0xFFFF ? 0 : (int)deg[l], d = __reduce_max_sync(0xffffffffu, dl);
    const unsigned longs_of = d > kRingLong ? __ballot_sync(0xffffffffu, dl > kRingTail) : 0u;
    if (lane == 0) {
      s_sl[s] = (d + 1) & ~1;
      longs[(size_t)b * kRingSlices + s] = longs_of;
      if (d > kRegEntries) atomicAdd(&s_tail, 32 * (((d + 1) & ~1) - kRegEntries));
      if (longs_of) s_long = 1;
    }
  }
  __syncthreads();
  const int depth = tid < nsl ? s_sl[tid] : 0;
  int nent = 0;
  const int off = block_exclusive_scan(32 * depth, s_warp, nent);
  static_assert(kRingSlices <= kPlanThreads, "one thread per slice");
  if (nent > ecap) bad = kRingBadRoom;
  if (tid < nsl && !bad) {
    s_sl[tid] = off << kDepthBits | depth;
    slc[(size_t)b * kRingSlices + tid] = (uint32_t)(off << kDepthBits | depth);
  }
  __syncthreads();
  // entries
  int maxcost = 0;
  if (!bad) {
    const int zero_slot = ownp + HH;
    int2* out = ent + (size_t)b * ecap;
    for (int p = tid; p < slots; p += kPlanThreads) order[(size_t)b * kRingSlots + p] = ord[p];
    for (int l = tid; l < own; l += kPlanThreads) pos[lo + l] = h.word0 + inv[l];
    auto local_of = [&](int c) { return c >= lo && c < hi ? (int)inv[c - lo] : ownp + hash_find(keys, vals, c); };
    for (int s = warp; s < nsl; s += kPlanThreads / 32) {
      const int l = ord[s * 32 + lane], o = s_sl[s] >> kDepthBits, dep = s_sl[s] & kDepthMask;
      const int g = l == 0xFFFF ? -1 : node_of(l);
      const int a = g >= 0 ? irp[g] : 0, d = g >= 0 ? irp[g + 1] - a : 0;
      for (int k = 0; k < dep; k += 2) {
        int4 q = make_int4(zero_slot, 1 << 30, zero_slot, 1 << 30);
        if (k < d) {
          const int2 r = iec[a + k];
          q.x = local_of(r.x);
          q.y = r.y << F;  // cost in units 2^-F
          maxcost = max(maxcost, r.y);
        }
        if (k + 1 < d) {
          const int2 r = iec[a + k + 1];
          q.z = local_of(r.x);
          q.w = r.y << F;
          maxcost = max(maxcost, r.y);
        }
        *reinterpret_cast<int4*>(out + o + k * 32 + lane * 2) = q;
      }
    }
  }
  maxcost = __reduce_max_sync(0xffffffffu, maxcost);
  if (lane == 0) atomicMax(&s_maxcost, maxcost);
  __syncthreads();
  if (tid == 0) {
    h.halo = HH;
    h.nsl = nsl;
    h.nent = nent;
#pragma unroll
    for (int k = 0; k < kRingMax; ++k) h.sec_end[k] = sec_slice[k + 1];  // slices of sections 0 .. k
    hdr[b] = h;
    // shared memory: entries, two lambda arrays, ring words, rows of slots, slices
    const int rest = 8 * (ownp + HH + 2) + 4 * HH + 2 * slots + 4 * nsl + 64;
    atomicMax(&stats->bytes8, 8 * nent + rest);
    atomicMax(&stats->bytes4, 4 * nent + rest);
    atomicMax(&stats->slices, nsl);
    if (s_long) stats->longs = 1;
    atomicMax(&stats->locals, ownp + HH + 2);
    atomicMax(&stats->maxcost, s_maxcost);
    const int bytes_reg = 2 * kRingLamBytes + 4 * (HH + nsl) + 8 * s_tail + 64;
    atomicMax(&stats->bytes_reg, bytes_reg);
    if (limit.smem && (bad || bytes_reg > limit.smem || nsl > limit.slices || ownp + HH + 2 > limit.locals ||
                       s_maxcost >= limit.cost))
      seg[tl.seg].unfit = 1;
    if (bad) atomicOr(&stats->bad, bad);
  }
}

namespace {

// two entries of a lane's row: {local index, cost * 2^F} each
template <bool PACKED>
__device__ __forceinline__ int4 two_entries(const void* ent, int at, int F) {
  if constexpr (PACKED) {
    const uint2 e = *reinterpret_cast<const uint2*>(reinterpret_cast<const uint32_t*>(ent) + at);
    constexpr uint32_t m = (1u << kPackIdx) - 1;
    return make_int4((int)(e.x & m), (int)(e.x >> kPackIdx) << F, (int)(e.y & m), (int)(e.y >> kPackIdx) << F);
  } else {
    return *reinterpret_cast<const int4*>(reinterpret_cast<const int2*>(ent) + at);
  }
}

// Entries from kRingTail on of the slice's rows flagged in `rows`: the warp takes one
// row after the other, its lanes pairs of that row's entries, whose top-3 (and
// sum of min(0, z)) go to the row's lane.  As one lane's chain an entry cost 40
// cycles, and every tile waits for the one with the longest row: 128 sweeps of 3,000
// points, one with 256 neighbours, 826 us, so 355; 100,000 points, one with 300,
// 1,016 and 474 (the streaming kernel 2,150).  All lanes of the warp call it.
template <bool BOUND, typename Two>
__device__ __forceinline__ void long_rows(unsigned rows, int depth, int lv, const Two& two, const int* s_in, int& a,
                                          int& zb, int& zc, long long& neg) {
  const int lane = threadIdx.x & 31;
  for (; rows; rows &= rows - 1) {
    const int row = __ffs(rows) - 1, l = __shfl_sync(0xffffffffu, lv, row);
    int x = INT_MAX, y = INT_MAX, w = INT_MAX;
    long long sum = 0;
    for (int k = kRingTail + 2 * lane; k < depth; k += 64) {
      const int4 q = two(k, row);
      const int z = q.y - l - s_in[q.x], z1 = q.w - l - s_in[q.z];
      if (BOUND) sum += min(z, 0) + min(z1, 0);
      top3_insert_minmax(z, x, y, w);
      top3_insert_minmax(z1, x, y, w);
    }
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
      const int x1 = __shfl_xor_sync(0xffffffffu, x, o), y1 = __shfl_xor_sync(0xffffffffu, y, o),
                w1 = __shfl_xor_sync(0xffffffffu, w, o);
      top3_merge(x1, y1, w1, x, y, w);
    }
    if (BOUND) sum = warp_sum_ll(sum);
    if (lane == row) {
      top3_merge(x, y, w, a, zb, zc);
      if (BOUND) neg += sum;
    }
  }
}

// z(2) and z(3) of one row (Eq. 10): two top-3 chains over alternate entries,
// merged; if BOUND, also the row's sum of min(0, z)
template <bool PACKED, bool BOUND>
__device__ __forceinline__ void row_top3(const void* ent, int at, int depth, int F, int lv, const int* s_in,
                                         const uint32_t* longs, int& zb, int& zc, long long& neg) {
  int a = INT_MAX, a1 = INT_MAX, b1 = INT_MAX, c1 = INT_MAX;
  zb = INT_MAX;
  zc = INT_MAX;
  const int stop = depth > kRingLong ? kRingTail : depth;
#pragma unroll 4
  for (int k = 0; k < stop; k += 2) {
    const int4 q = two_entries<PACKED>(ent, at + k * 32, F);
    const int z = q.y - lv - s_in[q.x];  // Eq. 9
    const int z1 = q.w - lv - s_in[q.z];
    if (BOUND) neg += min(z, 0) + min(z1, 0);
    top3_insert_minmax(z, a, zb, zc);
    top3_insert_minmax(z1, a1, b1, c1);
  }
  top3_merge(a1, b1, c1, a, zb, zc);
  if (depth > kRingLong) {
    const int row0 = at - (threadIdx.x & 31) * 2;
    long_rows<BOUND>(*longs, depth, lv, [&](int k, int row) { return two_entries<PACKED>(ent, row0 + k * 32 + row * 2, F); },
                     s_in, a, zb, zc, neg);
  }
}

// Degree requirements b_v (Section 3 with Eq. 8): z(b_v) and z(b_v + 1) of one
// row.  NB > 0 (every b_v < NB): the row's NB smallest values kept sorted in
// registers; NB = 0: counting, the entry value t being z(r) iff #{z < t} < r <=
// #{z <= t}.  Padding entries have z above every real one and at least b_v + 1
// entries are real.
template <bool PACKED, bool BOUND, int NB>
__device__ __forceinline__ void row_pair_deg(const void* ent, int at, int depth, int F, int lv, const int* s_in, int bv,
                                             int& zb, int& zc, long long& neg) {
  zb = INT_MAX;
  zc = INT_MAX;
  if constexpr (NB > 0) {
    int a[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) a[k] = INT_MAX;
    auto insert = [&](int z) {
#pragma unroll
      for (int j = NB - 1; j > 0; --j) a[j] = min(a[j], max(a[j - 1], z));
      a[0] = min(a[0], z);
    };
#pragma unroll 2
    for (int k = 0; k < depth; k += 2) {
      const int4 q = two_entries<PACKED>(ent, at + k * 32, F);
      const int z = q.y - lv - s_in[q.x], z1 = q.w - lv - s_in[q.z];
      if (BOUND) neg += min(z, 0) + min(z1, 0);
      insert(z);
      insert(z1);
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      if (k == bv - 1) zb = a[k];
      if (k == bv) zc = a[k];
    }
  } else {
    // two entries counted against two at a time: a pair's load and its two gathers
    // serve four comparisons (128 sweeps of 100,000 points with b_v up to 10: 1.64 ms,
    // 3.43 with a load and a gather for each)
    auto z_of = [&](int k) {
      const int4 q = two_entries<PACKED>(ent, at + k * 32, F);
      return make_int2(q.y - lv - s_in[q.x], q.w - lv - s_in[q.z]);
    };
    for (int j = 0; j < depth; j += 2) {
      const int2 t = z_of(j);
      if (BOUND) neg += min(t.x, 0) + min(t.y, 0);
      int lt0 = 0, le0 = 0, lt1 = 0, le1 = 0;
#pragma unroll 4
      for (int k = 0; k < depth; k += 2) {
        const int2 z = z_of(k);
        lt0 += (z.x < t.x) + (z.y < t.x);
        le0 += (z.x <= t.x) + (z.y <= t.x);
        lt1 += (z.x < t.y) + (z.y < t.y);
        le1 += (z.x <= t.y) + (z.y <= t.y);
      }
      if (lt0 < bv && bv <= le0) zb = min(zb, t.x);
      if (lt0 <= bv && bv + 1 <= le0) zc = min(zc, t.x);
      if (lt1 < bv && bv <= le1) zb = min(zb, t.y);
      if (lt1 <= bv && bv + 1 <= le1) zc = min(zc, t.y);
    }
  }
}

// A word of the exchange: lambda (30 bits, |lambda| < 2^29) and, in the low two
// bits, 1 + bit 1 of its round.  A buffer holds round r over round r - 2's words,
// so that bit tells them apart; 0 is no round (the buffers start cleared).
__device__ __forceinline__ unsigned word_tag(int r) { return 1u + ((unsigned)(r >> 1) & 1u); }
__device__ __forceinline__ unsigned word_of(int lam, unsigned tag) { return (unsigned)lam << 2 | tag; }
__device__ __forceinline__ unsigned ld_word(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(unsigned* p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_slot(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void add_slot(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// A wait on another tile, bounded: by `budget` cycles, and by any tile's
// time-out (polled now and then), so that all end when one does.
struct RingWait {
  long long t0, budget;
  int* status;
  unsigned polls = 0;
  __device__ __forceinline__ bool give_up() {
    if (clock64() - t0 <= budget &&
        ((++polls & 255u) != 0u || !(*reinterpret_cast<volatile int*>(status) & kGdpTimeout)))
      return false;
    atomicOr(status, kGdpTimeout);
    return true;
  }
};

// A round's sweep for one row's new lambda: into the tile's array, and, from an
// own row, the flags (bit 0 changed, bit 16 overflow) and the word to publish.
struct RowOut {
  unsigned flags = 0;
  // Eq. 10 (Eq. 8), truncated toward 0; |lambda| < 2^29 and costs below
  // 1.5 10^6 2^8 keep z and the new lambda inside 32 bits
  __device__ __forceinline__ int step(int zb, int zc, int lv, int shift) { return lv + gdp_step32(zb, zc, shift); }
  __device__ __forceinline__ void own(int nl, int lv) {
    flags |= (unsigned)(nl != lv) | ((nl >= (int)kLamLimit || nl <= -(int)kLamLimit) ? 0x10000u : 0u);
  }
};

// A traced sweep's sums of the row warps' own rows, by the sweep's parity: written
// before the barrier that ends sweep t, read by the warp beside them behind it,
// and written again after the next one.  One atomic a tile, sweep and word: an
// atomic of every row on the sweep's two words had taken 7.6 ms for 128 sweeps of
// 100,000 points, now 0.36 (0.25 without a trace, in registers).
struct RingTrace {
  long long b2[2][32];
  unsigned ch[2][32];
};

// Rows whose entries stay in shared memory (any number that fits).
// MODE 0: b_v = 2 (top-3); 1: every b_v < 5; 2: every b_v < 8; 3: any b_v.
template <int MODE, bool BOUND, bool PACKED, int NW>
struct SmemRows {
  const void* s_ent;
  int* s_lam;
  const int* s_ring;
  const uint32_t* s_slc;
  const uint16_t* s_ord;
  const uint32_t* longs;
  const int32_t* bnode;  // node of a ring row (degree requirements)
  int L, own, ownp, lo;

  __device__ __forceinline__ int* lam(int par) const { return s_lam + (par ? L : 0); }

  __device__ __forceinline__ void init(const RingArgs& A, const RingHdr& h, int b, unsigned char* smem) {
    const int tid = threadIdx.x, T = blockDim.x, nent = h.nent, nsl = h.nsl;
    own = h.own;
    ownp = (own + 31) & ~31;
    lo = h.lo;
    L = ownp + h.halo + 1;
    bnode = A.halo + (size_t)b * kRingHalo;
    longs = A.longs + (size_t)b * kRingSlices;
    s_ent = smem;
    s_lam = reinterpret_cast<int*>(smem + (size_t)nent * (PACKED ? 4 : 8));  // two arrays of L
    int* ring = s_lam + 2 * L;
    uint32_t* slc = reinterpret_cast<uint32_t*>(ring + h.halo);
    uint16_t* ord = reinterpret_cast<uint16_t*>(slc + nsl);
    const int2* ent = A.ent + (size_t)b * A.ecap;
    if constexpr (PACKED) {
      for (int e = tid; e < nent; e += T) {
        const int2 q = ent[e];
        const uint32_t c = q.y == (1 << 30) ? kPackPadCost : (uint32_t)(q.y >> A.F);
        reinterpret_cast<uint32_t*>(smem)[e] = c << kPackIdx | (uint32_t)q.x;
      }
    } else {
      for (int e = tid; e < nent / 2; e += T)
        reinterpret_cast<int4*>(smem)[e] = reinterpret_cast<const int4*>(ent)[e];
    }
    for (int i = tid; i < h.halo; i += T) ring[i] = A.pos[bnode[i]];
    for (int i = tid; i < nsl; i += T) slc[i] = A.slc[(size_t)b * kRingSlices + i];
    for (int i = tid; i < 32 * nsl; i += T) ord[i] = A.order[(size_t)b * kRingSlots + i];
    if (tid == 0) lam(0)[L - 1] = lam(1)[L - 1] = PACKED ? kPackPadLam : 0;
    s_ring = ring;
    s_slc = slc;
    s_ord = ord;
  }
  __device__ __forceinline__ const int* ring() const { return s_ring; }

  __device__ __forceinline__ unsigned sweep(const RingArgs& A, int par, int end, int sown, bool last,
                                            unsigned* pub, unsigned tag, RingTrace* trace, int t) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int* in = lam(par);
    int* out = lam(par ^ 1);
    RowOut o;
    long long b2 = 0;
    unsigned ch = 0;
    for (int sl = warp; sl < end; sl += NW) {
      const uint32_t od = s_slc[sl];
      const int row = s_ord[sl * 32 + lane];
      const bool has = row != 0xFFFF;
      if (MODE != 0 && !has) continue;  // with b_v = 2 the warp stays together (long rows)
      const int vl = sl < sown ? sl * 32 + lane : ownp + row - own;  // its local index
      const int lv = has ? in[vl] : 0, at = (int)(od >> kDepthBits) + lane * 2, depth = (int)(od & kDepthMask);
      int zb, zc, bv = 2;
      long long neg = 0;
      if constexpr (MODE == 0) {
        row_top3<PACKED, BOUND>(s_ent, at, depth, A.F, lv, in, longs + sl, zb, zc, neg);
        if (!has) continue;
      } else {
        bv = __ldg(A.bint + (row < own ? lo + row : bnode[row - own]));
        row_pair_deg<PACKED, BOUND, MODE == 1 ? 5 : (MODE == 2 ? 8 : 0)>(s_ent, at, depth, A.F, lv, in, bv, zb, zc, neg);
      }
      const int nl = o.step(zb, zc, lv, A.shift);
      out[vl] = nl;
      if (sl < sown) {
        o.own(nl, lv);
        if (last) st_word(pub + vl, word_of(nl, tag));
        if constexpr (BOUND) {
          b2 += neg + 2LL * bv * lv;
          ch += nl != lv;
        }
      }
    }
    if constexpr (BOUND) {
      if (warp < sown) {  // the same warps every sweep: the others' sums stay 0
        b2 = warp_sum_ll(b2);
        ch = warp_sum_u(ch);
        if (lane == 0) {
          trace->b2[t & 1][warp] = b2;
          trace->ch[t & 1][warp] = ch;
        }
      }
    }
    return o.flags;
  }
};

// address bits of a packed entry in a register, by row warps; cost of a padding entry
__host__ __device__ constexpr int reg_address_bits(int nw) { return nw < 16 ? 13 : 14; }
__host__ __device__ constexpr int reg_pad_cost(int bits) { return (int)((1u << (32 - bits)) - 1u); }
__host__ __device__ __forceinline__ bool reg_packs(const RingStats& st, int nw) {
  const int bits = reg_address_bits(nw);
  return st.locals <= 1 << (bits - 2) && st.maxcost < reg_pad_cost(bits);
}

// Rows whose entries stay in registers: R rows a thread, at most kRegEntries
// entries each (deeper slices keep the rest in shared memory).  R = 1: an entry
// is the byte address of its lambda in the tile's array and its cost; R = 2:
// both in one register, cost << AB | address: 13 bits of address (2,048 nodes a
// tile, costs below 2^19 - 1) with two CTAs per SM, 14 with one.  The two
// lambda arrays lie a constant apart, so that a gather is one load with an
// immediate offset (the two parities are compiled separately).
// LONG: the warp takes what long rows have past kRingTail entries (b_v = 2); a form
// of its own, since it spills a few registers.
template <int MODE, int R, int NW, bool LONG>
struct RegRows {
  static constexpr bool PACKED = R > 1;
  static constexpr int AB = reg_address_bits(NW);
  static constexpr int D = kRegEntries;
  static constexpr int NB = MODE == 1 ? 5 : 8;
  unsigned char* sm;
  int* s_ring;
  const int2* s_tail;
  const uint32_t* s_dep;  // per slice: where its entries past D begin << kDepthBits | depth
  int F;
  uint16_t vl[R];         // local index, 0xFFFF for a padding row
  uint32_t ea[R][D];                  // address, or the packed entry
  int ec[PACKED ? 1 : R][PACKED ? 1 : D];  // cost * 2^F
  uint8_t bv[MODE ? R : 1];

  __device__ __forceinline__ int* lam(int par) const { return reinterpret_cast<int*>(sm + par * kRingLamBytes); }
  __device__ __forceinline__ const int* ring() const { return s_ring; }

  // a slice's entries past D to shared memory, after those of the slices before
  __device__ __forceinline__ static void keep(const uint32_t* slc, const int2* ent, int sl, int at, int depth,
                                              uint32_t* dep, int2* tl) {
    const int lane = threadIdx.x & 31;
    int o = 0;
    if (depth > D) {
      for (int q = lane; q < sl; q += 32) o += max(0, (int)(slc[q] & kDepthMask) - D) * 32;
      o = __reduce_add_sync(0xffffffffu, o);
      for (int k = D; k < depth; k += 2)
        *reinterpret_cast<int4*>(tl + o + (k - D) * 32 + lane * 2) = *reinterpret_cast<const int4*>(ent + at + k * 32);
    }
    if (lane == 0) dep[sl] = (uint32_t)o << kDepthBits | (uint32_t)depth;
  }

  __device__ __forceinline__ void init(const RingArgs& A, const RingHdr& h, int b, unsigned char* smem) {
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5;
    sm = smem;
    s_ring = reinterpret_cast<int*>(smem + 2 * kRingLamBytes);
    uint32_t* dep = reinterpret_cast<uint32_t*>(s_ring + h.halo);
    const int nsl = h.nsl;
    int2* tl = reinterpret_cast<int2*>(smem + ((2 * kRingLamBytes + 4 * (h.halo + nsl) + 15) & ~15));
    s_dep = dep;
    s_tail = tl;
    F = A.F;
    const int ownp = (h.own + 31) & ~31, zero_slot = ownp + h.halo;
    const int32_t* halo = A.halo + (size_t)b * kRingHalo;
    for (int i = tid; i < h.halo; i += T) s_ring[i] = A.pos[halo[i]];
    // padding entries' slots: of 8-byte entries, and of those packed here
    if (tid == 0) {
      lam(0)[zero_slot] = lam(1)[zero_slot] = 0;
      lam(0)[zero_slot + 1] = lam(1)[zero_slot + 1] = kPackPadLam;
    }
    const uint32_t* slc = A.slc + (size_t)b * kRingSlices;
    const int2* ent = A.ent + (size_t)b * A.ecap;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int sl = warp + r * NW;
      vl[r] = 0xFFFF;
      if (MODE) bv[MODE ? r : 0] = 2;
      int at = 0, depth = 0;
      if (warp < NW && sl < nsl) {
        const uint32_t od = slc[sl];
        depth = (int)(od & kDepthMask);
        at = (int)(od >> kDepthBits) + lane * 2;
        const int row = A.order[(size_t)b * kRingSlots + sl * 32 + lane];
        if (row != 0xFFFF) vl[r] = (uint16_t)(row < h.own ? sl * 32 + lane : ownp + row - h.own);
        if (MODE > 0 && row != 0xFFFF)
          bv[MODE ? r : 0] = (uint8_t)A.bint[row < h.own ? h.lo + row : halo[row - h.own]];
        keep(slc, ent, sl, at, depth, dep, tl);
      }
#pragma unroll
      for (int k = 0; k < D; k += 2) {
        int4 q = make_int4(zero_slot, 1 << 30, zero_slot, 1 << 30);
        if (k < depth) q = *reinterpret_cast<const int4*>(ent + at + k * 32);
        if constexpr (PACKED) {
          auto pack = [&](int at_, int c) {
            return c == (1 << 30) ? (uint32_t)reg_pad_cost(AB) << AB | (uint32_t)(zero_slot + 1) << 2
                                  : (uint32_t)(c >> F) << AB | (uint32_t)at_ << 2;
          };
          ea[r][k] = pack(q.x, q.y);
          ea[r][k + 1] = pack(q.z, q.w);
        } else {
          ea[r][k] = (uint32_t)q.x << 2;
          ec[r][k] = q.y;
          ea[r][k + 1] = (uint32_t)q.z << 2;
          ec[r][k + 1] = q.w;
        }
      }
    }
  }

  template <int PAR>
  __device__ __forceinline__ int z_of(uint32_t a, int c, int lam_v) const {
    if constexpr (PACKED) {
      asm volatile("" : "+r"(a));  // keeps the unpacked form from being held in registers across sweeps
      c = (int)(a >> AB) << F;
      a &= (1u << AB) - 1u;
    }
    return c - lam_v - *reinterpret_cast<const int*>(sm + PAR * kRingLamBytes + a);  // Eq. 9
  }

  // the row's order pair from its first N entries and the tail
  template <int PAR, int N>
  __device__ __forceinline__ void pair_of(const RingArgs& A, int r, int l, int depth, uint32_t dt, int& zb, int& zc) const {
    const int lane = threadIdx.x & 31;
    int z[N];
#pragma unroll
    for (int k = 0; k < N; ++k) z[k] = z_of<PAR>(ea[r][k], PACKED ? 0 : ec[PACKED ? 0 : r][PACKED ? 0 : k], l);
    const int4* tl = reinterpret_cast<const int4*>(s_tail + (dt >> kDepthBits) + lane * 2);
    if constexpr (MODE == 0) {
      int a;
      top3_of4(z[0], z[1], z[2], z[3], a, zb, zc);
#pragma unroll
      for (int k = 4; k < N; k += 4) {
        int a1, b1, c1;
        top3_of4(z[k], z[k + 1], z[k + 2], z[k + 3], a1, b1, c1);
        top3_join(a1, b1, c1, a, zb, zc);
      }
      if constexpr (N == D) {
        const int stop = LONG && depth > kRingLong ? kRingTail : depth;
        for (int k = D; k < stop; k += 2) {
          const int4 q = tl[(k - D) * 16];
          top3_insert_minmax(q.y - l - lam(PAR)[q.x], a, zb, zc);
          top3_insert_minmax(q.w - l - lam(PAR)[q.z], a, zb, zc);
        }
        if (LONG && depth > kRingLong) {
          const int4* row0 = reinterpret_cast<const int4*>(s_tail + (dt >> kDepthBits));
          long long none = 0;
          long_rows<false>(A.longs[(size_t)blockIdx.x * kRingSlices + (threadIdx.x >> 5) + r * NW], depth,
                           l, [&](int k, int row) { return row0[(k - D) * 16 + row]; }, lam(PAR), a, zb, zc, none);
        }
      }
    } else {
      int s[NB];
#pragma unroll
      for (int k = 0; k < NB; ++k) s[k] = INT_MAX;
      auto insert = [&](int x) {
#pragma unroll
        for (int j = NB - 1; j > 0; --j) s[j] = min(s[j], max(s[j - 1], x));
        s[0] = min(s[0], x);
      };
#pragma unroll
      for (int k = 0; k < N; ++k) insert(z[k]);
      zb = zc = INT_MAX;
      if constexpr (N == D) {
        for (int k = D; k < depth; k += 2) {
          const int4 q = tl[(k - D) * 16];
          insert(q.y - l - lam(PAR)[q.x]);
          insert(q.w - l - lam(PAR)[q.z]);
        }
      }
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        if (k == bv[MODE ? r : 0] - 1) zb = s[k];
        if (k == bv[MODE ? r : 0]) zc = s[k];
      }
    }
  }

  template <int PAR>
  __device__ __forceinline__ unsigned sweep_p(const RingArgs& A, int end, int sown, bool last, unsigned* pub,
                                              unsigned tag) {
    const int warp = threadIdx.x >> 5;
    RowOut o;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int sl = warp + r * NW;
      if (sl >= end) break;
      const uint32_t dt = s_dep[sl];
      const int depth = (int)(dt & kDepthMask), v = vl[r];
      const int l = v != 0xFFFF ? lam(PAR)[v] : 0;
      // no branch between a row's gathers: all are in flight together
      int zb, zc;
      if (depth <= 12)
        pair_of<PAR, 12>(A, r, l, depth, dt, zb, zc);
      else
        pair_of<PAR, D>(A, r, l, depth, dt, zb, zc);
      const int nl = o.step(zb, zc, l, A.shift);
      if (v != 0xFFFF) {
        lam(PAR ^ 1)[v] = nl;
        if (sl < sown) {
          o.own(nl, l);
          if (last) st_word(pub + v, word_of(nl, tag));
        }
      }
    }
    return o.flags;
  }
  __device__ __forceinline__ unsigned sweep(const RingArgs& A, int par, int end, int sown, bool last,
                                            unsigned* pub, unsigned tag, RingTrace*, int) {
    return par ? sweep_p<1>(A, end, sown, last, pub, tag) : sweep_p<0>(A, end, sown, last, pub, tag);
  }
};

// What the warps of a tile tell each other, by the round's parity where a warp may
// enter round r + 1 while another still reads round r's.
struct RingShared {
  int stop[2], abort[2];
  unsigned flags[2];  // sweeps of the round that changed (bit s) or overflowed (bit 16 + s) an own lambda
  int end[kRingMax];
};

// The stop test (and the trace's totals), by one warp beside those with the rows: the
// same barriers.
template <int NW>
__device__ __noinline__ void ring_boss(const RingArgs& A, const RingHdr& h, RingShared& S, const RingTrace* trace) {
  const int lane = threadIdx.x & 31, K = A.K, max_sweeps = A.max_sweeps;
  RingSeg* sg = A.seg + h.seg;
  const int width = 48 / K;  // bits of a slot's count of tiles a sweep changed, after 16 of arrivals
  RingWait wait{clock64(), A.budget, A.status};
  int done = -1, fixed = 0, ovf = 0;  // sweeps run, once known
  // a complete round's verdict: the first sweep that overflowed or changed nothing
  auto wait_slot = [&](int q) -> bool {
    wait.t0 = clock64();
    for (;;) {
      const unsigned long long v = ld_slot(&sg->slot[q % kRingRing]);
      if ((int)(v & 0xFFFFu) == h.count) {
        const unsigned of = *reinterpret_cast<volatile unsigned*>(&sg->ovf[q % kRingRing]);
        for (int s = 0; s < K && q * K + s < max_sweeps && done < 0; ++s) {
          ovf = (of >> s) & 1u;
          fixed = !ovf && ((v >> (16 + width * s)) & ((1ull << width) - 1)) == 0;
          if (ovf || fixed) done = q * K + s + 1;
        }
        return true;
      }
      if (wait.give_up()) return false;
    }
  };
  auto add_trace = [&](int t) {  // behind the barrier that ends sweep t
    if (!trace || t >= A.trace_cap) return;
    const long long b2 = warp_sum_ll(lane < NW ? trace->b2[t & 1][lane] : 0);
    const unsigned ch = warp_sum_u(lane < NW ? trace->ch[t & 1][lane] : 0u);
    if (lane == 0) {
      if (b2) atomicAdd(reinterpret_cast<unsigned long long*>(A.trace_b2 + t), (unsigned long long)b2);
      if (ch) atomicAdd(A.trace_ch + t, (unsigned long long)ch);
    }
  };
  int r = 0;
  for (;; ++r) {
    const int kk = min(max_sweeps - r * K, K);  // sweeps of this round
    if (lane == 0) {
      int stop = kk <= 0;
      if (r >= 3) {
        if (!wait_slot(r - 3)) S.abort[r & 1] = 1;
        if (done >= 0) stop = 1;
        // every tile has passed round r - 3, so none reads the slot of round
        // r - 5 any more; it is round r + 11's next
        if (h.first && r >= 5) {
          sg->slot[(r - 5) % kRingRing] = 0;
          sg->ovf[(r - 5) % kRingRing] = 0;
        }
      }
      S.stop[r & 1] = stop;
    }
    __syncthreads();
    if (S.abort[r & 1]) return;
    if (lane == 0 && r >= 1) {  // this tile's part of the last round
      const unsigned f = *reinterpret_cast<volatile unsigned*>(&S.flags[(r - 1) & 1]);
      S.flags[(r - 1) & 1] = 0;
      unsigned long long v = 1;
      for (int s = 0; s < K; ++s) v += (unsigned long long)((f >> s) & 1u) << (16 + width * s);
      if (f >> 16) atomicOr(&sg->ovf[(r - 1) % kRingRing], f >> 16);
      add_slot(&sg->slot[(r - 1) % kRingRing], v);
    }
    __syncwarp();
    if (r >= 1) add_trace(min(r * K, max_sweeps) - 1);
    if (S.stop[r & 1]) break;
    for (int s = 1; s < kk; ++s) {
      __syncthreads();
      add_trace(r * K + s - 1);
    }
  }
  // a phase that ran to its cap: the verdict of the last rounds
  if (lane == 0 && h.first) {
    bool ok = true;
    for (int q = max(r - 2, 0); ok && done < 0 && q < r; ++q) ok = wait_slot(q);
    sg->sweeps = done >= 0 ? done : max_sweeps;
    sg->fixed_point = fixed;
    sg->overflow = ovf;
  }
}

// The rounds of one tile: the last warp runs the stop test, the others hold the rows.
template <typename Rows, int T>
__device__ __forceinline__ void ring_run(const RingArgs& A, const RingHdr& h, unsigned char* smem,
                                         RingTrace* trace = nullptr) {
  constexpr int NW = T / 32 - 1;  // warps with rows
  __shared__ RingShared S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
  const int ownp = (h.own + 31) & ~31;
  const uint16_t* order = A.order + (size_t)b * kRingSlots;
  const int32_t* halo = A.halo + (size_t)b * kRingHalo;
  Rows rows;
  rows.init(A, h, b, smem);
  for (int i = tid; i < ownp; i += T) {
    const int row = order[i];
    if (row != 0xFFFF) rows.lam(0)[i] = A.lam_in[A.perm[h.lo + row]];
  }
  for (int i = tid; i < h.halo; i += T) rows.lam(0)[ownp + i] = A.lam_in[A.perm[halo[i]]];
  if (tid < kRingMax) S.end[tid] = A.hdr[b].sec_end[tid];
  if (tid < 2) S.abort[tid] = S.flags[tid] = 0;
  if (trace && tid < 64) {
    trace->b2[tid & 1][tid >> 1] = 0;
    trace->ch[tid & 1][tid >> 1] = 0;
  }
  __syncthreads();
  if (warp == NW) {
    ring_boss<NW>(A, h, S, trace);
    return;
  }
  const int* s_ring = rows.ring();
  const int HH = h.halo, K = A.K;
  int par = 0;  // the array that holds lambda now
  int left = A.max_sweeps;
  for (int r = 0;; ++r, left -= K) {
    if (r > 0 && left > 0) {
      const unsigned tag = word_tag(r);
      const unsigned* buf = A.words[r & 1];
      int* in = rows.lam(par) + ownp;
      RingWait wait{clock64(), A.budget, A.status};
      for (int i = tid; i < HH; i += NW * 32) {
        unsigned v;
        while (((v = ld_word(buf + s_ring[i])) & 3u) != tag)
          if (wait.give_up()) {
            S.abort[r & 1] = 1;
            break;
          }
        in[i] = (int)v >> 2;
      }
    }
    __syncthreads();
    if (S.abort[r & 1]) return;
    if (S.stop[r & 1]) break;
    const int kk = min(left, K);
    for (int s = 0; s < kk; ++s) {
      // in the round's last sweep nothing but own rows is needed
      const bool last = s == kk - 1;
      const int sown = S.end[0], end = last ? sown : S.end[K - 1 - s];
      if (warp < end) {
        unsigned flags = rows.sweep(A, par, end, sown, last, A.words[(r + 1) & 1] + h.word0, word_tag(r + 1), trace,
                                    r * K + s);
        flags = __reduce_or_sync(0xffffffffu, flags);
        if (lane == 0 && flags) atomicOr(&S.flags[r & 1], flags << s);
      }
      par ^= 1;
      if (!last) __syncthreads();
    }
  }
  // own lambda to caller order (row warps alone: the last sweep's stores are behind the round's barrier)
  for (int i = tid; i < ownp; i += NW * 32) {
    const int row = order[i];
    if (row != 0xFFFF) A.lam_out[A.perm[h.lo + row]] = rows.lam(par)[i];
  }
}

}  // namespace

// Every tile reads the same statistics, so all take the same form (two CTAs per SM,
// a batch: an instance's tiles read its own flag).
template <int MODE, bool BOUND, int T>
__global__ void __launch_bounds__(T, T == 512 && MODE < 2 ? 2 : 1)
gdp_ring_smem_kernel(const __grid_constant__ RingArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  const RingStats st = *A.stats;
  const bool wide = st.bytes8 <= A.smem, packed = st.bytes4 <= A.smem && (uint32_t)st.maxcost < kPackPadCost;
  if (st.bad || !(wide || packed)) {
    if (threadIdx.x == 0) atomicOr(A.status, kGdpNoFit);
    return;
  }
  const RingHdr h = A.hdr[blockIdx.x];
  RingTrace* trace = nullptr;
  if constexpr (BOUND) {
    __shared__ RingTrace s_trace;
    trace = &s_trace;
  }
  if (wide)
    ring_run<SmemRows<MODE, BOUND, false, T / 32 - 1>, T>(A, h, smem, trace);
  else
    ring_run<SmemRows<MODE, BOUND, true, T / 32 - 1>, T>(A, h, smem, trace);
}

template <int MODE, int R, int T, bool LONG = false>
__global__ void __launch_bounds__(T, 1024 / T)
gdp_ring_reg_kernel(const __grid_constant__ RingArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NW = T / 32 - 1;
  const RingHdr h = A.hdr[blockIdx.x];
  if constexpr (T == 512) {
    if (A.seg[h.seg].unfit) return;
  } else {
    const RingStats st = *A.stats;
    if (st.bad || st.bytes_reg > A.smem || st.slices > R * NW || (R > 1 && !reg_packs(st, NW)) ||
        (MODE == 0 && LONG != (st.longs != 0))) {
      if (threadIdx.x == 0) atomicOr(A.status, kGdpNoFit);
      return;
    }
  }
  ring_run<RegRows<MODE, R, NW, LONG>, T>(A, h, smem);
}

// ---- host side -------------------------------------------------------------------------

#define RCK(call)                    \
  do {                               \
    cudaError_t e_ = (call);         \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

template <typename T>
static cudaError_t grow(T** p, int64_t* cap, int64_t need) {
  if (*p && *cap >= need) return cudaSuccess;
  if (*p) dev_free(*p);
  *p = nullptr;
  *cap = 0;
  cudaError_t e = dev_malloc((void**)p, sizeof(T) * (size_t)need);
  if (e == cudaSuccess) *cap = need;
  return e;
}

void ring_free(RingPlan& p) {
  void* ptrs[] = {p.hdr, p.halo, p.order, p.slc, p.longs, p.ent, p.pos, p.rec, p.words};
  for (void* q : ptrs)
    if (q) dev_free(q);
  p = RingPlan();
}

static cudaError_t ring_records(RingPlan& p, int32_t nseg) {
  if (p.seg_cap >= nseg) return cudaSuccess;
  if (p.rec) dev_free(p.rec);
  p.rec = nullptr;
  p.seg_cap = 0;
  RCK(dev_malloc((void**)&p.rec, sizeof(RingRecord) + sizeof(RingSeg) * (size_t)nseg));
  p.seg_cap = nseg;
  return cudaSuccess;
}

cudaError_t ring_build(const GdpPlan& g, const int32_t* seg_off, const RingTile* list, int32_t tiles, int32_t K,
                       int32_t F, int64_t entries_per_tile, int32_t maxdeg, int32_t nseg, RingPlan& p,
                       cudaStream_t st, const RingLimit& limit, int32_t first, int32_t room) {
  // room for a tile's sliced entries: its own and its inner rings'
  const int64_t want = entries_per_tile < 0 ? kMaxEntries
                       : K > 1              ? entries_per_tile * 2 + 16384
                                            : entries_per_tile * 3 / 2 + 4096;
  const int64_t ecap = (want < kMaxEntries ? want : kMaxEntries) / 64 * 64;
  p.version = -1;
  const int64_t m = room > tiles ? room : tiles;
  RCK(grow(&p.hdr, &p.hdr_cap, m));
  RCK(grow(&p.halo, &p.halo_cap, m * kRingHalo));
  RCK(grow(&p.pos, &p.pos_cap, g.n));
  RCK(grow(&p.order, &p.order_cap, m * kRingSlots));
  RCK(grow(&p.slc, &p.slc_cap, m * kRingSlices));
  RCK(grow(&p.longs, &p.longs_cap, m * kRingSlices));
  RCK(grow(&p.ent, &p.ent_cap, m * ecap));
  RCK(ring_records(p, nseg));
  RCK(cudaMemsetAsync(&p.rec->stats, 0, sizeof(RingStats), st));
  constexpr size_t smem = 4 * (kHash + 2 * kRingHalo) + 2 * (kHash + kRingHalo + 2 * kRingLocals + kRingSlots);
  RCK(cudaFuncSetAttribute(ring_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ring_plan_kernel<<<tiles, kPlanThreads, smem, st>>>(g.irp, g.iec, list, seg_off, tiles, K, F, (int32_t)ecap, maxdeg, p.hdr,
                                                      p.halo, p.order, p.slc, p.longs, p.ent, p.pos, &p.rec->stats, p.rec->seg, limit, first);
  count_launch();
  RCK(cudaGetLastError());
  p.ecap = (int32_t)ecap;
  p.K = K;
  p.tiles = tiles;
  p.F = F;
  p.version = g.version;
  return cudaSuccess;
}

cudaError_t ring_start(RingPlan& p, int32_t n, int32_t tiles, int32_t nseg, cudaStream_t st) {
  RCK(ring_records(p, nseg));
  const int64_t m = (int64_t)n + 32LL * tiles;  // a tile's own slots are whole slices
  RCK(grow(&p.words, &p.words_cap, 2 * m));
  p.words_n = m;
  RCK(cudaMemsetAsync(p.words, 0, sizeof(unsigned) * 2 * m, st));
  return cudaMemsetAsync(&p.rec->status, 0,
                         offsetof(RingRecord, seg) - offsetof(RingRecord, status) + sizeof(RingSeg) * nseg, st);
}

template <int MODE, int T>
static const void* ring_kernel_of(bool bound) {
  return bound ? (const void*)gdp_ring_smem_kernel<MODE, true, T> : (const void*)gdp_ring_smem_kernel<MODE, false, T>;
}

template <int R>
static const void* ring_reg_kernel_of(int mode, bool longs) {
  return mode == 0   ? (longs ? (const void*)gdp_ring_reg_kernel<0, R, 1024, true>
                              : (const void*)gdp_ring_reg_kernel<0, R, 1024>)
         : mode == 1 ? (const void*)gdp_ring_reg_kernel<1, R, 1024>
                     : (const void*)gdp_ring_reg_kernel<2, R, 1024>;
}

int ring_reg_rows(const RingStats& st) {
  if (st.bad || st.bytes_reg > ring_smem(false, false)) return 0;
  if (st.slices <= 31) return 1;
  return st.slices <= 62 && reg_packs(st, 31) ? 2 : 0;
}

RingLimit ring_pair_limit() {
  constexpr int bits = reg_address_bits(15);
  return RingLimit{ring_smem(true, false), 2 * 15, 1 << (bits - 2), reg_pad_cost(bits)};
}

int32_t ring_smem(bool half, bool traced) {
  int dev = 0, optin = 0, sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess)
    return 0;
  // less what the kernel holds statically, and what the system keeps of each CTA
  return ((half ? sm / 2 - 1024 : optin) - 128 - (traced ? (int)sizeof(RingTrace) : 0)) & ~15;
}

cudaError_t launch_gdp_ring(const GdpPlan& g, RingPlan& p, int32_t tiles, const int32_t* lam_in,
                            int32_t* lam_out, int32_t shift, int32_t max_sweeps, long long* trace_b2,
                            unsigned long long* trace_ch, int64_t trace_cap, long long budget, const int32_t* bint,
                            int32_t bmax, RingForm form, bool longs, cudaStream_t st) {
  const bool bound = trace_cap > 0, half = form == kRingHalf || form == kRingPair, reg = form > 0;
  const int mode = !bint ? 0 : (bmax < 5 ? 1 : (bmax < 8 ? 2 : 3));
  if (reg && (bound || mode > (form == kRingPair ? 0 : 2))) return cudaErrorInvalidValue;
  const int T = reg ? (half ? 512 : 1024) : (half || mode >= 2 ? 512 : 1024);
  const void* kern = form == kRingReg1   ? ring_reg_kernel_of<1>(mode, longs)
                     : form == kRingReg2 ? ring_reg_kernel_of<2>(mode, longs)
                     : form == kRingPair ? (const void*)gdp_ring_reg_kernel<0, 2, 512>
                     : half && mode == 0 ? ring_kernel_of<0, 512>(bound)
                     : mode == 0       ? ring_kernel_of<0, 1024>(bound)
                     : mode == 1       ? (half ? ring_kernel_of<1, 512>(bound) : ring_kernel_of<1, 1024>(bound))
                     : mode == 2       ? ring_kernel_of<2, 512>(bound)
                                       : ring_kernel_of<3, 512>(bound);
  const int dyn = ring_smem(half, bound);
  RCK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
  RingArgs a{};
  a.hdr = p.hdr;
  a.halo = p.halo;
  a.order = p.order;
  a.slc = p.slc;
  a.longs = p.longs;
  a.ent = p.ent;
  a.stats = &p.rec->stats;
  a.seg = p.rec->seg;
  a.words[0] = p.words;
  a.words[1] = p.words + p.words_n;
  a.pos = p.pos;
  a.status = &p.rec->status;
  a.lam_in = lam_in;
  a.lam_out = lam_out;
  a.perm = g.perm;
  a.bint = bint;
  a.trace_b2 = trace_b2;
  a.trace_ch = trace_ch;
  a.trace_cap = trace_cap;
  a.max_sweeps = (int32_t)max_sweeps;
  a.budget = budget;
  a.K = p.K;
  a.F = p.F;
  a.shift = shift;
  a.ecap = p.ecap;
  a.smem = dyn;
  void* args[] = {(void*)&a};
  cudaError_t e = cudaLaunchCooperativeKernel(kern, dim3(tiles), dim3(T), args, (size_t)dyn, st);
  count_launch();
  return e;
}

}  // namespace f2m
