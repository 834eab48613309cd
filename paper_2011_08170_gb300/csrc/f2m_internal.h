// Internal declarations of the f2m library (not part of the C ABI).
//
// Device data layout (one instance, n nodes, nnz directed CSR entries):
//   xy    int2[n]          point coordinates, each in [0, 2^20)
//   rp    int32[n+1]       CSR row offsets (both directions of every edge stored)
//   ec    int2[nnz]        per entry {col, cost}: 8 bytes streamed per entry
//   lam   int32[2][n]      lambda, Jacobi double buffer (units 2^-F)
//   lam2  int32[n]         lambda of the finisher (units 2^-(F+1))
//   x2    uint8[nnz]       primal x in half units
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

namespace f2m {

constexpr int32_t kCoordLimit = 1 << 20;   // coordinates in [0, 2^20)
constexpr int64_t kLamLimit = 1LL << 29;   // |lambda| < 2^29 in units 2^-F
constexpr int kMaxFracBits = 8;            // of lambda, F
constexpr int kMaxCutLayers = 8;           // layers of subtour-elimination cuts (cuts.cu)

// Control block of the persistent GDP kernel (device memory, zeroed per phase).
struct GdpCtl {
  unsigned int bar_count;      // arrivals at the current barrier
  unsigned int bar_gen;        // barrier generation
  int status;                  // bit 0: lambda overflow, bit 1: barrier timeout
  int fixed_point;             // 1 if the last sweep changed no lambda
  long long slot_b2[3];        // per-sweep bound2 accumulators (ring of 3)
  unsigned long long slot_ch[3];  // per-sweep changed counts (ring of 3)
  long long sweeps;            // sweeps completed
};

constexpr int kGdpOverflow = 1;
constexpr int kGdpTimeout = 2;
constexpr int kGdpNoFit = 4;        // shared-memory tiles: some tile does not fit

// Validation result written by the create-time check kernel.
struct CheckCtl {
  int flags;                   // bit set per violated rule
  int first_bad;               // smallest offending node (or entry)
};

enum CheckBits {
  kBadRowPtr = 1,
  kBadCol = 2,
  kUnsorted = 4,
  kSelfLoop = 8,
  kAsymmetric = 16,
  kLowDegree = 32,
  kBadCoord = 64,
  kBadPair = 128,
  kBadDegreeReq = 256,
};

// Device memory of this library (api.cu): a process-wide cache of freed
// blocks per device.  dev_free waits for the device (as cudaFree does) before
// the block can be handed out again; dev_free_synced is for a caller that has
// already waited for every use of the block.
cudaError_t dev_malloc(void** p, size_t bytes);
void dev_free(void* p);
void dev_free_synced(void* p);
// Room for `need` items in *p, whose values are not kept: as it is, or a block of
// `room`.  Where there is no memory the old block stays, so that calls after a
// failed one find every array that the graph they see needs.
template <typename T>
cudaError_t dev_regrow(T** p, int64_t* cap, int64_t need, int64_t room) {
  if (*p && *cap >= need) return cudaSuccess;
  void* q = nullptr;
  const cudaError_t e = dev_malloc(&q, sizeof(T) * (size_t)room);
  if (e != cudaSuccess) return e;
  if (*p) dev_free(*p);
  *p = (T*)q;
  *cap = room;
  return cudaSuccess;
}
// whether a kernel on device `current` may write to memory of this kind on `device`
// (another GPU's memory only by a copy)
inline bool kernel_reaches(cudaMemoryType type, int device, int current) {
  return type == cudaMemoryTypeManaged || (type == cudaMemoryTypeDevice && device == current);
}
// waits for the device once; while it lives, dev_free on this thread waits no more
struct DevSyncedScope {
  DevSyncedScope();
  ~DevSyncedScope();
};

// process-wide count of kernel launches made by this library (api.cu)
void count_launch();
void count_launches(long long k);  // k launches replayed from a captured graph

// ---- launchers (each enqueues on `st`) -------------------------------------

// validation of the input CSR and points; ctl must be zeroed (first_bad = INT_MAX).
// Without col: offsets and points, and rp[n] into the record after ctl.
cudaError_t launch_check(const int2* xy, const int32_t* rp, const int32_t* col, int32_t n, CheckCtl* ctl,
                         cudaStream_t st);
// coordinates in [0, 2^20) (flag kBadCoord); ctl zeroed with first_bad = INT_MAX
cudaError_t launch_check_points(const int2* xy, int32_t n, CheckCtl* ctl, cudaStream_t st);
// degree requirements 1 <= b_v <= deg(v) - 1 (flag kBadDegreeReq); the
// largest b_v into *bmax (zeroed by the caller)
cudaError_t launch_check_degrees(const int32_t* rp, const int32_t* bdeg, int32_t n, CheckCtl* ctl,
                                 unsigned long long* bmax, cudaStream_t st);
// ec[e] = {col[e], c(row(e), col[e])}
cudaError_t launch_build_ec(const int2* xy, const int32_t* rp, const int32_t* col, int32_t n,
                            int2* ec, cudaStream_t st);
// one persistent cooperative GDP phase; bdeg: degree requirements b_v in
// caller order (NULL: b_v = 2, the fractional 2-matching) -- likewise below
// (bmax: the largest b_v, which picks the selection method)
cudaError_t launch_gdp(const int32_t* rp, const int2* ec, const int32_t* bdeg, int32_t bmax,
                       int32_t* lam0, int32_t* lam1, int32_t n, int32_t F, int32_t shift,
                       int64_t max_sweeps, GdpCtl* ctl, long long* trace_b2,
                       unsigned long long* trace_ch, int64_t trace_cap, long long budget,
                       int num_sms, cudaStream_t st);
// bound2 at lam with fb fractional bits, into *out (zeroed by the launcher)
cudaError_t launch_bound(const int32_t* rp, const int2* ec, const int32_t* bdeg, const int32_t* lam,
                         int32_t n, int32_t fb, long long* out, cudaStream_t st);
// rule (7) extraction; *bad zeroed by the launcher
cudaError_t launch_extract(const int32_t* rp, const int2* ec, const int32_t* bdeg, const int32_t* lam,
                           int32_t n, int32_t fb, uint8_t* x2, unsigned long long* bad,
                           cudaStream_t st);
// lam_out = lam_in >> 1 (F+1 bits -> F bits, floor)
cudaError_t launch_halve(const int32_t* lam_in, int32_t* lam_out, int32_t n, cudaStream_t st);
// all-pairs pricing scan (pricing.cu): pairs (u < v) outside the CSR with z < 0,
// over the points in the renumbered order, in blocks of kPriceBlock positions
constexpr int kPriceBlock = 128;   // positions of a block: the small tile, i and j
constexpr int kPriceLargeI = 512;  // the large tile
constexpr int kPriceLargeJ = 512;
struct PriceCtl {
  unsigned long long count;  // pairs found (past the capacity too)
  unsigned long long listed; // block pairs of the culled scan's list (past its capacity too)
  unsigned int next;         // tile pairs handed out
  unsigned int rows;         // i-points of a scan of some rows
};
struct PriceScan {
  const int2* xy;             // by node
  const int32_t* lam;         // by node, units 2^-fb
  const int32_t* rp;          // the candidate CSR
  const int2* ec;
  const float4* pts;          // by position: {x, y, s (the filter radius), node}
  const float4* box;          // per block of pts: {min x, min y, max x, max y}
  const float* smax;          // and its largest s
  const float4* pts_i;        // the i-points: pts, or some rows gathered
  const float4* box_i;
  const float* smax_i;
  const uint8_t* inU;         // by node: gathered into pts_i (NULL: the i-points are all points)
  const int32_t* seg_off;     // [nseg + 1] positions of the segments
  const int32_t* seg_blk;     // [nseg + 1] their first blocks
  const int32_t* seg_tile;    // [nseg + 1] their first tile pairs (full scan)
  const int2* list;           // block pairs (culled scan)
  int2* pairs;                // the result
  PriceCtl* ctl;
  long long cap;              // of pairs
  int32_t list_cap;
  int32_t nseg, n, fb;
  int32_t split;              // CTAs that share a tile pair (set by the launchers)
};
// room for a list of `listed` block pairs, which the scan hands out by 32-bit
// numbers; 0: too many
inline long long price_list_room(unsigned long long listed) {
  const unsigned long long most = 0x7fffffffull, room = listed + (listed >> 3) + 1024;
  return listed >= most ? 0 : (long long)(room < most ? room : most);
}
// points, blocks and cleared counters of a scan of lambda sc.lam
cudaError_t launch_pricing_prep(const PriceScan& sc, const int32_t* perm, int32_t nblocks, float4* pts, float4* box,
                                float* smax, cudaStream_t st);
// all pairs of the segments' tile pairs, in large tiles or small
bool price_large_tiles(long long large_tiles, int num_sms);
cudaError_t launch_pricing_full(const PriceScan& sc, bool large, long long ntiles, int num_sms, cudaStream_t st);
// the block pairs that can hold a pair with z < 0, then the scan of them
cudaError_t launch_pricing_cull(const PriceScan& sc, const uint8_t* seg_scan, int32_t nblocks, int2* list,
                                cudaStream_t st);
cudaError_t launch_pricing_list(const PriceScan& sc, int num_sms, cudaStream_t st);
// nodes whose lambda rose above lam_ref << shift: flags, their points and
// blocks, their count in sc.ctl->rows; then their scan against all points
cudaError_t launch_pricing_raised(const int32_t* lam_ref, int32_t shift, const PriceScan& sc, uint8_t* inU,
                                  float4* pts_u, float4* box_u, float* smax_u, cudaStream_t st);
cudaError_t launch_pricing_rows(const PriceScan& sc, int num_sms, cudaStream_t st);
// the same scan on the tensor cores (pricing.cu): pts4[v] = {x, y, lambda, node
// perm[v]}; tiles {i0, i1, j0, j1} of at most kMmaTileI x kMmaTileJ positions
cudaError_t launch_pricing_mma_check(long long rounds, unsigned long long seed, unsigned long long* checked,
                                     unsigned long long* mismatches, int32_t* status, cudaStream_t st);
constexpr int kMmaTileI = 128;
constexpr int kMmaTileJ = 128;
cudaError_t launch_pricing_mma_prep(const int2* xy, const int32_t* lam, const int32_t* perm, int32_t n,
                                    int4* pts4, cudaStream_t st);
// ranges [nblocks]: the 128-point blocks; tblk [ntiles]: each tile pair's
// blocks {i-block, j-block, second j-block or -1}; box, lmax, frames: scratch;
// cand [cand_cap]: the filter's candidates (*ncand of them, more than
// cand_cap when the list overflowed: the scan is then incomplete)
cudaError_t launch_pricing_mma_scan(const int4* pts4, const int2* xy, const int32_t* lam, const int32_t* rp,
                                    const int2* ec, int32_t fb, const int4* tiles, const int4* tblk,
                                    int32_t ntiles, const int2* ranges, int32_t nblocks, int4* box, int32_t* lmax,
                                    int4* frames, int2* cand, int64_t cand_cap, unsigned long long* ncand,
                                    int2* pairs, int64_t cap, unsigned long long* count,
                                    int32_t* status, int num_sms, cudaStream_t st);
// CSR union with pairs; sizes: see graph.cu.  Returns the new nnz through *new_nnz_dev.
struct MergeBuffers {
  int32_t* deg;        // [n+1]
  int32_t* tmp_rp;     // [n+1]
  int32_t* tmp_col;    // [nnz + 2*npairs]
  int32_t* new_rp;     // [n+1]
  int32_t* block_sums; // scan scratch
  CheckCtl* ctl;
};
cudaError_t launch_merge_new(const int2* xy, const int32_t* rp, const int2* ec_in, const int2* pairs, int64_t npairs,
                             int32_t n, MergeBuffers& mb, const int32_t* perm, const int32_t* inv, int32_t* isums,
                             int2* ec_out, int32_t* irp, int2* iec, cudaStream_t st);
cudaError_t launch_merge_count(const int32_t* rp, const int2* pairs, int64_t npairs, int32_t n,
                               MergeBuffers& mb, cudaStream_t st);
cudaError_t launch_merge_fill(const int32_t* rp, const int2* ec, const int2* pairs, int64_t npairs,
                              int32_t n, MergeBuffers& mb, cudaStream_t st);
// ec_out: another array than ec_in (untouched rows are copied from ec_in)
cudaError_t launch_merge_finish(const int2* xy, const int32_t* rp, const int2* ec_in, int32_t n,
                                MergeBuffers& mb, int2* ec_out, cudaStream_t st);
// exclusive scan of in[0..m) into out[0..m], out[m] = total (m+1 outputs)
cudaError_t launch_scan(const int32_t* in, int32_t* out, int32_t m, int32_t* block_sums,
                        cudaStream_t st);
size_t scan_scratch_ints(int32_t m);
// split ec into col / cost arrays
cudaError_t launch_split_ec(const int2* ec, int64_t nnz, int32_t* col, int32_t* cost,
                            cudaStream_t st);

// ---- class-by-class GDP (gdp_classes.cu) ------------------------------------------
// greedy colouring of the caller-order CSR and the nodes grouped by class
struct ClassPlan {
  int32_t* color = nullptr;      // [n] colour of each node
  int32_t* order = nullptr;      // [n] nodes grouped by class
  int32_t* off = nullptr;        // [ncolors+1] class offsets into order
  unsigned int* ctl = nullptr;   // round counters
  int32_t cap = 0;
  int32_t ncolors = 0;
  int32_t rounds = 0;            // Jones-Plassmann rounds of the last colouring
  int64_t version = -1;          // GdpPlan::version of the graph coloured
  std::vector<int32_t> h_off;
};
cudaError_t color_classes(const int32_t* rp, const int2* ec, int32_t n, ClassPlan& cp,
                          cudaStream_t st);
void class_plan_free(ClassPlan& cp);
// one class-by-class phase, lambda updated in place (bdeg / bmax as launch_gdp)
cudaError_t launch_gdp_classes(const int32_t* rp, const int2* ec, const int32_t* bdeg, int32_t bmax,
                               int32_t* lam, const ClassPlan& cp, int32_t n, int32_t F,
                               int32_t shift, int64_t max_sweeps, GdpCtl* ctl, long long* trace_b2,
                               unsigned long long* trace_ch, int64_t trace_cap, long long budget,
                               int num_sms, cudaStream_t st);

// ---- spatial renumbering and the CSR in that order (plan.cu) --------------------
struct GdpPlan {
  int32_t n = 0;
  int64_t nnz = 0;               // entries of the internal CSR
  int64_t version = 0;           // bumped whenever the internal CSR is rebuilt
  int32_t* perm = nullptr;       // internal -> caller node
  int32_t* inv = nullptr;        // caller -> internal node
  int32_t* irp = nullptr;        // internal CSR offsets
  int2* iec = nullptr;           // internal {col, cost}
  int32_t* ilam[2] = {nullptr, nullptr};  // lambda in internal order
  uint64_t* keys = nullptr;
  uint64_t* keys2 = nullptr;
  int32_t* idx = nullptr;
  void* sort_tmp = nullptr;
  int32_t* scan_tmp = nullptr;
  int64_t irp_cap = 0, iec_cap = 0, scan_cap = 0;
  int64_t ilam_cap[2] = {0, 0};
};
cudaError_t sort_pairs_u64(void* temp, size_t& temp_bytes, const uint64_t* keys_in,
                           uint64_t* keys_out, const int32_t* vals_in, int32_t* vals_out,
                           int32_t count, int end_bit, cudaStream_t st);
// Morton renumbering inside each segment [seg_off[s], seg_off[s+1]) (segments stay contiguous)
cudaError_t plan_renumber(const int2* xy, int32_t n, const std::vector<int32_t>& seg_off, GdpPlan& p,
                          cudaStream_t st);
// merge of npairs pairs that are distinct and outside the CSR, into ec_out, mb.new_rp and the
// renumbered CSR of `nnz` = old entries + 2 npairs (MergeBuffers: above)
cudaError_t plan_merge(const int2* xy, const int32_t* rp, const int2* ec_in, const int2* pairs, int64_t npairs,
                       int32_t n, int64_t nnz, MergeBuffers& mb, int2* ec_out, GdpPlan& p, cudaStream_t st);
// the CSR in the renumbered order
// room for a graph of nnz entries (the arrays stay as they are where there is none)
cudaError_t plan_room(int32_t n, int64_t nnz, GdpPlan& p);
cudaError_t plan_build(const int32_t* rp, const int2* ec, int32_t n, int64_t nnz, GdpPlan& p, cudaStream_t st);
// dst[i] = src[perm[i]]  /  dst[perm[i]] = src[i]
cudaError_t gather_perm(const int32_t* src, const int32_t* perm, int32_t n, int32_t* dst,
                        cudaStream_t st);
cudaError_t scatter_perm(const int32_t* src, const int32_t* perm, int32_t n, int32_t* dst,
                         cudaStream_t st);
void plan_free(GdpPlan& p);
// ---- GDP on shared-memory tiles (gdp_ring.cu) --------------------------------------
constexpr int kRingMax = 4;          // rings around a tile: sweeps per exchange (ring_sweeps asks for no more)
constexpr int kRingLocals = 8192;    // nodes a tile knows (own, rings, two padding slots)
constexpr int kRingHalo = 4096;      // of them in rings
constexpr int kRingDepth = 1536;     // entries of a row at most: 32 such rows are all that a tile can hold
// A slice with a row of more than kRingLong entries leaves all but the first
// kRingTail of each of its rows to the warp (where lanes and warp cost the same: rows
// of 100 entries 405 against 416 us for 128 sweeps, of 66 301 against 400, of 256 826
// against 355)
constexpr int kRingLong = 112;
constexpr int kRingTail = 32;
constexpr int kRingSlots = 8192;     // rows it computes, in whole slices
constexpr int kRingSlices = kRingSlots / 32;
constexpr int kRingSweeps = 1 << 30;  // of one launch (a longer phase takes several)
constexpr int kRingRing = 16;        // rounds whose stop-test slots are live
constexpr int kRingBadSize = 1;      // RingStats::bad: some tile is too large,
constexpr int kRingBadRoom = 2;      // or has more sliced entries than the arrays have room for
struct RingTile {
  int32_t seg, j, count;  // the j-th of the count tiles of an instance (segment)
};
struct RingHdr {
  int32_t lo, own;        // first own node (internal), own nodes
  int32_t halo;           // nodes of all rings
  int32_t seg, count, first;
  int32_t word0;          // its first word in the exchange
  int32_t nsl, nent;      // slices, sliced entries
  int32_t sec_end[kRingMax];  // slices of own rows, and of those of rings 1 .. k
};
struct RingStats {        // over all tiles of a plan
  int32_t bytes8, bytes4;  // shared memory of the largest with 8- and 4-byte entries there,
  int32_t bytes_reg;       // and with entries in registers
  int32_t slices, locals, maxcost;
  int32_t longs;           // some row has more than kRingLong entries
  int32_t bad;
};
struct RingSeg {          // per instance, zeroed per phase
  unsigned long long slot[kRingRing];
  unsigned int ovf[kRingRing];
  long long sweeps;       // the result
  int32_t fixed_point, overflow;
  int32_t unfit;          // (batches) one of its tiles is past the form's limits: none of them runs
};
struct RingLimit {        // of a form, per tile (batches; smem 0: none)
  int32_t smem, slices, locals, cost;
};
struct RingRecord {       // what the host reads after a phase, in one copy
  RingStats stats;        // zeroed per plan
  int32_t status;         // from here on zeroed per phase
  RingSeg seg[1];         // one per instance
};
struct RingArgs {
  const RingHdr* hdr;
  const int32_t* halo;
  const uint16_t* order;
  const uint32_t* slc;
  const uint32_t* longs;   // per slice with a row of more than kRingLong entries: those past kRingTail
  const int2* ent;
  const RingStats* stats;
  const int32_t* pos;      // by internal node: its word
  RingSeg* seg;
  unsigned* words[2];
  int* status;
  const int32_t* lam_in;   // caller order; lam_out must be another array
  int32_t* lam_out;
  const int32_t* perm;
  const int32_t* bint;     // b_v in internal order (NULL: 2)
  long long* trace_b2;     // zeroed
  unsigned long long* trace_ch;
  long long trace_cap, budget;
  int32_t max_sweeps;      // at most kRingSweeps
  int32_t K, F, shift, ecap, smem;
};
struct RingPlan {
  int64_t version = -1;    // GdpPlan::version it was built from
  int32_t tiles = 0, K = 0, F = 0, ecap = 0;
  RingHdr* hdr = nullptr;
  int32_t* halo = nullptr;
  uint16_t* order = nullptr;
  uint32_t* slc = nullptr;
  uint32_t* longs = nullptr;
  int2* ent = nullptr;
  RingRecord* rec = nullptr;
  int32_t* pos = nullptr;
  unsigned* words = nullptr;  // the exchange: two buffers of words_n
  int64_t words_n = 0;
  int64_t hdr_cap = 0, halo_cap = 0, order_cap = 0, slc_cap = 0, longs_cap = 0, ent_cap = 0, seg_cap = 0, words_cap = 0, pos_cap = 0;
};
void ring_free(RingPlan& p);
// the tiles of K rings over the internal CSR: `tiles` equal shares of the one
// segment's nodes (list NULL), or those of the device list; seg_off on the device;
// first: of the phase's tiles, where these are some of them (their arrays have room
// for `room` tiles, and `first` sets their words apart from the others')
// maxdeg: the longest row a tile takes, at most kRingDepth; entries_per_tile: their
// mean (a tile's room is what near-even tiles need), -1: the most a tile can hold
cudaError_t ring_build(const GdpPlan& g, const int32_t* seg_off, const RingTile* list, int32_t tiles, int32_t K,
                       int32_t F, int64_t entries_per_tile, int32_t maxdeg, int32_t nseg, RingPlan& p, cudaStream_t st,
                       const RingLimit& limit = RingLimit{}, int32_t first = 0, int32_t room = 0);
RingLimit ring_pair_limit();  // of kRingPair
int32_t ring_smem(bool half, bool traced);  // dynamic shared memory of a CTA
// per phase: cleared segment records and status; with limits before ring_build, which
// flags the instances past them
cudaError_t ring_start(RingPlan& p, int32_t n, int32_t tiles, int32_t nseg, cudaStream_t st);
// whether tiles of n nodes and nnz entries in all might fit some form
inline bool ring_can_fit(int64_t n, int64_t nnz, int64_t tiles, int64_t smem, bool half) {
  const int64_t own = (n + tiles - 1) / tiles;
  if (own + 34 > kRingLocals) return false;
  return (!half && own <= 62 * 32) || 4 * (nnz / tiles) + 10 * own <= smem;
}
// Where the rows' entries are kept: registers (1 or 2 rows a thread, up to 1,984
// rows a tile), registers with two CTAs per SM (up to 960 rows a tile, b_v = 2),
// shared memory, or shared memory with two CTAs per SM.
enum RingForm { kRingHalf = -1, kRingSmem = 0, kRingReg1 = 1, kRingReg2 = 2, kRingPair = 3 };
int ring_reg_rows(const RingStats& st);  // rows a thread of the register form (0: does not fit)
// (longs: the register form for graphs with rows past kRingLong entries, b_v = 2)
// one cooperative launch over the plan's tiles: whole instances
cudaError_t launch_gdp_ring(const GdpPlan& g, RingPlan& p, int32_t tiles, const int32_t* lam_in,
                            int32_t* lam_out, int32_t shift, int32_t max_sweeps, long long* trace_b2,
                            unsigned long long* trace_ch, int64_t trace_cap, long long budget, const int32_t* bint,
                            int32_t bmax, RingForm form, bool longs, cudaStream_t st);

// ---- exact finisher (finisher_prep.cu on the device, finisher.cpp on the host) ---
// twin[e] for every internal entry; *missing (zeroed by the caller) counts
// entries without a reverse entry
cudaError_t fin_build_twin(const GdpPlan& p, int32_t* twin, unsigned long long* missing, cudaStream_t st);
// bdeg_caller: degree requirements in caller order (NULL: 2)
cudaError_t fin_prepare(const GdpPlan& p, const int32_t* lam_caller, const int32_t* bdeg_caller,
                        int32_t F, int32_t* lam_int, uint8_t* y, int32_t* exl, cudaStream_t st);
// x (half units, caller order) = y[e] + y[twin[e]] of the final flow; lambda
// at F+1 bits to caller order.  include (device, per segment; NULL = all): x
// of excluded segments is kept
cudaError_t fin_scatter(const GdpPlan& p, const int32_t* rp, const uint8_t* y_int,
                        const int32_t* twin, const int32_t* lam2_int, uint8_t* x_out,
                        int32_t* lam2_out, const int32_t* seg_off, int32_t nseg,
                        const uint8_t* include, cudaStream_t st);
// ---- batched GDP on thread-block clusters (gdp_cluster.cu) ------------------------
struct ClusterInst {
  int32_t node0;  // first internal node of the instance
  int32_t n;      // its nodes
  int32_t per;    // nodes per CTA (the last CTAs may hold fewer, or none)
  int32_t seg;    // instance id
};
struct ClusterOut {
  long long sweeps;
  int status;     // kGdpOverflow bit
  int fixed;      // 1 if the last sweep changed nothing
};
constexpr int kClusterNodes = 2048;      // most nodes one CTA holds
constexpr int kClusterEntries = 24000;   // most entries one CTA holds
size_t cluster_smem(int32_t emax, int32_t nmax);
// pk[e] = {owner rank << 16 | local index, cost << F} for the listed instances' entries
cudaError_t cluster_pack(const int32_t* irp, const int2* iec, const ClusterInst* d_insts, int32_t ninst,
                         int32_t F, int2* pk, cudaStream_t st);
// one cluster of C CTAs per listed instance; ilam (internal order) in and out; out zeroed
cudaError_t launch_gdp_cluster(int32_t C, int32_t threads, const int32_t* irp, const int2* pk,
                               const ClusterInst* d_insts, int32_t ninst, int32_t* ilam,
                               int32_t shift, int64_t max_sweeps, ClusterOut* out,
                               int32_t emax, int32_t nmax, cudaStream_t st);
// clusters of this shape that fit on the device at once (0: none)
int32_t cluster_max_smem_ok(int32_t C, int32_t threads, int32_t emax, int32_t nmax);

// ---- batched solver (batch_kernels.cu) --------------------------------------------
// Parameters of one launch of a batched GDP kernel, read from device memory so
// that a captured launch can be replayed with new values.
struct BatchChunk {
  int32_t ntiles;        // tiles in the list (those of the instances still active)
  int32_t pad;
  long long t_base;      // sweeps run by earlier launches of this phase
  long long max_sweeps;  // sweeps this launch may run
};
// tiles {first node, end node, segment, first entry} over the renumbered CSR
// with their end entries in tiles_e1; one cooperative launch of G CTAs of the
// given shape (see batch_kernels.cu); max_tiles sizes the per-CTA tile table
int batch_num_shapes();
// lambda of the buffer a batch GDP phase ended in, scattered to caller order
cudaError_t launch_batch_scatter_final(const int32_t* lam0, const int32_t* lam1, const GdpCtl* ctl,
                                       const int32_t* perm, int32_t n, int32_t* dst, cudaStream_t st);
int batch_shape_blocks(int shape, int mcap);  // CTAs per SM, 0 if the shape does not run
int batch_shape_tile(int shape, int* te, int* tn);  // tile entries and nodes of a shape
int batch_shape_units(int shape);  // tile owners per CTA: 1 (CTA form) or its warps (warp form)
cudaError_t launch_gdp_batch(int shape, const int32_t* irp, const int2* iec, const int4* tiles,
                             const int32_t* tiles_e1, const BatchChunk* chunk, int32_t max_tiles, int32_t G,
                             int32_t nseg, uint8_t* active, unsigned long long* seg_ch, long long* seg_sweeps,
                             int32_t* lam0, int32_t* lam1, int32_t F, int32_t shift, GdpCtl* ctl,
                             long long budget, cudaStream_t st);
cudaError_t launch_batch_extract_bound(const int32_t* rp, const int2* ec, const int32_t* lam,
                                       int32_t n, int32_t fb, const int32_t* seg_off, int32_t nseg,
                                       uint8_t* x2, long long* seg_b2, unsigned long long* seg_bad,
                                       const uint8_t* seg_write, cudaStream_t st);
cudaError_t launch_batch_union(const int32_t* rp_local, const int32_t* col_local,
                               const int32_t* seg_off, const int32_t* eoff, int32_t nseg, int32_t n,
                               int64_t nnz, int32_t* rp, int32_t* col, CheckCtl* ctl,
                               cudaStream_t st);
cudaError_t launch_batch_mask_surplus(int32_t* exl, const int32_t* seg_off, int32_t nseg,
                                      const uint8_t* include, int32_t n, cudaStream_t st);
// out[s] = rp[seg_off[s]], s = 0..nseg
cudaError_t launch_batch_seg_entry(const int32_t* rp, const int32_t* seg_off, int32_t nseg, int32_t* out,
                                   cudaStream_t st);
// results of the instances flagged in done (device mask) into the arenas, entries at eoff[s]
cudaError_t launch_batch_snapshot(const uint8_t* done, const int32_t* seg_off, int32_t nseg, const int32_t* rp,
                                  const int32_t* lam, const int2* ec, const uint8_t* x2, const long long* eoff,
                                  int32_t* res_lam, int32_t* res_rp, int2* res_ec, uint8_t* res_x2,
                                  cudaStream_t st);

struct FinisherWork;
FinisherWork* finisher_work_new();
// lets up to `threads` - 1 worker threads of the host finisher poll for a job
// that is about to come (a finisher call after some device work), so that the
// call does not wait for them to wake
void finisher_pool_wake(int32_t threads);
void finisher_work_reserve(FinisherWork* w, int32_t n);  // host work arrays for n nodes
FinisherWork* finisher_work_take(int32_t n);  // with room for n nodes, from the cache if it has one
void finisher_work_free(FinisherWork* w);     // back to the cache
// copies between host arrays, on the finisher's worker threads when they are idle
struct HostCopy {
  void* dst;
  const void* src;
  size_t bytes;
};
void host_copy(const std::vector<HostCopy>& parts);
// pinned host blocks from a bounded cache (api.cu)
cudaError_t pin_alloc(void** p, size_t bytes);
void pin_free(void* p);
// Min-cost flow on the bipartite double cover, internal node order; see
// finisher.cpp.  y is the initial flow (updated to the optimal one), exl the
// left surpluses, lam2 receives pi(L) - pi(R) (F+1 bits).  Blocks and segments
// [seg_off[s], seg_off[s+1]) go to up to `threads` host threads; with include
// (per segment; NULL = all) the other segments are neither read nor written.
// Returns 0 ok, 7 infeasible, 5 overflow.
// time and augmentations of the finisher, summed over its calls
struct FinisherStats {
  double ms_prep = 0, ms_phase[3] = {0, 0, 0}, ms_scatter = 0;
  int64_t aug[3] = {0, 0, 0};
  int32_t threads = 0;
  int32_t phase1_gpu = 0;  // 1 if phase 1 ran on the GPU
};
// ext_pi / ext_ex (NULL: none): potentials [2n] and surpluses [2n] that phase
// 1 left when it ran on the GPU; the host then runs phases 2 and 3 only (the
// augmentations it reports are its own)
int host_finisher(int32_t n, const int32_t* irp, const int2* iec, const int32_t* twin, uint8_t* y,
                  const int32_t* exl, const int32_t* lam, int32_t F, int32_t* lam2,
                  const int32_t* seg_off, int32_t nseg, const uint8_t* include, int32_t threads,
                  int64_t* augmentations, FinisherWork* w, FinisherStats* stats, int64_t* ext_pi = nullptr,
                  int32_t* ext_ex = nullptr);
// the finisher's phase 1 on the GPU (finisher_gpu.cu): one warp per block
size_t fin_heap_item_bytes();
cudaError_t launch_fin_block_caps(const int2* blocks, int32_t nblocks, const int32_t* irp, long long* caps,
                                  cudaStream_t st);
cudaError_t launch_fin_blocks(int32_t n, const int2* blocks, int32_t nblocks, const int32_t* irp, const int2* iec,
                              const int32_t* twin, uint8_t* y, const int32_t* exl, const int32_t* lam, int32_t F,
                              long long* pi, long long* dist, int32_t* excess, int32_t* via, int32_t* pred,
                              uint32_t* reached, uint32_t* closed, void* heaps, const long long* heap_off,
                              int32_t* orders, long long* pushes, int32_t* status, long long budget,
                              cudaStream_t st);
constexpr int32_t kFinBlockNodes = 2048;  // nodes per block of the finisher's phase 1 (host and GPU)
// lam_out = 2 * lam_in (F bits -> F+1 bits)
cudaError_t launch_double(const int32_t* lam_in, int32_t* lam_out, int32_t n, cudaStream_t st);


// ---- k nearest neighbours and warm-start features (knn.cu) -------------------------
constexpr int kKnnMax = 32;    // largest k of the k-NN kernel
constexpr int kFeatures = 16;  // neighbour distances per node in the warm-start features
// exact k-NN lists (ties by index): nbr [n][k], d2 [n][k] (may be NULL); device
// pointers.  All three synchronise: their work space goes back to the cache.
cudaError_t knn_device(const int2* d_xy, int32_t n, int32_t k, int32_t* d_nbr, long long* d_d2,
                       cudaStream_t st);
// symmetrised k-NN CSR; d_col holds up to 2 n k entries; *nnz_out on the host
cudaError_t knn_csr_device(const int2* d_xy, int32_t n, int32_t k, int32_t* d_row_ptr, int32_t* d_col,
                           int64_t* nnz_out, cudaStream_t st);
// feat [n][16] = sorted 16-NN distances / s, s = max(1, their mean)
cudaError_t features_device(const int2* d_xy, int32_t n, float* d_feat, float* d_scale, cudaStream_t st);

// ---- warm-start network (mlp.cu) ----------------------------------------------------
// flat fp32 parameters: W1 [128][16], b1 [128], W2 [128][128], b2 [128], w3 [128], b3
constexpr int kOW1 = 0, kOb1 = 2048, kOW2 = 2176, kOb2 = 18560, kOw3 = 18688, kOb3 = 18816;
constexpr int kMlpParams = 18817;
constexpr int kImgW1Bytes = 128 * 16 * 2;   // bf16 operand image of W1
constexpr int kImgW2Bytes = 128 * 128 * 2;  // bf16 operand image of W2 (and of W2^T)
constexpr int kMlpImgBytes = kImgW1Bytes + 2 * kImgW2Bytes;
constexpr int kLambda0Limit = 1 << 27;      // |lambda0| clamp of the warm start
struct MlpAdam {
  float lr, beta1, beta2, eps, lr_final_frac;
  long long total_steps;  // linear decay of lr to lr * lr_final_frac over this many steps
  long long log_base;     // the loss of step t goes to loss_log[t - 1 - log_base]
};
cudaError_t mlp_pack(const float* master, uint8_t* img, cudaStream_t st);
int mlp_grid(int num_sms, long long count);
cudaError_t mlp_forward(const uint8_t* img, const float* master, const float* feat, long long count,
                        float* y, const float* scale, int32_t* lam, int32_t F, int num_sms, int* status,
                        cudaStream_t st);
cudaError_t mlp_train_launch(const uint8_t* img, const float* master, const float* feat, const float* target,
                             const int32_t* perm, long long s0, long long count, float two_over_b,
                             float* partial, int grid, long long* step_ctr, int* status, cudaStream_t st);
cudaError_t mlp_reduce_launch(const float* partial, int nparts, float* grad, float* master, float* m1,
                              float* m2, uint8_t* img, const long long* step_ctr, const MlpAdam& hp,
                              float* loss_log, cudaStream_t st);
cudaError_t mlp_perm_keys(uint64_t key, long long n, uint64_t* keys, int32_t* idx, cudaStream_t st);
}  // namespace f2m
