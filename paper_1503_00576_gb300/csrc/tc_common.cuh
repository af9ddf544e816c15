// tc_common.cuh -- definitions shared by the library's CUDA translation units.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace tc {

// Device-side error bits (Ctrl::err).
enum : uint32_t { kErrIdRange = 1u, kErrTimeout = 2u, kErrInternal = 4u };

// Upper bound on iterations of any spin-wait in a kernel.  Every wait in this
// library is on a predecessor tile that is already resident (tiles are handed
// out in launch order through an atomic ticket), so the bound is a safety
// net: if it is ever reached the kernel records kErrTimeout, stops waiting
// and the host reports TC_ERR_TIMEOUT.  What a timed-out tile would have
// written is not trusted: the tile publishes a poisoned status instead of its
// prefix and writes nothing, every tile that reads a poisoned status does the
// same, and every later kernel of the call returns at entry once kErrTimeout
// is set (see aborted()), so no kernel runs on incomplete data.
constexpr uint32_t kSpinLimit = 1u << 24;
constexpr uint32_t kNoTile = 0xffffffffu;  // no tile withholds its status (see set_wait_hooks)

// Sorted forward lists (the padded column array col4).  Lists of up to 2
// kWarpSortMax entries are sorted by one warp, up to kCtaSortMax by a CTA in
// shared memory; longer ones (never met in the workloads: they need a dense
// core of more than 8192 vertices) by a CTA in sorted chunks of kCtaSortMax
// merged in global memory.  Every list is sorted, and repeated entries (an
// edge given more than once) are dropped there.
constexpr int kWarpSortMax = 512;
constexpr int kCtaSortMax = 8192;
// Group keys carry, above the 2b bits of h and l, the number of leading
// 32-byte blocks of the streamed list that the intersection skips; there is
// room for it when 2b <= kSkipShift.
constexpr int kSkipShift = 48;
// Skip value of an edge whose triangles the dense hub block counts: the
// streamed list is skipped whole.
constexpr uint32_t kSkipAll = 0xFFFFu;

// Bitmaps of the top ranks (bits.cu): kBitCols columns; a list has one if at
// least kBitMinBlocks of its 32-byte blocks lie among them, a group uses them
// if it has at least kBitMinPartners partners.  A list's record is (slot + 1)
// << kBitTbBits | tb, tb the first block that the bitmap stands for; 0: none.
// Per vertex (PV) an edge costs about three times as much (counts per column
// and partner), so the lines lie higher there.  R-MAT 20 of 44.5M pairs / 21 of
// 91M / 24 of 180M / 22 of 180M, whole calls in ms:
//   T only      4 blocks 7.16 15.63 31.19 37.55   8 partners 7.08 15.50 30.15 37.11
//               6        7.05 15.50 30.16 37.12  16          (the same call)
//               8        7.05 15.58 30.10 37.03  32          7.06 15.50 30.15 37.13
//   per vertex  8        8.67 20.20 37.26 47.45  32          8.72 20.13 37.12 47.28
//              12        8.70 20.09 37.11 47.33  64          (the same call)
//              16        8.77 20.17 36.89 47.30 128          8.71 20.08 37.08 47.36
// so only fewer blocks than 6 cost anything; 8192 columns instead of 4096 cost
// 10% more per call for 4% more of the lookups.
constexpr int kBitCols = 4096;
template <bool PV> constexpr int kBitMinBlocks = PV ? 12 : 6;
template <bool PV> constexpr int kBitMinPartners = PV ? 64 : 16;
// Partners that a warp intersects at a time.  With per-vertex counts the bit
// planes hold 255, and emptying them costs the same for any number.
template <bool PV> constexpr uint32_t kBitRange = PV ? 248u : 128u;
constexpr int kBitTbBits = 11;
constexpr uint32_t kBitTbMask = (1u << kBitTbBits) - 1;
constexpr uint32_t kBitMaxSlots = (1u << (32 - kBitTbBits)) - 1;
// Only for single graphs of at least this many pairs.  T only: below it few
// lists are that long, and two launches cost more (R-MAT 16 of 2.5M pairs,
// without / with them when they came: 0.64 / 0.61 ms, 21 of 91M 22.5 / 16.9).
// Per vertex, without / with them: R-MAT 18 of 4M pairs 0.88 / 0.93 ms, of 10.5M
// 2.14 / 2.14, 20 of 16.8M with repeats 3.01 / 3.18, of 25M 4.94 / 4.77, of 33M
// 7.12 / 6.21, of 44.5M 10.7 / 8.69, 21 of 91M 26.1 / 20.2, 24 of 180M 38.5 /
// 37.2, 22 of 180M 62.9 / 47.3: where they pay depends on the density, and the
// line lies where they do on all of these.
template <bool PV> constexpr int64_t kBitMinPairs = PV ? 1 << 25 : 1 << 18;

// Counting sorts by atomics (direct.cu) instead of radix passes: runs of at
// most this many pairs (a single graph; a batch, an engine by its capacity) with
// ids of at most 24 bits, but for shares of a run (their dealing needs the exact
// vertex order).  Whole calls, radix passes / counting sorts: 19,900 pairs 0.15 /
// 0.11 ms, 320,000 0.20 / 0.14; uniform of 8M 1.35 / 1.06 ms, of 24M 3.65 / 3.30,
// of 32M 4.81 / 4.67, of 50M 7.46 / 7.80; Barabasi-Albert of 12M 1.75 / 1.53, of
// 24M 3.29 / 3.07, of 32M 4.32 / 4.18; R-MAT 20 of 16M 2.52 / 2.45, of 32M 4.90 /
// 4.70, of 44M 6.97 / 6.89 (per vertex 8.57 / 8.61); ring lattice of 32M 3.00 /
// 2.81, of 50M 4.52 / 4.77; geometric of 24M 3.04 / 2.71, of 32M 4.01 / 3.84, of
// 67M 8.16 / 8.97 (the scattered writes leave L2).  So the two cross between 32M
// and 50M pairs; the line for single graphs was drawn before the kernels behind
// it changed, when Barabasi-Albert of 32M took 4.42 / 4.72 ms.  Batches: 300
// graphs of 3.3M pairs 0.75 / 0.54 ms, 64 of 33M 4.55 / 4.21, 30 of 42M 5.84 /
// 5.69, 76 of 48M 6.46 / 6.25, 96 of 62.5M 8.26 / 8.27, 128 of 72M 9.54 / 9.70,
// 1500 of 66M 9.04 / 8.48: the line lies below where they cross, too.
constexpr int64_t kDirectMaxPairs = 20ll << 20;
constexpr int64_t kDirectMaxBatchPairs = 1ll << 25;
// ... but for runs of more than kCrowdedPairs pairs with more than kCrowdedMean
// of them per vertex, mostly pairs given many times: their counters share so few
// L2 sectors that the places taken from them cost more than the passes (m/n the
// mean): K_200 x 200 (20,000) 2.94 / 3.86 ms, K_1000 x 8 (4,000) 1.11 / 1.49,
// K_2000 x 8 (8,000) 2.68 / 3.76, 20,000 edges x 200 (2,000) 0.98 / 1.11 ms,
// 160,000 x 100 (1,000) 1.66 / 1.83; 6,000 x 66 (660) 0.36 / 0.34, 80,000 x 50
// (500) 0.50 / 0.48, 320,000 x 50 (500) 1.25 / 1.24, 99,840 pairs of 64 vertices
// (1,560) 0.22 / 0.21 ms.
constexpr int64_t kCrowdedPairs = 1 << 18;
constexpr int64_t kCrowdedMean = 768;
constexpr int kRankClasses = 1024;
// Runs whose kernels are launched early (see launch()).  Whole calls, in turn /
// early: 8,191 pairs 135 / 85 us, 131,072 with clustering 259 / 198 us, R-MAT
// 16 of 2.5M 541 / 469 us, R-MAT 18 of 10.5M 2.03 / 1.96 ms; R-MAT 20 of 16.8M
// 3.13 / 3.22 ms, 21 of 91M 15.5 / 18.6 ms, 24 of 180M 38.2 / 43.4 ms.
constexpr int64_t kEarlyMaxPairs = 12ll << 20;
constexpr uint64_t kHole = ~0ull;            // no edge (dropped pair or edge)
constexpr uint64_t kOwnEdge = 1ull << 63;    // emitted edge of its owner's group

// Dense hub block (hub.cu): the kHubSize vertices of highest rank, counted
// on the tensor cores when they hold at least kHubMinEdges edges.  Only for
// single graphs with n >= kHubMinVertices and ids of at most 24 bits (the
// group keys must carry the skips).
constexpr int32_t kHubSize = 1 << 14;     // default size of the hub set
constexpr int32_t kHubMaxSize = 1 << 15;  // largest allowed (a multiple of 128)
constexpr int32_t kHubMinVertices = 1 << 17;
constexpr int64_t kHubMinEdges = 1 << 21;

constexpr int kMaxSort2Passes = 4;  // 31 owner bits / 8-bit digits
constexpr int kMaxRankPasses = 4;   // 31 degree bits / 8-bit digits
constexpr int kMaxGroupPasses = 4;  // 31 group bits / 8-bit digits
constexpr int kMaxPasses = kMaxSort2Passes + kMaxRankPasses + kMaxGroupPasses;
// First histogram slot of each sort.
constexpr int kSort2Slot = 0;
constexpr int kRankSlot = kMaxSort2Passes;
constexpr int kGroupSlot = kMaxSort2Passes + kMaxRankPasses;

// Hub sets of the work instrumentation: the 2^(kHubLog2Min + i) highest
// ranks, i < kHubSizes.
constexpr int kHubSizes = 4;
constexpr int kHubLog2Min = 12;

// Control block: zeroed at the start of every call.
struct Ctrl {
  uint32_t err;                    // kErr* bits
  uint32_t m;                      // oriented edges: set by orient (repeats included), then,
                                   //   if any list held repeats, by the recount of its node array
  uint32_t tile_ticket[24];        // per look-back kernel: next tile to hand out
  uint32_t n_warp_groups;          // partner groups counted by one warp each
  uint32_t n_cta_groups;           // ... by a 256-thread CTA each
  uint32_t n_big_groups;           // ... by a 512-thread CTA with a large table
  uint32_t next_warp_group;        // work cursors of the counting kernels
  uint32_t next_cta_group;
  uint32_t next_big_group;
  unsigned long long total;        // triangle count T
  uint32_t m_in;                   // input pairs that are real (not batch padding)
  uint32_t n_part;                 // partners of all groups (set by the group scan)
  uint32_t n_warp_lists;           // queued forward lists: sorted by one warp each
  uint32_t n_cta_lists;            // ... by a CTA each
  uint32_t next_warp_list;         // work cursors of the queued lists
  uint32_t next_cta_list;
  uint32_t n_bit_items;            // work items of the bitmap path
  uint32_t pad_;
  uint32_t hub_on;                 // the hub block is counted densely (hub.cu)
  uint32_t hub_lo;                 // its first rank
  uint32_t hub_size;               // its number of vertices (hub_lo + hub_size = n)
  uint32_t dups;                   // some forward list held a repeated edge (set by the list sort)
  unsigned long long hub_triangles;  // triangles the dense block counted
  unsigned long long hub_est[4];   // hash lookups inside each candidate hub set (hub.cu)
  // work of the counting phase (filled only when asked for; see launch_work and
  // launch_run_work):
  // hash lookups, hash inserts, merge work W, max out-degree, then the
  // lookups of edges with both endpoints among the 2^12 .. 2^15 top ranks
  unsigned long long work[4 + kHubSizes];
};
static_assert(sizeof(Ctrl) % 16 == 0, "Ctrl must keep 16-byte alignment");

// Ticket slots in Ctrl::tile_ticket.
enum {
  kTicketSort = 0 /* .. kMaxPasses-1, one per radix pass */,
  kTicketOrient = kMaxPasses,
  kTicketScan = kMaxPasses + 1,
  kTicketGroupScan = kMaxPasses + 2,
  kTicketRecount = kMaxPasses + 3
};
static_assert(kTicketRecount < 24, "ticket slots");

// Look-back status words: value in the low 62 bits, flag in the top 2.
constexpr unsigned long long kFlagAggregate = 1ull << 62;
constexpr unsigned long long kFlagInclusive = 2ull << 62;
constexpr unsigned long long kFlagPoison = 3ull << 62;  // the tile gave up: its prefix is unknown
constexpr unsigned long long kValueMask = (1ull << 62) - 1;

#ifdef __CUDACC__
// True once some kernel of this call has recorded a wait that ran out: the
// data it left behind is incomplete, so later kernels must not read it.  A
// plain load: what an earlier kernel recorded is seen, and the threads of an
// SM share one L1 line (a volatile load per thread, 300,000 of them on one
// L2 word, made a kernel that had nothing to do last 6 us instead of 2).
__device__ __forceinline__ bool aborted(const Ctrl *ctrl) {
  return (ctrl->err & kErrTimeout) != 0u;
}

// The stream of a partner whose list has record ld, from its first block that
// can meet the hashed list on (the `skip` leading blocks cannot): {first col4
// word, entries (d+ <= sqrt(2m) < 2^16) in the low half; in the high half the
// entries left to the hash path when the group's list has a bitmap and this
// one's takes over (0xffff: it does not)}.
__device__ __forceinline__ int2 stream_desc(int2 ld, int32_t skip, uint32_t cut) {
  return make_int2(ld.x + 2 * skip, (int32_t)((uint32_t)max(ld.y - 8 * skip, 0) | cut << 16));
}

// Whether a group of np partners whose list has bitmap record rec (0: none)
// intersects by bitmaps.
template <bool PV>
__device__ __forceinline__ bool bits_group(uint32_t rec, int32_t np) {
  return rec != 0u && np >= kBitMinPartners<PV>;
}

// Whether a partner whose list of len entries has bitmap record rec (0: none)
// and skips its first `skip` blocks is intersected by bitmaps from block tb
// on (if the group's list has a bitmap too): enough blocks must be left there.
template <bool PV>
__device__ __forceinline__ bool bits_used(uint32_t rec, int32_t skip, int32_t len) {
  if (rec == 0u || skip == (int32_t)kSkipAll) return false;
  return ((len + 7) >> 3) - max(skip, (int32_t)(rec & kBitTbMask)) >= kBitMinBlocks<PV>;
}

#endif

// Partner groups whose hashed forward list has at most kWarpMaxRow entries
// are counted by one warp, up to kCtaMaxRow by a 256-thread CTA, and longer
// ones by a 512-thread CTA with a larger table.
constexpr int kWarpMaxRow = 128;
constexpr int kWarpMaxPartners = 64;
constexpr int kCtaMaxRow = 1024;

// Runtime tuning of the counting layout (what an autotuner varies).
struct Tuning {
  int32_t warp_max_list;      // a group goes to one warp if its hashed list has
  int32_t warp_max_partners;  //   at most this many entries and partners
  int32_t heavy_ratio_pct;    // edge (u,v) is grouped at v when |N+(v)| * 100 >
                              //   |N+(u)| * heavy_ratio_pct, else at its owner u
  int64_t hub_min_edges;      // the dense hub block runs when it holds at least
                              //   this many edges (< 0: never)
  int32_t hub_vertices;       // size of the hub set: a multiple of 128, <= kHubMaxSize
};
constexpr Tuning kDefaultTuning = {128, 64, 100, kHubMinEdges, kHubSize};

// A batch of graphs counted as one disjoint union (device-side descriptor).
// Graph g owns input pairs [edge_off[g], edge_off[g+1]) and union vertex ids
// [voff[g], voff[g+1]); pairs at or beyond edge_off[num_graphs] are padding
// and are dropped like self-loops.
struct BatchDesc {
  int32_t num_graphs;
  int32_t pad_;
  const int32_t *edge_off;  // [num_graphs + 1]
  const int32_t *voff;      // [num_graphs + 1]
  int32_t *gerr;            // [num_graphs], zero on entry; set: an id outside its graph
};

// Edges emitted to their partner groups by the list sort (direct.cu scatters
// them).  Slot off[u] + i holds the i-th entry of the sorted N+(u) as
//   skip << kSkipShift | h << b | l, h the endpoint whose list is hashed, l
//   the other, skip the leading blocks of N+(l) that cannot match; with
//   kOwnEdge when h = u, the skip field (0 then) being the edge's number among
//   u's own edges;
// or kHole: the entry was a repeat, or no triangle can be found there.
// gcnt[h] counts the edges emitted to h by others, own[u] gets u's own.  len:
// the list lengths with repeats.
struct GroupOut {
  uint64_t *gkeys;
  int32_t *gcnt, *own;
  const int32_t *len;
  int32_t b, heavy_ratio_pct;
};

// The bitmaps' records and the work items of the bitmap path (bits.cu):
// {group, first partner} for every kBitRange partners of every group that
// intersects by bitmaps, ctrl->n_bit_items of them in any order.
struct BitItems {
  uint32_t *rec;
  int2 *items;
};

// Workspace layout for an input of m_in pairs and n vertices.  All offsets
// are 256-byte aligned.
struct Layout {
  // zeroed by every run, in one piece: deg (unless the caller's array is
  // used), ctrl .. dcorr, t_rank (runs that need it), st_sort (runs that sort
  // by radix passes)
  size_t deg, ctrl, hist, st_orient, st_scan, st_scan2, st_scan4, outdeg, gcnt, dcorr, t_rank,
      st_sort;
  size_t keys_a, keys_b, off, voff, goff, groups;
  size_t col4;
  size_t rank, vkeys_a, vkeys_b;
  size_t hub;  // dense hub block (0 bytes unless the layout asked for it)
  // bitmaps (single graphs of at least kBitMinPairs pairs): without per-vertex
  // counts the records take the place of t_rank and the bitmaps that of the
  // group sort's free key buffer; with them both have their own.  Per-vertex
  // runs that sort by counting have each partner's stream in `desc` (others in
  // the group sort's free key buffer).  That is up to 8 bytes per pair more than
  // without per-vertex counts; a lean layout has neither, and takes as much as
  // one without.
  size_t desc;
  bool has_desc;
  bool has_bits;
  size_t bit_rec, bits;
  uint32_t bit_slots;
  bool has_hub;
  int32_t hub_vertices;  // size of the hub set the hub region was laid out for
  size_t total;
  uint32_t sort_tiles, orient_tiles, scan_tiles;
  size_t st_sort_words_per_pass;
};

// Radix sort tiles: 256 threads x 16 keys.
constexpr int kSortThreads = 256;
constexpr int kSortKeysPerThread = 16;
constexpr int kSortTile = kSortThreads * kSortKeysPerThread;
// Orientation/compaction tiles.
constexpr int kOrientThreads = 256;
constexpr int kOrientKeysPerThread = 16;
constexpr int kOrientTile = kOrientThreads * kOrientKeysPerThread;
// Offset-scan tiles.
constexpr int kScanThreads = 256;
constexpr int kScanItemsPerThread = 16;
constexpr int kScanTile = kScanThreads * kScanItemsPerThread;

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Number of bits that hold any id in [0, n): at least 1.
inline int id_bits(int32_t n) {
  int b = 1;
  while (b < 31 && ((int64_t)1 << b) < (int64_t)n) ++b;
  return b;
}

// Radix passes of one run over ids of b bits: the rank keys (degree <
// 2^b), the oriented keys (owner bits) and the group keys (group bits).
inline int radix_passes(int b) { return 3 * ((b + 7) / 8); }

// Whether a run of m pairs and n vertices (a batch: of the union) sorts by
// counting.
inline bool counting_sorts(int64_t m, int32_t n, bool batch) {
  return m <= (batch ? kDirectMaxBatchPairs : kDirectMaxPairs) && 2 * id_bits(n) <= kSkipShift &&
         (m <= kCrowdedPairs || m <= kCrowdedMean * n);
}

// Whether a single-graph run of n vertices has the dense hub block.
inline bool hub_enabled(int32_t n, int b) { return n >= kHubMinVertices && 2 * b <= kSkipShift; }

inline Layout make_layout(int64_t m_in, int32_t n, bool with_hub = false,
                          int32_t hub_vertices = kHubSize, bool batch = false,
                          bool per_vertex = false, bool lean = false) {
  Layout L{};
  size_t p = 0;
  auto take = [&](size_t bytes) {
    size_t at = p;
    p = align256(p + bytes);
    return at;
  };
  const uint64_t m = (uint64_t)(m_in > 0 ? m_in : 1);
  const uint64_t nv = (uint64_t)(n > 0 ? n : 1);
  const uint64_t keys_max = m > nv ? m : nv;  // the rank sort has n keys
  L.sort_tiles = (uint32_t)((keys_max + kSortTile - 1) / kSortTile);
  L.orient_tiles = (uint32_t)((m + kOrientTile - 1) / kOrientTile);
  L.scan_tiles = (uint32_t)((nv + 1 + kScanTile - 1) / kScanTile);
  L.st_sort_words_per_pass = (size_t)L.sort_tiles * 256;
  L.deg = take(sizeof(int32_t) * nv);
  L.ctrl = take(sizeof(Ctrl));
  L.hist = take(sizeof(uint32_t) * 256 * kMaxPasses);
  L.st_orient = take(sizeof(unsigned long long) * L.orient_tiles);
  L.st_scan = take(sizeof(unsigned long long) * L.scan_tiles);
  L.st_scan2 = take(sizeof(unsigned long long) * L.scan_tiles);
  L.st_scan4 = take(sizeof(unsigned long long) * L.scan_tiles);
  L.outdeg = take(sizeof(int32_t) * nv);
  L.gcnt = take(sizeof(int32_t) * nv);
  L.dcorr = take(sizeof(int32_t) * nv);
  L.t_rank = take(sizeof(int64_t) * nv);
  L.has_bits =
      !batch && !lean && m_in >= (per_vertex ? kBitMinPairs<true> : kBitMinPairs<false>);
  const uint64_t slots = m / (kBitCols / 32);  // two bitmaps each, in 8 m bytes
  L.bit_slots = (uint32_t)(slots < kBitMaxSlots ? slots : kBitMaxSlots);
  L.bit_rec = per_vertex && L.has_bits ? take(sizeof(uint32_t) * nv) : L.t_rank;
  // look-back status words for the passes that ids of [0, n) need (a run
  // with fewer vertices needs no more)
  L.st_sort = take(sizeof(unsigned long long) * L.st_sort_words_per_pass *
                   (size_t)radix_passes(id_bits(n > 0 ? n : 1)));
  L.keys_a = take(sizeof(uint64_t) * m);
  L.keys_b = take(sizeof(uint64_t) * m);
  L.off = take(sizeof(int32_t) * (nv + 1));
  L.voff = take(sizeof(int32_t) * (nv + 1));
  L.goff = take(sizeof(int32_t) * (nv + 1));
  L.groups = take(sizeof(int32_t) * nv);
  L.rank = take(sizeof(int32_t) * nv);
  L.vkeys_a = take(sizeof(uint64_t) * nv);
  L.vkeys_b = take(sizeof(uint64_t) * nv);
  // forward lists padded to whole 32-byte blocks: at most m + 7 min(n, m)
  // elements, since each non-empty list adds at most 7
  L.col4 = take(sizeof(int32_t) * (m + 7 * (nv < m ? nv : m)));
  L.bits = per_vertex && L.has_bits ? take((size_t)L.bit_slots * (kBitCols / 4)) : 0;
  L.has_desc = per_vertex && !lean && counting_sorts(m_in, n, batch);
  L.desc = L.has_desc ? take(sizeof(uint64_t) * m) : 0;
  const bool hub = with_hub && hub_enabled(n, id_bits(n > 0 ? n : 1));
  const size_t H = (size_t)hub_vertices;
  L.hub = take(hub ? H * H + 4 * H : 0);
  L.has_hub = hub;
  L.hub_vertices = hub_vertices;
  L.total = p;
  return L;
}


// Kernel-launch bookkeeping (defined in tc_api.cu).
void note_launch();

#ifdef __CUDACC__
// Every kernel of the library begins with grid_begin(), before any access to
// memory that another kernel of the stream may write or read: it lets the next
// kernel's blocks be launched as this one's have started, and waits until the
// kernels before this one have completed.  launch() marks a launch as allowed
// to begin that early while an EarlyLaunches of a small run is alive on the
// calling thread, so the kernels of the run follow each other without the gap
// of a launch (about 1 us each, of 4 to 20 us of kernel).  Blocks that wait
// take shared memory, and with it L1, from the kernel that runs, so larger
// runs launch in turn (kEarlyMaxPairs).
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Device memory is read by ordinary loads throughout, never as read-only data
// (ld.global.nc, __ldg, const __restrict__): a block of an early launch is
// resident while the kernels before it still write what it is going to read,
// and the read-only path is for data that no one writes during the life of a
// kernel; the wait above orders ordinary loads alone.  The loads keep their
// order among themselves and behind the wait (volatile), and may pass the
// kernel's own stores (no memory clobber): never for data that the same kernel
// writes.  Read-only / ordinary loads, whole calls: ring lattice of 50M pairs 4.49 /
// 4.49 ms, geometric of 67M 9.13 / 9.13 ms, R-MAT 21 of 91M 15.53 / 15.53 ms, 24 of
// 180M per vertex 37.13 / 37.12 ms.
__device__ __forceinline__ int32_t load(const int32_t *p) {
  int32_t x;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ uint32_t load(const uint32_t *p) {
  uint32_t x;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ int64_t load(const int64_t *p) {
  int64_t x;
  asm volatile("ld.global.b64 %0, [%1];" : "=l"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ int2 load(const int2 *p) {
  int2 x;
  asm volatile("ld.global.v2.b32 {%0, %1}, [%2];" : "=r"(x.x), "=r"(x.y) : "l"(p));
  return x;
}
__device__ __forceinline__ int4 load(const int4 *p) {
  int4 x;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
               : "l"(p));
  return x;
}
__device__ __forceinline__ uint4 load(const uint4 *p) {
  uint4 x;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
               : "l"(p));
  return x;
}

struct EarlyLaunches {
  explicit EarlyLaunches(int64_t pairs);
  ~EarlyLaunches();
  EarlyLaunches(const EarlyLaunches &) = delete;
  EarlyLaunches &operator=(const EarlyLaunches &) = delete;
  static bool allowed();
};

template <typename... Params, typename... Args>
void launch(void (*kernel)(Params...), uint32_t grid, uint32_t block, size_t smem,
            cudaStream_t st, Args &&...args) {
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = EarlyLaunches::allowed() ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
  note_launch();
}
#endif

// Test hooks of the wait paths (preprocess.cu), on the current device:
// spin_limit bounds every spin-wait (kSpinLimit by default); the radix-pass
// tile numbered unpublished_tile (kNoTile: none) never publishes its
// status, so the tiles after it wait on a word that nothing sets.
cudaError_t set_wait_hooks(uint32_t spin_limit, uint32_t unpublished_tile);
// The same for a tile of the offset scan of the lists (0) and of the groups (1),
// in all launches and captures from now on.
void set_unpublished_scan(int scan, uint32_t tile);

// ---- launchers (preprocess.cu) ----
// Undirected keys min << b | max of the pairs (self-loops and pairs with an
// id out of range: the sentinel 2^(2b) - 1) and deg[v] += 1 at both ends of
// every other pair (the degree with repeats; deg must be zero on entry).
void launch_canon(const int32_t *src, const int32_t *dst, uint32_t m_in, int32_t n, int b,
                  uint64_t *keys, int32_t *deg, Ctrl *ctrl, cudaStream_t st);
// The same for a batch: ids of pair i are local to its graph, checked against
// that graph's vertex count, and shifted by the graph's first union id.
// Zeroes totals[0 .. num_graphs_bound).
void launch_canon_batch(const int32_t *src, const int32_t *dst, uint32_t m_in, int b,
                        const BatchDesc *batch, int32_t num_graphs_bound,
                        unsigned long long *totals, uint64_t *keys, int32_t *deg, Ctrl *ctrl,
                        cudaStream_t st);
// Output of a radix pass: the keys themselves; the column array (low bits,
// to `out`) plus the row array (key >> owner_shift, to `row_out`) with the
// out-degrees added to `outdeg`; or the rank scatter rank[low bits] =
// sorted position (to `out`).
// kOutPartSkip: the group sort's last pass: low bits to `out` (partners),
// key >> kSkipShift to `row_out` (skipped blocks) and the group sizes (the
// field at owner_shift, under col_mask) added to `outdeg`.
enum RadixOut { kOutKeys = 0, kOutColRow = 1, kOutRank = 2, kOutPartSkip = 4 };
// unstable: keys of equal digit may leave in any order (kOutKeys only; the
// first pass of a sort whose input order does not matter).
void launch_radix_pass(const uint64_t *in, void *out, RadixOut mode, uint32_t *row_out,
                       int32_t *outdeg, uint32_t n_keys_bound, const uint32_t *n_keys_dev,
                       int shift, uint32_t col_mask, int owner_shift, const uint32_t *hist,
                       unsigned long long *status, uint32_t *ticket, Ctrl *ctrl,
                       cudaStream_t st, bool unstable = false);
// Keys deg(v) << b | v for every vertex, with the digit histograms of the
// degree field (the rank sort).
void launch_rank_keys(const int32_t *deg, int32_t n, int b, int passes, uint64_t *vkeys,
                      uint32_t *hist, cudaStream_t st);
// Every non-sentinel key (in any order) as (lower rank) << b | (higher
// rank), compacted, with the digit histograms of the owner field; sets
// ctrl->m to the number written.
void launch_orient(const uint64_t *keys, uint32_t m_in, int b, const int32_t *rank,
                   uint64_t *okeys, uint32_t *hist2, int passes2, unsigned long long *status,
                   Ctrl *ctrl, cudaStream_t st);
// The two node arrays of the forward lists from the list lengths counts[0..n):
// off[0..n], their exclusive scan, and voff[0..n], the exclusive scan of 2
// ceil(counts / 8): the node array of the padded column array (lists in
// whole 32-byte blocks), in 16-byte words.  Sets ctrl->m = off[n].
void launch_offsets(const int32_t *counts, int32_t n, int32_t *off, int32_t *voff,
                    unsigned long long *status, uint32_t *ticket, Ctrl *ctrl, cudaStream_t st);
// Exclusive scan of the partner-group sizes counts[h] (+ own[h], if not
// nullptr) -> goff[0..n], ctrl->n_part = goff[n]; the groups are binned into
// the lists by the length of their hashed list (ldesc): warp groups from
// the front of `groups` up, CTA groups from its end down (n entries hold
// both), big groups into big_list.  Only the groups h with h mod shards =
// shard are binned (the share of the counting work this run does; shards = 1
// bins them all).
void launch_group_offsets(const int32_t *counts, const int32_t *own, int32_t n, int32_t *goff,
                          const int2 *ldesc, int32_t *groups, int32_t *big_list,
                          Tuning tune, unsigned long long *status, uint32_t *ticket, Ctrl *ctrl,
                          cudaStream_t st, int32_t shard = 0, int32_t shards = 1);
// The node array again, from the list lengths left after the list sort
// dropped repeated edges, and ctrl->m = their sum; nothing (the kernel
// returns at once) when no list held a repeat.
void launch_recount(const int32_t *counts, int32_t n, int32_t *off, unsigned long long *status,
                    uint32_t *ticket, Ctrl *ctrl, cudaStream_t st);
// ---- launchers (hub.cu) ----
// Workspace of the dense hub block of H vertices: the H x H fp8 matrix and
// the per-vertex sums.
size_t hub_bytes(int32_t H);
// Decides on the device (into ctrl->hub_on, hub_size, hub_lo) whether, and
// with how many of the top ranks (a candidate up to Hmax), the hub block is
// counted densely; needs the node array and the column array (any order
// within a list).  An edge is taken to save at most `cap` lookups of
// ps_per_lookup picoseconds each.
void launch_hub_decide(const int32_t *off, const int32_t *col, int32_t n, int32_t Hmax,
                       int64_t min_edges, int32_t cap, double ps_per_lookup, Ctrl *ctrl,
                       cudaStream_t st);
// Counts the triangles inside the hub block (if ctrl->hub_on): adds them to
// ctrl->total and, if t != nullptr, to the per-vertex counts t (rank space).
// Needs the forward lists; region: hub_bytes(Hmax) bytes, 256-byte aligned.
cudaError_t launch_hub_count(const int2 *ldesc, const int32_t *col4, int32_t n, int32_t Hmax,
                             uint8_t *region, Ctrl *ctrl, int64_t *t, cudaStream_t st);
// ---- launchers (group.cu) ----
// Sorts every forward list (the column array col, grouped by owner, node
// array off) into the padded column array col4 (list v from 16-byte word
// voff[v], padded with -1 to whole 32-byte blocks) and writes ldesc[v] =
// {voff[v], length}: each list's first word and length in one record.  A
// repeated entry (an edge given more than once) is dropped: the list's
// length goes to dlen[v] (written only for such lists; dlen holds the
// lengths with repeats on entry), each dropped copy adds one to dcorr at
// both its ends (rank space; zero on entry) and ctrl->dups is set.
// emit (may be nullptr): the list sort also emits every edge to its partner
// group (see GroupOut), and leaves dlen alone.
// queue: n entries; the lists of more than 64 entries, ctrl->n_warp_lists
// of them from its front and ctrl->n_cta_lists (the longest) from its end
// down; col is scratch for lists longer than kCtaSortMax.
void launch_sort_lists(int32_t *col, const int32_t *off, const int32_t *voff, int32_t n,
                       Ctrl *ctrl, int32_t *col4, int32_t *queue, int32_t *dlen,
                       int32_t *dcorr, int2 *ldesc, const GroupOut *emit, cudaStream_t st);
// After the list sort, if some list held repeats: the row array again
// (row[off[v] + i] = v, from the recounted node array) and the degrees
// without repeats (deg[v] -= dcorr[rank[v]], caller ids).  Returns at once
// otherwise.  row == nullptr: the degrees alone.
void launch_fix_repeats(const int32_t *off, int32_t n, const int32_t *dcorr, const int32_t *rank,
                        Ctrl *ctrl, int32_t *row, int32_t *deg, cudaStream_t st);
// Group keys s << kSkipShift | h << b | l of the forward edges (h: the
// endpoint whose list is hashed, l: the other one, s: the leading blocks of
// N+(l) the intersection skips, 0 when 2b > kSkipShift), with the digit
// histograms of the h field for the group sort.  Reads the sorted lists (col4;
// their first words and lengths from ldesc, the lengths alone from len) in
// owner order (row, node array off).  whole: every edge, h the endpoint with
// the longer list; otherwise (2b <= kSkipShift) only the edges that need an
// intersection, by what is streamed, and ctrl->n_part (zero on entry) is
// their number.
void launch_group_keys(const int32_t *row, const int32_t *col4, const int32_t *off,
                       const int2 *ldesc, const int32_t *len, uint32_t m_bound, int b, int passes,
                       int32_t heavy_ratio_pct, bool whole, Ctrl *ctrl, uint64_t *gkeys,
                       uint32_t *hist, cudaStream_t st);
// Instrumentation: adds the counting phase's work into ctrl->work (from the
// partner groups, the node array and the skipped blocks), over the groups h
// with h mod shards = shard (the share one part counts).
void launch_work(const int32_t *off, const int32_t *goff, const int32_t *part,
                 const int32_t *pskip, int32_t n, Ctrl *ctrl, cudaStream_t st,
                 int32_t shard = 0, int32_t shards = 1);
// Instrumentation: what the counting kernels of this run read, into ctrl->work
// (see k_run_work).  desc != nullptr: each partner's stream instead of pskip.
void launch_run_work(const int32_t *goff, const int32_t *part, const int32_t *pskip,
                     const int2 *desc, const int2 *ldesc, const uint32_t *rec, int32_t n,
                     int32_t least, bool per_vertex, Ctrl *ctrl, cudaStream_t st);
// ---- launchers (direct.cu) ----
// rank[v] in an order by degree classes (ties in any order).  counters: 2
// kRankClasses words, zero on entry.
void launch_rank_classes(const int32_t *deg, int32_t n, uint32_t *counters, int32_t *rank,
                         cudaStream_t st);
// Every key as (lower rank) << b | (higher rank) with its place in the owner's
// list, the out-degrees counted (zero on entry); dropped pairs as kHole.
void launch_direct_orient(const uint64_t *keys, uint32_t m_in, int b, const int32_t *rank,
                          uint64_t *okeys, int32_t *place, int32_t *outdeg, Ctrl *ctrl,
                          cudaStream_t st);
// The column array from the oriented keys, their places and the node array.
void launch_direct_lists(const uint64_t *okeys, const int32_t *place, uint32_t m_in, int b,
                         const int32_t *off, int32_t *col, Ctrl *ctrl, cudaStream_t st);
// The partner and skip arrays from the emitted edges and the group offsets;
// gcnt counts down to zero.  desc != nullptr (no bitmaps): each partner's stream
// (see stream_desc) instead of its skip.
void launch_direct_groups(const uint64_t *gkeys, uint32_t m_bound, int b, int32_t n,
                          const int32_t *goff, int32_t *gcnt, int32_t *part, int32_t *pskip,
                          const int2 *ldesc, int2 *desc, Ctrl *ctrl, cudaStream_t st);
// ---- launchers (bits.cu) ----
// Bitmaps of the queued lists (launch_sort_lists) that have enough entries
// among the top ranks, at most `slots` - 1 of them: 2 kBitCols bits each into
// bits, their records into items.rec (zero on entry), and the work items of
// the groups h with h mod shards = shard (group offsets goff).
void launch_bits_build(const int32_t *queue, int32_t n, const int2 *ldesc, const int32_t *col4,
                       const int32_t *goff, uint32_t slots, bool per_vertex, uint32_t *bits,
                       const BitItems &items, Ctrl *ctrl, cudaStream_t st, int32_t shard,
                       int32_t shards);
// Intersections by bitmaps: adds what they find to ctrl->total and, if t !=
// nullptr, to the per-vertex counts t (rank space).  launch_count leaves
// exactly this part out when it is given the records.
void launch_count_bits(const int2 *ldesc, const int32_t *col4, const int32_t *goff,
                       const int32_t *part, const int32_t *pskip, const BitItems &items,
                       const uint32_t *bits, int32_t n, Ctrl *ctrl, int64_t *t, cudaStream_t st);
// ---- launchers (count.cu) ----
// t != nullptr: per-vertex counts (rank space).  Otherwise, if tg is not
// nullptr, tg[h] += triangles found in group h (their sum per graph is the
// graph's count).  desc: scratch of 8 bytes per partner (each partner's
// stream, written first unless desc_ready; with t only).
// groups, big_groups: the binned groups (launch_group_offsets).  rec: the
// bitmap records (nullptr: no bitmaps).
cudaError_t launch_count(const int2 *ldesc, const int32_t *col4, const int32_t *goff,
                         const int32_t *part, const int32_t *pskip, int2 *desc,
                         bool desc_ready, const int32_t *groups, const int32_t *big_groups,
                         const uint32_t *rec, int32_t n, Ctrl *ctrl, int64_t *t, int64_t *tg,
                         cudaStream_t st);
// Sets the counting kernels' attributes and occupancy for the current
// device (done lazily otherwise; needed before capturing a CUDA graph).
cudaError_t prepare_count_kernels();
// Adds every graph's group totals (tg, rank space) to totals[g] (zero on
// entry); ~0 (TC_COUNT_ERROR) for a graph that had an id out of range.  n:
// bound of the union's vertices.
void launch_batch_totals(const int64_t *tg, const int32_t *rank, const BatchDesc *batch,
                         int32_t n, const Ctrl *ctrl, unsigned long long *totals,
                         cudaStream_t st);
// ---- clustering (count.cu) ----
void launch_clustering(const int64_t *t, const int32_t *deg, int32_t n, double *cc,
                       unsigned long long *sums /* [2]: sum t, sum C(deg,2) */, cudaStream_t st);
void launch_transitivity(const unsigned long long *sums, double *out, cudaStream_t st);
// t_out[v] = t_rank[rank[v]]: per-vertex counts back to the caller's ids.
void launch_gather_counts(const int64_t *t_rank, const int32_t *rank, int32_t n, int64_t *t_out,
                          const Ctrl *ctrl, cudaStream_t st);

}  // namespace tc
