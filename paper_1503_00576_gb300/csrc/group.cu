// group.cu -- partner groups for the counting phase.
//
// The counting phase adds |N+(u) & N+(v)| over every forward edge (u, v)
// (Sec. II-B).  The intersection is symmetric in u and v, and the counting
// kernel computes it by hashing one list and streaming the other through
// the hash set, which costs one probe per element of the streamed list.
// Streaming the shorter list is cheapest.  When the hashed list is N+(v)'s,
// only the entries of N+(u) after v can match, so every forward edge is
// assigned to
//
//   h = v if what follows v in N+(u) is shorter by a third (in 32-byte
//   blocks) than N+(v), else h = u;     l = the other endpoint,
//
// and the edges are grouped by h, either by a counting sort (the list sort
// emits every edge, direct.cu scatters it) or by k_group_keys and radix passes
// over the h bits (preprocess.cu), whose last pass counts the group sizes.
// (Shares of a run and the work counters weigh the whole lists instead, see
// k_group_keys.)  A group then hashes N+(h) once and streams N+(l) for each of
// its partners l.  On the R-MAT graphs of the benchmarks this cuts the probes
// by a factor of 3 against always streaming N+(v).
//
// The lists themselves are sorted here (Sec. II-B sorts every forward list;
// the paper merges them, this path hashes, and uses the order only to skip
// the leading blocks of a streamed list that lie below the hashed list's
// smallest id -- a third of all blocks on R-MAT scale 24).
#include <climits>

#include "tc_common.cuh"

namespace tc {
namespace {

constexpr int kGroupThreads = 256;
constexpr int kGroupUnroll = 4;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// sorted forward lists
// ---------------------------------------------------------------------------
constexpr int kListThreads = 256;
constexpr int kListWarps = kListThreads / 32;
constexpr int kLongListThreads = 512;
constexpr int kLongListBlocks = 2;  // CTAs per SM (64 registers a thread)
// Lists of up to kWarpLaneMax entries are sorted where they are met, longer
// ones are queued (see k_sort_lists).
constexpr int kWarpLaneMax = 64;
constexpr int kWarpLongMax = 2 * kWarpSortMax;

__device__ __forceinline__ void cswap(int32_t &a, int32_t &b) {
  const int32_t x = min(a, b);
  b = max(a, b);
  a = x;
}

// Batcher's odd-even merge sort network for 8 keys (19 comparators).
__device__ __forceinline__ void sort8(int32_t (&x)[8]) {
  cswap(x[0], x[1]); cswap(x[2], x[3]); cswap(x[4], x[5]); cswap(x[6], x[7]);
  cswap(x[0], x[2]); cswap(x[1], x[3]); cswap(x[4], x[6]); cswap(x[5], x[7]);
  cswap(x[1], x[2]); cswap(x[5], x[6]);
  cswap(x[0], x[4]); cswap(x[1], x[5]); cswap(x[2], x[6]); cswap(x[3], x[7]);
  cswap(x[2], x[4]); cswap(x[3], x[5]);
  cswap(x[1], x[2]); cswap(x[3], x[4]); cswap(x[5], x[6]);
}

// Bitonic sort of 32 E keys held E per lane, key e*32 + lane in x[e] of
// lane `lane` (a warp-striped layout: loads and stores stay coalesced),
// ascending.  Exchanges between keys 32 or more apart stay in a lane;
// closer ones are shuffles.
template <int E>
__device__ __forceinline__ void warp_sort_regs(int32_t (&x)[E]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
        const int je = j >> 5;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if ((e & je) == 0) {
            const bool up = ((e * 32) & k) == 0;
            const int32_t a = x[e], b = x[e | je];
            x[e] = up ? min(a, b) : max(a, b);
            x[e | je] = up ? max(a, b) : min(a, b);
          }
        }
      } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int32_t y = __shfl_xor_sync(kFull, x[e], j);
          const bool up = ((e * 32 + lane) & k) == 0, low = (lane & j) == 0;
          x[e] = low == up ? min(x[e], y) : max(x[e], y);
        }
      }
    }
  }
}

// Where the list sort leaves its results (see launch_sort_lists).
struct ListOut {
  int32_t *col4;   // sorted lists, padded with -1 to whole 32-byte blocks
  int32_t *dlen;   // length of a list that held repeats, after dropping them (may be nullptr)
  int32_t *dcorr;  // per rank: repeated edges dropped at that vertex
  int2 *ldesc;     // per vertex: {first col4 word, length without repeats}
  Ctrl *ctrl;
};

// What the list sort needs to emit edges (GroupOut) beside the lists.
struct Emit {
  GroupOut g;
  const int32_t *len;  // list lengths: with repeats where the list sort emits, so that no
                       //   warp writes them meanwhile; otherwise without
  int32_t hub_lo;      // lists of vertices from this rank on are counted densely
  int32_t *hot;        // shared counters of the edges emitted to the ranks from
  int32_t hot_lo;      //   hot_lo on (nullptr: none)
};

__device__ __forceinline__ void count_edge(const Emit &o, int32_t h) {
  if (o.hot && h >= o.hot_lo) atomicAdd(&o.hot[h - o.hot_lo], 1);
  else atomicAdd(&o.g.gcnt[h], 1);
}

// The key of edge (u, v), v entry i of the du entries of the sorted N+(u);
// kHole if it needs no intersection.  The longer side is hashed, and what
// could be streamed of N+(u) is only its entries after v (those before it are
// below everything in N+(v)): so N+(u) from entry i + 1 on is weighed against
// N+(v), in whole 32-byte blocks.  (Weighing the whole lists, as
// k_group_keys does for shares, streams 10% to 25% more blocks.)  The lists of
// the later v are the hot ones in L2, so N+(u)'s rest has to be a third shorter
// to be streamed instead: against any shorter rest, Barabasi-Albert of 10M to
// 32M edges takes 4% to 11% less, R-MAT and lattices the same, geometric and
// uniform graphs 0.4% more.  A heavy ratio other than 100 weighs the whole lists
// by it.
__device__ __forceinline__ uint64_t edge_key(const Emit &o, int32_t u, int32_t du, int32_t i,
                                             int32_t v, bool &own) {
  const int32_t dv = o.len[v];
  bool at_v;
  int32_t skip;
  if (o.g.heavy_ratio_pct == 100) {
    skip = (i + 1) >> 3;
    if (i + 1 == du || dv == 0) return kHole;
    at_v = 3 * (((du + 7) >> 3) - skip) < 2 * ((dv + 7) >> 3);
  } else {
    skip = i >> 3;
    at_v = (int64_t)dv * 100 > (int64_t)du * o.g.heavy_ratio_pct;
  }
  own = !at_v;
  const uint64_t hu = (uint64_t)(uint32_t)u, hv = (uint64_t)(uint32_t)v;
  return at_v ? ((uint64_t)skip << kSkipShift) | (hv << o.g.b) | hu : (hu << o.g.b) | hv;
}

// Emits entry i (value x; valid: it exists) of the du entries of list u to
// slot `slot`; called by all lanes of `members` (a power-of-two part of the
// warp that works on list u) together.  own: u's own edges so far.
__device__ __forceinline__ void emit_entry(const Emit &o, int32_t u, int32_t du, int32_t i,
                                           int32_t x, bool valid, int64_t slot, uint32_t members,
                                           int32_t &own) {
  uint64_t key = kHole;
  bool mine = false;
  if (valid && u < o.hub_lo) key = edge_key(o, u, du, i, x, mine);
  mine = mine && key != kHole;
  const uint32_t bits = __ballot_sync(kFull, mine) & members;
  if (mine) {
    const int32_t k = own + __popc(bits & ((1u << (threadIdx.x & 31)) - 1u));
    key |= kOwnEdge | ((uint64_t)k << kSkipShift);
  }
  own += __popc(bits);
  if (valid) {
    o.g.gkeys[slot] = key;
    if (key != kHole && !mine) count_edge(o, x);
  }
}

// The list of u held `dropped` repeats and keeps len entries.  A repeat of
// edge (u, x) had added one to the degree of both ends: u's share is taken
// back here in one atomic for the list, x's where the repeat is met.  The
// flag is stored only until the SM's L1 has seen it set: with every edge
// given twice (50M pairs) a store and two atomics per repeat took 1.1 of the
// list sort's 1.65 ms.  Called by one lane.
__device__ __forceinline__ void note_repeats(int32_t u, int32_t dropped, int32_t len,
                                             const ListOut &o) {
  atomicAdd(&o.dcorr[u], dropped);
  if (o.dlen) o.dlen[u] = len;
  uint32_t seen;
  asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(seen) : "l"(&o.ctrl->dups));
  if (!seen) *(volatile uint32_t *)&o.ctrl->dups = 1u;
}

// Key e*32 + lane of a warp-striped sorted list repeats the key before it.
template <int E>
__device__ __forceinline__ bool warp_repeat(const int32_t (&x)[E], int e, int32_t d) {
  const int lane = threadIdx.x & 31;
  int32_t p = __shfl_up_sync(kFull, x[e], 1);
  const int32_t q = __shfl_sync(kFull, x[e > 0 ? e - 1 : 0], 31);
  if (lane == 0) p = q;
  const int i = e * 32 + lane;
  return i > 0 && i < d && x[e] == p;
}

// The warp emits the len entries of the finished list u (slots from b on, d of
// them); returns its own edges.
__device__ __forceinline__ int32_t emit_list(const Emit &em, int32_t u, int32_t b, int32_t d,
                                             int32_t len, const int32_t *list) {
  const int lane = threadIdx.x & 31;
  int32_t own = 0;
#pragma unroll 2
  for (int32_t i0 = 0; i0 < d; i0 += 32) {
    const int32_t i = i0 + lane;
    const int32_t x = i < len ? list[i] : 0;
    emit_entry(em, u, len, i, x, i < len, (int64_t)b + i, kFull, own);
    if (i >= len && i < d) em.g.gkeys[(int64_t)b + i] = kHole;
  }
  return own;
}

// The warp sorts list v (d entries from col + b) into col4 from entry w4,
// with E keys per lane (32 E >= d), dropping repeated entries; returns the
// entries left.
template <int E, bool EMIT>
__device__ __forceinline__ int32_t warp_sort_list(const int32_t *col, int32_t b,
                                                  int32_t d, long long w4, int32_t v,
                                                  const ListOut &o, const Emit &em) {
  const int lane = threadIdx.x & 31;
  int32_t x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * 32 + lane;
    x[e] = i < d ? load(col + b + i) : INT32_MAX;
  }
  warp_sort_regs<E>(x);
  const int r8 = (d + 7) & ~7;
  uint32_t reps = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) reps |= __ballot_sync(kFull, warp_repeat<E>(x, e, d));
  if (reps == 0) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = e * 32 + lane;
      if (i < r8) o.col4[w4 + i] = i < d ? x[e] : -1;
    }
    if (EMIT) {
      int32_t own = 0;
      if constexpr (E <= 2) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = e * 32 + lane;
          emit_entry(em, v, d, i, x[e], i < d, (int64_t)b + i, kFull, own);
        }
      } else {  // from memory: the keys' registers are needed
        __syncwarp();
        own = emit_list(em, v, b, d, d, o.col4 + w4);
      }
      if (lane == 0) em.g.own[v] = own;
    }
    return d;
  }
  // some entry repeats (an edge given more than once): compact the rest
  const uint32_t lt = (1u << lane) - 1u;
  int len = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * 32 + lane;
    const bool rep = warp_repeat<E>(x, e, d);
    const bool keep = i < d && !rep;
    const uint32_t bk = __ballot_sync(kFull, keep);
    if (keep) o.col4[w4 + len + __popc(bk & lt)] = x[e];
    if (rep) atomicAdd(&o.dcorr[x[e]], 1);
    len += __popc(bk);
  }
  for (int i = len + lane; i < r8; i += 32) o.col4[w4 + i] = -1;
  if (lane == 0) note_repeats(v, d - len, len, o);
  if (EMIT) {
    __syncwarp();
    const int32_t own = emit_list(em, v, b, d, len, o.col4 + w4);
    if (lane == 0) em.g.own[v] = own;
  }
  return len;
}

// Both halves of the warp sort one list of 9 to 16 entries each, one entry
// per lane (d = 0: that half has none); returns the entries left.  Half the
// steps of a whole warp per list, which these lists (most of a random
// geometric graph's) would leave half empty.
template <bool EMIT>
__device__ __forceinline__ int32_t half_sort_list(const int32_t *col, int32_t b,
                                                  int32_t d, long long w4, int32_t v,
                                                  const ListOut &o, const Emit &em) {
  const int lane = threadIdx.x & 31, i = lane & 15;
  int32_t x = i < d ? load(col + b + i) : INT32_MAX;
#pragma unroll
  for (int k = 2; k <= 16; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const int32_t y = __shfl_xor_sync(kFull, x, j);
      const bool up = (i & k) == 0, low = (i & j) == 0;
      x = low == up ? min(x, y) : max(x, y);
    }
  }
  const int32_t p = __shfl_up_sync(kFull, x, 1, 16);
  const bool rep = i > 0 && i < d && x == p;
  const uint32_t half = lane & 16 ? 0xffff0000u : 0x0000ffffu;
  const uint32_t reps = __ballot_sync(kFull, rep) & half;
  const uint32_t kept = __ballot_sync(kFull, i < d && !rep) & half;
  const int32_t len = __popc(kept);
  if (d == 0) {
    // this half has no list
  } else if (reps == 0) {
    o.col4[w4 + i] = i < d ? x : -1;
  } else {  // an edge given more than once
    if (i < d && !rep) o.col4[w4 + __popc(kept & ((1u << lane) - 1u))] = x;
    if (rep) atomicAdd(&o.dcorr[x], 1);
    if (i >= len) o.col4[w4 + i] = -1;
    if (i == 0) note_repeats(v, d - len, len, o);
  }
  if (EMIT) {
    __syncwarp();
    if (reps != 0) x = i < len ? o.col4[w4 + i] : 0;
    int32_t own = 0;
    emit_entry(em, v, len, i, x, i < len, (int64_t)b + i, half, own);
    if (i >= len && i < d) em.g.gkeys[(int64_t)b + i] = kHole;
    if (i == 0 && d > 0) em.g.own[v] = own;
  }
  return len;
}

// Bitonic sort of buf[0..P) (P a power of two) by a whole block of G
// threads, ascending.
template <int G>
__device__ __forceinline__ void bitonic_smem(int32_t *buf, int P, int rank) {
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = rank; i < P / 2; i += G) {
        const int lo = ((i & ~(j - 1)) << 1) | (i & (j - 1)), hi = lo + j;
        const int32_t a = buf[lo], b = buf[hi];
        if ((a > b) == ((lo & k) == 0)) {
          buf[lo] = b;
          buf[hi] = a;
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ int pow2_at_least(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Exclusive scan of one value per thread over a block of G threads; *total
// gets the sum.  All threads must call it; s_warp holds G / 32 words.
template <int G>
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *s_warp, uint32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < G / 32; ++w) {
    const uint32_t t = s_warp[w];
    if (w < warp) before += t;
    all += t;
  }
  __syncthreads();  // s_warp is reused by the next call
  *total = all;
  return before + incl - x;
}

// Copies the sorted list buf[0..d) of vertex v to dst without its repeated
// entries, padded with -1 up to r8 entries, by a block of G threads (buf in
// shared or global memory, written before the last barrier); returns the
// entries left.
template <int G>
__device__ int32_t cta_unique_copy(const int32_t *buf, int32_t d, int32_t *__restrict__ dst,
                                   int32_t r8, int32_t v, const ListOut &o, uint32_t *s_warp) {
  constexpr int PER = 16;  // consecutive entries per thread
  const int tid = threadIdx.x;
  int32_t len = 0;  // uniform: entries written so far
  for (int32_t t0 = 0; t0 < d; t0 += G * PER) {
    const int32_t j0 = t0 + tid * PER;
    uint32_t keep = 0, cnt = 0;
    int32_t prev = (j0 > 0 && j0 < d) ? buf[j0 - 1] : 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int32_t j = j0 + q;
      if (j < d) {
        const int32_t x = buf[j];
        const bool k = j == 0 || x != prev;
        if (!k) atomicAdd(&o.dcorr[x], 1);
        prev = x;
        keep |= (uint32_t)k << q;
        cnt += k;
      }
    }
    uint32_t total;
    uint32_t pos = (uint32_t)len + block_scan<G>(cnt, s_warp, &total);
#pragma unroll
    for (int q = 0; q < PER; ++q)
      if ((keep >> q) & 1u) dst[pos++] = buf[j0 + q];
    len += (int32_t)total;
  }
  for (int32_t j = len + tid; j < r8; j += G) dst[j] = -1;
  if (tid == 0 && len < d) note_repeats(v, d - len, len, o);
  return len;
}

// Every forward list into col4, sorted ascending, without repeated entries
// and padded with -1 to whole 32-byte blocks.  Warps take `per` consecutive
// vertices at a time (32, or fewer so that a small graph's lists spread over
// all SMs: 16,384 vertices, 20 / 7 us): a list of up to 8 entries is sorted by its own lane in
// registers (a sorting network), one of up to 16 by half a warp, one of up
// to kWarpLaneMax by the warp (bitonic, in registers).  Longer ones are
// queued for k_sort_long_lists, where every warp of the GPU takes one at a
// time: the long lists belong to neighbouring ranks, and a warp that met 32
// of them finished long after all others (all lists of R-MAT scale 16 with
// 2.5M edges: 168 us, with the queue 64 us).
template <bool EMIT>
__global__ void __launch_bounds__(kListThreads)
k_sort_lists(const int32_t *col, const int32_t *off,
             const int32_t *voff, int32_t n, uint32_t per, ListOut o, GroupOut g,
             int32_t *__restrict__ queue) {
  grid_begin();
  Ctrl *ctrl = o.ctrl;
  if (aborted(ctrl)) return;  // an earlier wait of this call ran out
  const Emit em{g, g.len, ctrl->hub_on ? (int32_t)ctrl->hub_lo : n, nullptr, n};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t warps = gridDim.x * kListWarps;
  const uint32_t lt = (1u << lane) - 1u;
  for (uint32_t c = blockIdx.x * kListWarps + warp; c * per < (uint32_t)n; c += warps) {
    const uint32_t v = c * per + lane;
    const bool exists = (uint32_t)lane < per && v < (uint32_t)n;
    int32_t b = 0, d = 0, w = 0, len = 0;
    if (exists) {
      b = load(off + v);
      d = load(off + v + 1) - b;
      w = load(voff + v);
    }
    const long long w4 = 4ll * w;  // first col4 entry of the list
    if (d > 0 && d <= 8) {
      int32_t x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = i < d ? load(col + b + i) : INT32_MAX;
      sort8(x);
      uint32_t reps = 0;  // bit i: entry i repeats entry i - 1
#pragma unroll
      for (int i = 1; i < 8; ++i) reps |= (uint32_t)(i < d && x[i] == x[i - 1]) << i;
      if (reps == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i >= d) x[i] = -1;
        int4 *dst = reinterpret_cast<int4 *>(o.col4 + w4);
        dst[0] = make_int4(x[0], x[1], x[2], x[3]);
        dst[1] = make_int4(x[4], x[5], x[6], x[7]);
        len = d;
      } else {  // an edge given more than once
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i < d && ((reps >> i) & 1u)) atomicAdd(&o.dcorr[x[i]], 1);
          else if (i < d) o.col4[w4 + len++] = x[i];
        }
        for (int i = len; i < 8; ++i) o.col4[w4 + i] = -1;
        note_repeats((int32_t)v, d - len, len, o);
      }
      if (EMIT) {
        int32_t own = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i >= d) break;
          uint64_t key = kHole;
          if (i < len && (int32_t)v < em.hub_lo) {
            const int32_t y = reps == 0 ? x[i] : o.col4[w4 + i];
            bool mine = false;
            key = edge_key(em, (int32_t)v, len, i, y, mine);
            if (key != kHole && mine) key |= kOwnEdge | ((uint64_t)own++ << kSkipShift);
            else if (key != kHole) count_edge(em, y);
          }
          em.g.gkeys[(int64_t)b + i] = key;
        }
        em.g.own[v] = own;
      }
    }
    if (EMIT && d == 0 && exists) em.g.own[v] = 0;
    uint32_t todo = __ballot_sync(kFull, d > 8 && d <= 16);
    while (todo) {  // two lists at a time
      const int s0 = __ffs(todo) - 1;
      todo &= todo - 1;
      const int s1 = todo ? __ffs(todo) - 1 : s0;
      const bool second = lane >= 16, none = second && s1 == s0;
      todo &= todo - 1;
      const int src = second ? s1 : s0;
      const int32_t lb = __shfl_sync(kFull, b, src), ld = __shfl_sync(kFull, d, src);
      const long long lw = __shfl_sync(kFull, w4, src);
      const int32_t l = half_sort_list<EMIT>(col, lb, none ? 0 : ld, lw,
                                             (int32_t)(c * per) + src, o, em);
      const int32_t l0 = __shfl_sync(kFull, l, 0), l1 = __shfl_sync(kFull, l, 16);
      if (lane == s0) len = l0;
      else if (lane == s1) len = l1;
    }
    todo = __ballot_sync(kFull, d > 16 && d <= kWarpLaneMax);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int32_t lb = __shfl_sync(kFull, b, src), ld = __shfl_sync(kFull, d, src);
      const long long lw = __shfl_sync(kFull, w4, src);
      const int32_t lv = (int32_t)(c * per) + src;
      const int32_t l = ld <= 32 ? warp_sort_list<1, EMIT>(col, lb, ld, lw, lv, o, em)
                                 : warp_sort_list<2, EMIT>(col, lb, ld, lw, lv, o, em);
      if (lane == src) len = l;
    }
    if (exists && d <= kWarpLaneMax) o.ldesc[v] = make_int2(w, len);
    // the queues: lists for a warp from the front of the array, lists for a
    // CTA from its end down
    const bool is_warp = d > kWarpLaneMax && d <= kWarpLongMax, is_cta = d > kWarpLongMax;
    const uint32_t bw = __ballot_sync(kFull, is_warp), bc = __ballot_sync(kFull, is_cta);
    if (bw | bc) {
      uint32_t at = 0;
      if (lane == 0 && bw) at = atomicAdd(&ctrl->n_warp_lists, (uint32_t)__popc(bw));
      if (lane == 1 && bc) at = atomicAdd(&ctrl->n_cta_lists, (uint32_t)__popc(bc));
      const uint32_t aw = __shfl_sync(kFull, at, 0), ac = __shfl_sync(kFull, at, 1);
      if (is_warp) queue[aw + __popc(bw & lt)] = (int32_t)v;
      if (is_cta) queue[(uint32_t)n - 1u - (ac + __popc(bc & lt))] = (int32_t)v;
    }
  }
}

// Number of entries of the sorted a[0..len) below x (lower) or not above x
// (upper); plain loads (a may have been written by this kernel).
__device__ __forceinline__ int32_t count_below(const int32_t *a, int32_t len, int32_t x,
                                               bool or_equal) {
  int32_t lo = 0, hi = len;
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    const int32_t y = a[mid];
    if (y < x || (or_equal && y == x)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// The queued lists: first those longer than kWarpLongMax, one CTA each, then
// the others, one warp each with up to 32 keys per lane in registers.  A CTA
// sorts up to kCtaSortMax entries in shared memory; a longer list (only with
// a dense core of more than kCtaSortMax vertices) is sorted in chunks of
// kCtaSortMax, which are then merged pairwise in global memory, alternating
// between the list's own region of the column array and its region of col4
// so that the last merge lands in the column array.  Then the repeats are
// dropped on the way into col4.
template <bool EMIT>
__global__ void __launch_bounds__(kLongListThreads, kLongListBlocks)
k_sort_long_lists(int32_t *col, const int32_t *off,
                  const int32_t *voff, int32_t n, ListOut o, GroupOut g,
                  const int32_t *queue) {
  grid_begin();
  constexpr int G = kLongListThreads;
  __shared__ int32_t s_buf[kCtaSortMax];
  __shared__ uint32_t s_warp[G / 32];
  __shared__ uint32_t s_i;
  Ctrl *ctrl = o.ctrl;
  if (aborted(ctrl)) return;
  __shared__ int32_t s_own;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t n_cta = ctrl->n_cta_lists, n_warp = ctrl->n_warp_lists;
  Emit em{g, g.len, ctrl->hub_on ? (int32_t)ctrl->hub_lo : n, nullptr, n};
  while (n_cta) {
    if (tid == 0) s_i = atomicAdd(&ctrl->next_cta_list, 1u);
    __syncthreads();
    const uint32_t i = s_i;
    if (i >= n_cta) break;
    const int32_t v = load(queue + ((uint32_t)n - 1u - i));
    const int32_t b = load(off + v), d = load(off + v + 1) - b, w = load(voff + v);
    int32_t *dst = o.col4 + 4ll * w;
    const int r8 = (d + 7) & ~7;
    int32_t len;
    if (d <= kCtaSortMax) {
      const int P = pow2_at_least(d);
      for (int j = tid; j < P; j += G) s_buf[j] = j < d ? col[b + j] : INT32_MAX;
      __syncthreads();
      bitonic_smem<G>(s_buf, P, tid);
      len = cta_unique_copy<G>(s_buf, d, dst, r8, v, o, s_warp);
    } else {
      int32_t *A = col + b;  // the list's region of the column array: d entries
      int32_t *B = dst;      // its region of col4: r8 >= d entries
      const int32_t chunks = (d + kCtaSortMax - 1) / kCtaSortMax;
      int levels = 0;
      while ((1 << levels) < chunks) ++levels;
      int32_t *src = (levels & 1) ? B : A;
      for (int32_t c0 = 0; c0 < d; c0 += kCtaSortMax) {
        const int32_t part = min(kCtaSortMax, d - c0);
        for (int j = tid; j < kCtaSortMax; j += G) s_buf[j] = j < part ? A[c0 + j] : INT32_MAX;
        __syncthreads();
        bitonic_smem<G>(s_buf, kCtaSortMax, tid);
        for (int j = tid; j < part; j += G) src[c0 + j] = s_buf[j];
        __syncthreads();
      }
      int32_t *to = src == A ? B : A;
      for (int32_t run = kCtaSortMax; run < d; run <<= 1) {
        // runs [s0, s0 + run) and [s0 + run, s0 + 2 run) merged into
        // to[s0 ..): an entry's place is its place in its run plus the
        // entries of the other run before it (ties: the first run's first)
        for (int32_t j = tid; j < d; j += G) {
          const int32_t s0 = j / (2 * run) * (2 * run);
          const int32_t am = min(s0 + run, d), be = min(s0 + 2 * run, d);
          const int32_t x = src[j];
          const int32_t at = j < am ? (j - s0) + count_below(src + am, be - am, x, false)
                                    : (j - am) + count_below(src + s0, am - s0, x, true);
          to[s0 + at] = x;
        }
        __syncthreads();
        int32_t *t = src;
        src = to;
        to = t;
      }
      len = cta_unique_copy<G>(A, d, B, r8, v, o, s_warp);
    }
    if (tid == 0) o.ldesc[v] = make_int2(w, len);
    if (EMIT) {
      // the warps' own edges take numbers from a shared counter, a chunk at
      // a time
      if (tid == 0) s_own = 0;
      __syncthreads();  // also: the list is written
      for (int32_t i0 = 32 * (tid >> 5); i0 < d; i0 += G) {
        const int32_t i = i0 + lane;
        const int32_t x = i < len ? dst[i] : 0;
        bool mine = false;
        uint64_t key = kHole;
        if (i < len && v < em.hub_lo) key = edge_key(em, v, len, i, x, mine);
        mine = mine && key != kHole;
        const uint32_t bal = __ballot_sync(kFull, mine);
        int32_t first = 0;
        if (lane == 0 && bal) first = atomicAdd(&s_own, __popc(bal));
        first = __shfl_sync(kFull, first, 0);
        if (mine)
          key |= kOwnEdge |
                 ((uint64_t)(first + __popc(bal & ((1u << lane) - 1u))) << kSkipShift);
        if (i < d) em.g.gkeys[(int64_t)b + i] = key;
        if (key != kHole && !mine) count_edge(em, x);
      }
      __syncthreads();
      if (tid == 0) em.g.own[v] = s_own;
    }
    __syncthreads();  // s_buf, s_i and s_own are reused
  }
  if (n_warp == 0) return;
  if (EMIT) {
    // most edges of these lists go to the groups of the highest ranks: counted
    // in shared memory first (one counter in L2 took 30,000 additions of a
    // graph of 2.5M edges, and the kernel 90 us instead of 30)
    __syncthreads();
    for (int j = tid; j < kCtaSortMax; j += G) s_buf[j] = 0;
    __syncthreads();
    em.hot = s_buf;
    em.hot_lo = max(n - kCtaSortMax, 0);
  }
  for (;;) {
    uint32_t i = 0;
    if (lane == 0) i = atomicAdd(&ctrl->next_warp_list, 1u);
    i = __shfl_sync(kFull, i, 0);
    if (i >= n_warp) break;
    const int32_t v = load(queue + i);
    const int32_t b = load(off + v), d = load(off + v + 1) - b, w = load(voff + v);
    const int32_t len = d <= 128   ? warp_sort_list<4, EMIT>(col, b, d, 4ll * w, v, o, em)
                        : d <= 256 ? warp_sort_list<8, EMIT>(col, b, d, 4ll * w, v, o, em)
                        : d <= 512 ? warp_sort_list<16, EMIT>(col, b, d, 4ll * w, v, o, em)
                                   : warp_sort_list<32, EMIT>(col, b, d, 4ll * w, v, o, em);
    if (lane == 0) o.ldesc[v] = make_int2(w, len);
  }
  if (EMIT) {
    __syncthreads();
    for (int j = tid; j < kCtaSortMax; j += G)
      if (s_buf[j]) atomicAdd(&g.gcnt[em.hot_lo + j], s_buf[j]);
  }
}

// After repeats were dropped: the row array again, row[off[v] + i] = v (off:
// the recounted node array), one warp per vertex, and the degrees without
// the repeats, deg[v] -= dcorr[rank[v]] (caller ids).  Nothing when no list
// held a repeat.
__global__ void __launch_bounds__(kListThreads)
k_fix_repeats(const int32_t *off, int32_t n, const int32_t *dcorr,
              const int32_t *rank, const Ctrl *ctrl, int32_t *__restrict__ row,
              int32_t *__restrict__ deg) {
  grid_begin();
  if (aborted(ctrl) || ctrl->dups == 0u) return;
  const int lane = threadIdx.x & 31;
  const uint32_t first = blockIdx.x * kListThreads + threadIdx.x;
  const uint32_t stride = gridDim.x * kListThreads;
  for (uint32_t v = first; v < (uint32_t)n; v += stride) deg[v] -= load(dcorr + load(rank + v));
  if (!row) return;
  for (uint32_t v = first >> 5; v < (uint32_t)n; v += stride >> 5) {
    const int32_t b = load(off + v), e = load(off + v + 1);
    for (int32_t i = b + lane; i < e; i += 32) row[i] = (int32_t)v;
  }
}

// heavy_ratio_pct = 100: the longer list is always the one hashed; larger
// values keep an edge at its owner unless v's list is that much longer.
__device__ __forceinline__ void split_edge(int32_t u, int32_t v, int64_t du, int64_t dv,
                                           int32_t heavy_ratio_pct, int32_t &h, int32_t &l) {
  if (dv * 100 > du * heavy_ratio_pct) {
    h = v;
    l = u;
  } else {
    h = u;
    l = v;
  }
}

// One pass over the forward edges in owner order (row[e] = u; the sorted
// list N+(u) of col4 holds v at position i = e - off[u]; row and off are
// those left after the list sort dropped repeated edges): the group key of
// every edge with the digit histograms of its h field.
//
// WHOLE: the whole lists are weighed against each other, every edge has a
// key.  When the longer list is v's (h = v), the intersection streams N+(u),
// whose entries before position i are all below v; N+(h) holds only ids above
// h = v, so those entries cannot match and the whole blocks among them,
// i >> 3, are skipped.  Their count rides in the key's top bits to the partner
// array.  (When h = u, N+(v) is streamed and all its entries lie above v,
// itself in N+(u): nothing to skip.)  This is the split whose work
// tc_count_work reports and whose shares tc_count_part deals out.
//
// Otherwise edge_key() decides, and the edges that need no intersection (the
// last entry of a list, an empty N+(v), an edge inside the dense hub block) are
// left out: a warp takes the places of its round's keys with one atomic (the
// first pass of the sort orders equal digits freely, so their order does not
// matter).  R-MAT scale 21 (91M edges): a quarter of the keys and an eighth
// of the streamed blocks less.
template <bool WHOLE>
__global__ void __launch_bounds__(kGroupThreads)
k_group_keys(const int32_t *row, const int32_t *col4,
             const int32_t *off, const int2 *ldesc,
             const int32_t *len, int b, int passes, int32_t heavy_ratio_pct,
             Ctrl *ctrl, uint64_t *__restrict__ gkeys,
             uint32_t *__restrict__ hist) {
  grid_begin();
  constexpr int UNROLL = WHOLE ? kGroupUnroll : 2 * kGroupUnroll;
  __shared__ uint32_t s_hist[kMaxGroupPasses * 256];
  if (aborted(ctrl)) return;  // an earlier wait of this call ran out
  for (int i = threadIdx.x; i < passes * 256; i += kGroupThreads) s_hist[i] = 0;
  __syncthreads();
  const uint32_t m = ctrl->m;
  const bool carry_skip = 2 * b <= kSkipShift;
  const bool hub_on = carry_skip && ctrl->hub_on != 0u;
  const int32_t hub_lo = (int32_t)ctrl->hub_lo;
  const Emit em{GroupOut{nullptr, nullptr, nullptr, nullptr, b, heavy_ratio_pct}, len, 0, nullptr, 0};
  const uint32_t stride = gridDim.x * kGroupThreads;
  // UNROLL edges per thread per round, each step's loads issued for
  // all of them together: the offsets are gathers that depend on the edge
  const int lane = threadIdx.x & 31;
  for (uint32_t e0 = blockIdx.x * kGroupThreads + threadIdx.x; e0 - lane < m;
       e0 += UNROLL * stride) {
    int32_t u[UNROLL], ub[UNROLL], ue[UNROLL], uw[UNROLL];
#pragma unroll
    for (int q = 0; q < UNROLL; ++q) {
      const uint32_t e = e0 + q * stride;
      u[q] = e < m ? load(row + e) : 0;
    }
#pragma unroll
    for (int q = 0; q < UNROLL; ++q) {
      ub[q] = load(off + u[q]);
      const int2 ld = load(ldesc + u[q]);  // {first col4 word, length}
      ue[q] = ub[q] + ld.y;
      uw[q] = ld.x;
    }
    int32_t v[UNROLL];
#pragma unroll
    for (int q = 0; q < UNROLL; ++q) {
      const uint32_t e = e0 + q * stride;
      v[q] = e < m ? load(col4 + 4ll * uw[q] + ((int32_t)e - ub[q])) : 0;
    }
    uint64_t key[UNROLL];
    uint32_t kept = 0;
    if (WHOLE) {
      int32_t vd[UNROLL];
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) vd[q] = load(ldesc + v[q]).y;
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) {
        const uint32_t e = e0 + q * stride;
        int32_t h, l;
        split_edge(u[q], v[q], ue[q] - ub[q], vd[q], heavy_ratio_pct, h, l);
        // an edge inside the dense hub block (owner u, hence v, of rank >=
        // hub_lo) is left to it: its stream is skipped whole
        uint64_t skip =
            (carry_skip && h == v[q]) ? (uint64_t)(((int32_t)e - ub[q]) >> 3) : 0ull;
        if (hub_on && u[q] >= hub_lo) skip = kSkipAll;
        key[q] = (skip << kSkipShift) | ((uint64_t)(uint32_t)h << b) | (uint32_t)l;
        kept |= (uint32_t)(e < m) << q;
      }
    } else {
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) {
        const uint32_t e = e0 + q * stride;
        bool own;
        key[q] = kHole;
        if (e < m && !(hub_on && u[q] >= hub_lo))
          key[q] = edge_key(em, u[q], ue[q] - ub[q], (int32_t)e - ub[q], v[q], own);
        kept |= (uint32_t)(key[q] != kHole) << q;
      }
    }
    uint32_t at[UNROLL];
    if (WHOLE) {
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) at[q] = e0 + q * stride;
    } else {  // the warp takes the places of its round's keys
      uint32_t total = 0;
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) {
        const uint32_t bits = __ballot_sync(kFull, (kept >> q) & 1u);
        at[q] = total + __popc(bits & ((1u << lane) - 1u));
        total += __popc(bits);
      }
      uint32_t base = 0;
      if (lane == 0 && total) base = atomicAdd(&ctrl->n_part, total);
      base = __shfl_sync(kFull, base, 0);
#pragma unroll
      for (int q = 0; q < UNROLL; ++q) at[q] += base;
    }
#pragma unroll
    for (int q = 0; q < UNROLL; ++q) {
      if (!((kept >> q) & 1u)) continue;
      gkeys[at[q]] = key[q];
      const uint32_t h = (uint32_t)(key[q] >> b) & (uint32_t)((1ull << b) - 1);
      for (int p = 0; p < passes; ++p) atomicAdd(&s_hist[p * 256 + ((h >> (8 * p)) & 255u)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * 256; i += kGroupThreads)
    if (s_hist[i]) atomicAdd(&hist[i], s_hist[i]);
}

// Work of the counting phase, for instrumentation only (never on the path
// of a count): per forward edge (h, l) of group h, the entries of N+(l)
// streamed through the hash set (d+(l) less the skipped leading blocks),
// and the merge work d+(h) + d+(l) of
// Sec. II-B; per non-empty group, the list hashed once, d+(h) inserts; the
// largest d+.  Also, per hub set H = the 2^12 .. 2^15 highest ranks, the
// lookups of the edges with both endpoints in H: ranks follow (degree, id),
// so every forward neighbour of a vertex of H is in H, and those edges'
// intersections lie wholly inside H (what a dense count of the hub block
// A_HH would take over, Sec. VI).  One warp per vertex h.
__global__ void __launch_bounds__(kGroupThreads)
k_work(const int32_t *off, const int32_t *goff,
       const int32_t *part, const int32_t *pskip, int32_t n,
       Ctrl *ctrl, uint32_t shard, uint32_t shards) {
  grid_begin();
  if (aborted(ctrl)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (kGroupThreads / 32);
  unsigned long long lookups = 0, inserts = 0, merge = 0, dmax = 0, hub[kHubSizes] = {};
  for (uint32_t h = (blockIdx.x * kGroupThreads + threadIdx.x) >> 5; h < (uint32_t)n;
       h += warps) {
    if (h % shards != shard) continue;  // another part's group (uniform per warp)
    const unsigned long long dh = (unsigned long long)(load(off + h + 1) - load(off + h));
    const int32_t pb = load(goff + h), pe = load(goff + h + 1);
    if (lane == 0) {
      if (pe > pb) inserts += dh;
      dmax = dh > dmax ? dh : dmax;
    }
    for (int32_t i = pb + lane; i < pe; i += 32) {
      const int32_t l = load(part + i);
      const int32_t dfull = load(off + l + 1) - load(off + l);
      const int32_t ds = max(dfull - 8 * load(pskip + i), 0);  // entries streamed
      const unsigned long long dl = (unsigned long long)ds;
      lookups += dl;
      merge += dh + (unsigned long long)dfull;
#pragma unroll
      for (int k = 0; k < kHubSizes; ++k) {
        const int64_t lo = (int64_t)n - ((int64_t)1 << (kHubLog2Min + k));
        if ((int64_t)h >= lo && (int64_t)l >= lo) hub[k] += dl;
      }
    }
  }
  for (int o = 16; o; o >>= 1) {
    lookups += __shfl_xor_sync(0xffffffffu, lookups, o);
    inserts += __shfl_xor_sync(0xffffffffu, inserts, o);
    merge += __shfl_xor_sync(0xffffffffu, merge, o);
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, dmax, o);
    dmax = x > dmax ? x : dmax;
#pragma unroll
    for (int k = 0; k < kHubSizes; ++k) hub[k] += __shfl_xor_sync(0xffffffffu, hub[k], o);
  }
  if (lane == 0) {
    atomicAdd(&ctrl->work[0], lookups);
    atomicAdd(&ctrl->work[1], inserts);
    atomicAdd(&ctrl->work[2], merge);
    atomicMax(&ctrl->work[3], dmax);
#pragma unroll
    for (int k = 0; k < kHubSizes; ++k)
      if (hub[k]) atomicAdd(&ctrl->work[4 + k], hub[k]);
  }
}

// What a run's counting kernels read (instrumentation): work[0] += entries
// streamed through hash tables, work[1] += entries hashed, work[2] += partners
// intersected by bitmaps too.  The groups and the streams are told apart by the
// rules of the counting kernels (count.cu, bits.cu): a group of a list shorter
// than `least` is not binned.  pskip or, where it is not nullptr, desc holds
// what is streamed.  One warp per vertex h.
template <bool PV>
__global__ void __launch_bounds__(kGroupThreads)
k_run_work(const int32_t *goff, const int32_t *part, const int32_t *pskip, const int2 *desc,
           const int2 *ldesc, const uint32_t *rec, int32_t n, int32_t least, Ctrl *ctrl) {
  grid_begin();
  if (aborted(ctrl)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (kGroupThreads / 32);
  unsigned long long lookups = 0, inserts = 0, pairs = 0;
  for (uint32_t h = (blockIdx.x * kGroupThreads + threadIdx.x) >> 5; h < (uint32_t)n;
       h += warps) {
    const int32_t pb = load(goff + h), pe = load(goff + h + 1), dh = load(ldesc + h).y;
    if (pe == pb || dh < least) continue;  // uniform
    const bool bits = rec && bits_group<PV>(load(rec + h), pe - pb);
    if (lane == 0) inserts += (unsigned)dh;
    for (int32_t i = pb + lane; i < pe; i += 32) {
      int32_t ds;
      if (desc) {
        ds = load(desc + i).y & 0xffff;
      } else {
        const int32_t l = load(part + i), skip = load(pskip + i);
        const uint32_t rl = bits ? load(rec + l) : 0u;
        ds = load(ldesc + l).y;
        if (bits_used<PV>(rl, skip, ds)) {
          ds = 8 * (int32_t)(rl & kBitTbMask);
          ++pairs;
        }
        ds = max(ds - 8 * skip, 0);
      }
      lookups += (unsigned)ds;
    }
  }
  for (int o = 16; o; o >>= 1) {
    lookups += __shfl_xor_sync(0xffffffffu, lookups, o);
    inserts += __shfl_xor_sync(0xffffffffu, inserts, o);
    pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
  }
  if (lane == 0) {
    atomicAdd(&ctrl->work[0], lookups);
    atomicAdd(&ctrl->work[1], inserts);
    atomicAdd(&ctrl->work[2], pairs);
  }
}

uint32_t group_grid(uint32_t m_bound) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t want = (m_bound + kGroupThreads * 8 - 1) / (kGroupThreads * 8);
  return max(1u, min(want, (uint32_t)(sms > 0 ? sms : 1) * 8));
}

}  // namespace

static uint32_t num_sms() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (uint32_t)(sms > 0 ? sms : 1);
}

void launch_sort_lists(int32_t *col, const int32_t *off, const int32_t *voff, int32_t n,
                       Ctrl *ctrl, int32_t *col4, int32_t *queue, int32_t *dlen,
                       int32_t *dcorr, int2 *ldesc, const GroupOut *emit, cudaStream_t st) {
  const ListOut o{col4, emit ? nullptr : dlen, dcorr, ldesc, ctrl};
  const uint32_t warps = num_sms() * 8u * kListWarps;
  uint32_t per = 4;
  while (per < 32 && per * warps < (uint32_t)n) per <<= 1;
  const uint32_t chunks = ((uint32_t)n + per - 1) / per;
  const uint32_t grid = max(1u, min((chunks + kListWarps - 1) / kListWarps, num_sms() * 8u));
  const GroupOut g = emit ? *emit : GroupOut{};
  const auto lists = emit ? k_sort_lists<true> : k_sort_lists<false>;
  const auto long_lists = emit ? k_sort_long_lists<true> : k_sort_long_lists<false>;
  launch(lists, grid, kListThreads, 0, st, col, off, voff, n, per, o, g, queue);
  launch(long_lists, num_sms() * kLongListBlocks, kLongListThreads, 0, st, col, off, voff, n, o, g,
         queue);
}

void launch_fix_repeats(const int32_t *off, int32_t n, const int32_t *dcorr, const int32_t *rank,
                        Ctrl *ctrl, int32_t *row, int32_t *deg, cudaStream_t st) {
  launch(k_fix_repeats, num_sms() * 8u, kListThreads, 0, st, off, n, dcorr, rank, ctrl, row, deg);
}

void launch_group_keys(const int32_t *row, const int32_t *col4, const int32_t *off,
                       const int2 *ldesc, const int32_t *len, uint32_t m_bound, int b, int passes,
                       int32_t heavy_ratio_pct, bool whole, Ctrl *ctrl, uint64_t *gkeys,
                       uint32_t *hist, cudaStream_t st) {
  const auto kernel = whole ? k_group_keys<true> : k_group_keys<false>;
  launch(kernel, group_grid(m_bound), kGroupThreads, 0, st, row, col4, off, ldesc, len, b, passes,
         heavy_ratio_pct, ctrl, gkeys, hist);
}

void launch_work(const int32_t *off, const int32_t *goff, const int32_t *part,
                 const int32_t *pskip, int32_t n, Ctrl *ctrl, cudaStream_t st, int32_t shard,
                 int32_t shards) {
  const uint32_t lanes = n > (1 << 28) ? (1u << 30) : (uint32_t)n * 4u;  // grid is capped anyway
  launch(k_work, group_grid(lanes), kGroupThreads, 0, st, off, goff, part, pskip, n, ctrl,
         (uint32_t)shard, (uint32_t)shards);
}

void launch_run_work(const int32_t *goff, const int32_t *part, const int32_t *pskip,
                     const int2 *desc, const int2 *ldesc, const uint32_t *rec, int32_t n,
                     int32_t least, bool per_vertex, Ctrl *ctrl, cudaStream_t st) {
  const auto kernel = per_vertex ? k_run_work<true> : k_run_work<false>;
  const uint32_t lanes = n > (1 << 28) ? (1u << 30) : (uint32_t)n * 4u;  // grid is capped anyway
  launch(kernel, group_grid(lanes), kGroupThreads, 0, st, goff, part, pskip, desc, ldesc, rec, n,
         least, ctrl);
}

}  // namespace tc
