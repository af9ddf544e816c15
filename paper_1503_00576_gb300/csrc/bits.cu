// bits.cu -- intersections of long lists as bitmaps of the top ranks.
//
// In the (degree, id) order of Sec. II-B the entries of a long forward list
// crowd among the highest ranks: on the R-MAT graphs of the benchmarks 60% to
// 75% of all hash lookups look for one of the 4096 highest ranks in a list
// that holds at least 32 of them.  For such a list a bitmap of those ranks is
// no longer than the entries, and the intersection of two of them is an AND
// and a bit count over 512 bytes, one 16-byte load per lane: no hashing, no
// shared memory, every load coalesced.
//
//   bitmaps   list l (len entries, sorted) gets one if at least
//             kBitMinBlocks of its 32-byte blocks lie among the top ranks;
//             the bitmap stands for its entries from block tb on, the first
//             block that lies there whole.
//   edges     for the edge of group h and partner l, both with bitmaps, the
//             hash path (count.cu) streams N+(l) only up to block tb of l,
//             and the rest is counted here: popcount(F(h) & B(l)), F(h)
//             being B(h) completed by the up to 7 entries of its block tb - 1
//             that are top ranks too (those of l are streamed, so none is
//             counted twice).  A slot of the region holds B, then F.
//   use       decided per group by bits_group() and per edge by bits_used()
//             alone, from what both paths have, so that they agree.
//
// T only an edge costs 22 instructions of a warp and 512 bytes from L2 (R-MAT
// scale 21, 91M edges: 48M edges in 1.8 ms, about 11 clocks each on an SM,
// L2 60% busy; the same edges took 8 of 13.8 ms by hashing).
#include "tc_common.cuh"

namespace tc {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWords = kBitCols / 32;
constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
// The per-vertex kernel's CTAs: eight warps share one set of hub counters, and a
// warp's queue and planes one buffer, so that 110 KB of an SM stay L1, where the
// loads in flight are held (four CTAs of four warps with both: 3.8 ms at R-MAT
// scale 24, five 5.2 ms, these 3.3 ms).
constexpr int kVertexThreads = 256;
static_assert(kWords == 4 * 32, "a lane holds four words of a bitmap");

// First of the top ranks: column 0 of the bitmaps.
__device__ __forceinline__ int32_t bits_base(int32_t n) { return max(n - kBitCols, 0); }

// One warp per queued list (group.cu: every list longer than 64 entries; the
// first n_warp_lists of the array, and n_cta_lists from its end down): the
// bitmap goes to slot i + 1 of the region, its record to rec[v].  A list whose
// slot does not fit the region has none.  Slot 0 is the empty bitmap.
template <bool PV>
__global__ void __launch_bounds__(kThreads)
k_bits_build(const int32_t *queue, int32_t n, const int2 *ldesc,
             const int32_t *col4, const int32_t *goff, uint32_t slots,
             uint32_t *__restrict__ bits, uint32_t *__restrict__ rec, int2 *__restrict__ items,
             Ctrl *ctrl, uint32_t shard, uint32_t shards) {
  grid_begin();
  __shared__ uint32_t s_bits[kWarps][kWords];
  if (aborted(ctrl)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t n_warp = ctrl->n_warp_lists;
  const uint32_t count = min(n_warp + ctrl->n_cta_lists, slots - 1u);
  const int32_t base = bits_base(n);
  uint32_t *sb = s_bits[warp];
  uint4 *rows = reinterpret_cast<uint4 *>(bits);  // 32 per bitmap, two bitmaps per slot
  if (blockIdx.x == 0 && warp == 0) rows[lane] = make_uint4(0, 0, 0, 0);
  // the groups of up to 32 lists (one per lane) before their items are placed
  int pending = 0;
  int32_t group = 0;
  uint32_t from = 0, to = 0;
  auto place_items = [&] {
    const uint32_t mine = lane < pending ? (to - from + kBitRange<PV> - 1) / kBitRange<PV> : 0u;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    uint32_t at = 0;
    if (lane == 31) at = atomicAdd(&ctrl->n_bit_items, incl);
    at = __shfl_sync(kFull, at, 31) + incl - mine;
    for (uint32_t k = 0; k < mine; ++k)
      items[at + k] = make_int2(group, (int32_t)(from + k * kBitRange<PV>));
    pending = 0;
  };
  for (uint32_t i = blockIdx.x * kWarps + warp; i < count; i += gridDim.x * kWarps) {
    const int32_t v = load(queue + (i < n_warp ? i : (uint32_t)n - 1u - (i - n_warp)));
    const int2 ld = load(ldesc + v);
    const int32_t len = ld.y, blocks = (len + 7) >> 3;
    const int32_t *list = col4 + 4ll * ld.x;
    // enough top ranks at all?
    constexpr int32_t kLeast = 8 * (kBitMinBlocks<PV> - 1) + 1;
    if (blocks < kBitMinBlocks<PV> || load(list + len - kLeast) < base) continue;
    for (int w = lane; w < kWords; w += 32) sb[w] = 0u;
    __syncwarp();
    int32_t top = 0;  // entries before the first top rank
    for (int32_t e1 = len; e1 > 0; e1 -= 32) {
      const int32_t e = e1 - 1 - lane;
      const int32_t x = e >= 0 ? load(list + e) : -1;
      const bool in = x >= base;  // lanes 0 .. k-1: the list is sorted
      if (in) atomicOr(&sb[(uint32_t)(x - base) >> 5], 1u << ((x - base) & 31));
      const int k = __popc(__ballot_sync(kFull, in));
      if (k < 32) {
        top = e1 - k;
        break;
      }
    }
    __syncwarp();
    const int32_t tb = (top + 7) >> 3;
    if (blocks - tb >= kBitMinBlocks<PV> && tb <= (int32_t)kBitTbMask) {
      uint4 *dst = rows + (size_t)(i + 1u) * 64 + lane;
      dst[32] = reinterpret_cast<const uint4 *>(sb)[lane];  // F
      __syncwarp();
      if (lane < 8 * tb - top) {  // top ranks of the block before tb: streamed
        const int32_t c = load(list + top + lane) - base;
        atomicAnd(&sb[c >> 5], ~(1u << (c & 31)));
      }
      __syncwarp();
      dst[0] = reinterpret_cast<const uint4 *>(sb)[lane];  // B
      const uint32_t r = ((i + 1u) << kBitTbBits) | (uint32_t)tb;
      if (lane == 0) rec[v] = r;
      const int32_t gs = load(goff + v), ge = load(goff + v + 1);
      if (bits_group<PV>(r, ge - gs) && (uint32_t)v % shards == shard) {
        if (lane == pending) {
          group = v;
          from = (uint32_t)gs;
          to = (uint32_t)ge;
        }
        if (++pending == 32) place_items();
      }
    }
    __syncwarp();
  }
  if (pending) place_items();
}

// Carry-save adder: a + b + c = sum + 2 carry, bit by bit.
__device__ __forceinline__ void csa(uint32_t &sum, uint32_t &carry, uint32_t a, uint32_t b,
                                    uint32_t c) {
  const uint32_t x = a ^ b ^ c;
  carry = (a & b) | (c & (a | b));
  sum = x;
}

struct BitArgs {
  const int32_t *goff, *part, *pskip;
  const int2 *ldesc;
  const int32_t *col4;
  const uint32_t *rec, *bits;
  const int2 *items;
  int32_t n;
  Ctrl *ctrl;
  int64_t *t;
};

// The partners of a segment that are intersected by bitmaps: their slots and
// (per-vertex mode) themselves and their counts.
constexpr int kBatch = 8;  // partners loaded before any is added
template <bool PV>
struct __align__(16) Queue {
  uint32_t slot[kBitRange<PV> + kBatch];
  int32_t l[PV ? kBitRange<PV> : 1];
  uint16_t cnt[PV ? kBitRange<PV> + kBatch : 2];
};

// Fills the queue from partners [s, t), at most kBitRange<PV>, and pads it with
// the empty bitmap to whole batches; returns the number of partners.  All
// gathers of the segment are issued before any is used, so that a segment
// costs two memory latencies, not two per 32 partners.
template <bool PV>
__device__ __forceinline__ int fill_queue(const BitArgs &a, uint32_t s, uint32_t t,
                                          Queue<PV> &qu) {
  constexpr int N = (kBitRange<PV> + 31) / 32;
  const int lane = threadIdx.x & 31;
  int32_t l[N], skip[N], len[N];
  uint32_t r[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t e = s + 32 * i + lane;
    l[i] = e < t ? load(a.part + e) : -1;
    skip[i] = e < t ? load(a.pskip + e) : 0;
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    r[i] = l[i] >= 0 ? load(a.rec + l[i]) : 0u;
    len[i] = l[i] >= 0 ? load(a.ldesc + l[i]).y : 0;
  }
  int count = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (s + 32 * i >= t) break;  // uniform
    const bool use = bits_used<PV>(r[i], skip[i], len[i]);
    const uint32_t mask = __ballot_sync(kFull, use);
    const int at = count + __popc(mask & ((1u << lane) - 1u));
    if (use) {
      qu.slot[at] = r[i] >> kBitTbBits;
      if (PV) qu.l[at] = l[i];
    }
    count += __popc(mask);
  }
  if (lane < kBatch) qu.slot[count + lane] = 0u;
  __syncwarp();
  return count;
}

// The words of this lane of four queued partners' bitmaps.
__device__ __forceinline__ void load_four(const uint4 *lane_bits, const uint32_t *slot,
                                          uint4 *x) {
  const uint4 sl = *reinterpret_cast<const uint4 *>(slot);
  x[0] = load(lane_bits + (size_t)sl.x * 64);
  x[1] = load(lane_bits + (size_t)sl.y * 64);
  x[2] = load(lane_bits + (size_t)sl.z * 64);
  x[3] = load(lane_bits + (size_t)sl.w * 64);
}

// T only: Harley-Seal over the words of all partners a lane meets, whatever
// their group: six carry-save adders and one population count per two
// partners.
struct Sums {
  uint32_t ones, twos, fours;
  unsigned long long eights;
};

__device__ __forceinline__ uint32_t add_words(Sums &s, const uint4 &x, const uint32_t (&hw)[4]) {
  uint32_t ta, tb, f;
  csa(s.ones, ta, s.ones, x.x & hw[0], x.y & hw[1]);
  csa(s.ones, tb, s.ones, x.z & hw[2], x.w & hw[3]);
  csa(s.twos, f, s.twos, ta, tb);
  return f;
}

// Partners [s, t) of group h.
__device__ __forceinline__ void bits_total(const BitArgs &a, uint32_t rh, uint32_t s,
                                           uint32_t t, Queue<false> &qu, Sums &sums) {
  const uint4 *lane_bits = reinterpret_cast<const uint4 *>(a.bits) + (threadIdx.x & 31);
  const uint4 f = load(lane_bits + (size_t)(rh >> kBitTbBits) * 64 + 32);
  const uint32_t hw[4] = {f.x, f.y, f.z, f.w};
  const int count = fill_queue<false>(a, s, t, qu);
  if (count) {
    for (int c = 0; c < count; c += kBatch) {
      uint4 x[kBatch];
      load_four(lane_bits, qu.slot + c, x);
      load_four(lane_bits, qu.slot + c + 4, x + 4);
#pragma unroll
      for (int i = 0; i < kBatch; i += 2) {
        uint32_t e;
        const uint32_t f0 = add_words(sums, x[i], hw), f1 = add_words(sums, x[i + 1], hw);
        csa(sums.fours, e, sums.fours, f0, f1);
        sums.eights += (unsigned)__popc(e);
      }
    }
  }
  __syncwarp();  // the queue is filled again
}

// Per-vertex mode: per partner its own count (t(l)), per group their sum
// (t(h)), and per column how many partners matched there (t(w)), kept as
// eight bit planes per word (positional counts by carry-save adders) and
// emptied at the end of the group or range.
constexpr int kPlanes = 8;
static_assert(kBitRange<true> < 1 << kPlanes, "a range's partners fit the planes");

struct Planes {
  uint32_t p[4][kPlanes];
};

// The planes go to shared memory as they are, and every top rank of h's list
// (the only columns that can have matched; none before entry `from`) collects
// its bits: emptying costs in proportion to the list, not to the columns
// (turning all planes into byte counters first took 1000 instructions per
// group or range, three times the work of its partners).  used: partners
// added.  s_t: the CTA's counts of t(w), one per column (a pair adds at most
// one to each, so 32 bits hold them); straight to t in global memory they
// took a third of the kernel, all CTAs adding to the same few hubs.
__device__ __forceinline__ void empty_planes(const BitArgs &a, const Planes &pl, int32_t h,
                                             int32_t from, int used, uint32_t *sb,
                                             uint32_t *s_t) {
  const int lane = threadIdx.x & 31;
  const int np = 32 - __clz(used);  // planes in use
#pragma unroll
  for (int k = 0; k < kPlanes; ++k)
    if (k < np)  // uniform
      reinterpret_cast<uint4 *>(sb)[k * 32 + lane] =
          make_uint4(pl.p[0][k], pl.p[1][k], pl.p[2][k], pl.p[3][k]);
  __syncwarp();
  const int2 ld = load(a.ldesc + h);
  const int32_t *list = a.col4 + 4ll * ld.x;
  const int32_t base = bits_base(a.n);
  for (int32_t e = from + lane; e < ld.y; e += 32) {
    const int32_t x = load(list + e), c = x - base;
    if (c >= 0) {
      uint32_t cnt = 0;
#pragma unroll
      for (int k = 0; k < kPlanes; ++k)
        if (k < np) cnt += ((sb[k * kWords + (c >> 5)] >> (c & 31)) & 1u) << k;
      if (cnt) atomicAdd(&s_t[c], cnt);
    }
  }
  __syncwarp();  // sb is written again
}

// Four partners: their bits into the planes of 1 and 2, the fours to f, their
// counts to cnt (two per reduction: each is at most kBitCols < 2^16) and
// summed up.
__device__ __forceinline__ uint32_t add_four(Planes &pl, uint4 (&x)[4], const uint32_t (&hw)[4],
                                             uint32_t (&f)[4], uint16_t *cnt) {
  uint32_t n[4], sum = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[i].x &= hw[0];
    x[i].y &= hw[1];
    x[i].z &= hw[2];
    x[i].w &= hw[3];
    n[i] = (uint32_t)(__popc(x[i].x) + __popc(x[i].y) + __popc(x[i].z) + __popc(x[i].w));
  }
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    const uint32_t two = __reduce_add_sync(kFull, n[i] | n[i + 1] << 16);
    sum += (two & 0xffffu) + (two >> 16);
    if ((threadIdx.x & 31) == 0) *reinterpret_cast<uint32_t *>(cnt + i) = two;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t w[4], ta, tb;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = q == 0 ? x[i].x : q == 1 ? x[i].y : q == 2 ? x[i].z : x[i].w;
    csa(pl.p[q][0], ta, pl.p[q][0], w[0], w[1]);
    csa(pl.p[q][0], tb, pl.p[q][0], w[2], w[3]);
    csa(pl.p[q][1], f[q], pl.p[q][1], ta, tb);
  }
  return sum;
}

__device__ __forceinline__ void bits_vertex(const BitArgs &a, int32_t h, uint32_t rh, uint32_t s,
                                            uint32_t t, Queue<true> &qu, uint32_t *sb,
                                            uint32_t *s_t, unsigned long long &total) {
  const int lane = threadIdx.x & 31;
  const uint4 *lane_bits = reinterpret_cast<const uint4 *>(a.bits) + lane;
  const uint4 fh = load(lane_bits + (size_t)(rh >> kBitTbBits) * 64 + 32);
  const uint32_t hw[4] = {fh.x, fh.y, fh.z, fh.w};
  const int count = fill_queue<true>(a, s, t, qu);
  uint32_t sum = 0;  // matches of the segment (uniform; at most kBitRange kBitCols)
  if (count) {
    Planes pl;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < kPlanes; ++k) pl.p[q][k] = 0u;
    // four partners are added while the next four are on their way
    uint4 xa[4], xb[4];
    load_four(lane_bits, qu.slot, xa);
    for (int c = 0; c < count; c += kBatch) {
      uint32_t f0[4], f1[4];
      load_four(lane_bits, qu.slot + c + 4, xb);
      sum += add_four(pl, xa, hw, f0, qu.cnt + c);
      if (c + kBatch < count) load_four(lane_bits, qu.slot + c + kBatch, xa);
      sum += add_four(pl, xb, hw, f1, qu.cnt + c + 4);
      // the fours, and the eights rippled through the planes above
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t carry;
        csa(pl.p[q][2], carry, pl.p[q][2], f0[q], f1[q]);
#pragma unroll
        for (int k = 3; k < kPlanes; ++k) {
          const uint32_t up = pl.p[q][k] & carry;
          pl.p[q][k] ^= carry;
          carry = up;
        }
      }
    }
    __syncwarp();
    for (int i = lane; i < count; i += 32) {
      const uint32_t ci = qu.cnt[i];
      if (ci) atomicAdd((unsigned long long *)&a.t[qu.l[i]], (unsigned long long)ci);
    }
    __syncwarp();  // the planes take the queue's place
    if (sum) {
      empty_planes(a, pl, h, 8 * max((int32_t)(rh & kBitTbMask) - 1, 0), count, sb, s_t);
      if (lane == 0) atomicAdd((unsigned long long *)&a.t[h], (unsigned long long)sum);
      total += sum;
    }
  }
  __syncwarp();  // the queue is filled again
}

// Shared memory of a warp: its queue, and in the queue's place the planes that
// it empties.
template <bool PV>
constexpr __host__ __device__ size_t warp_bytes() {
  return PV && sizeof(uint32_t) * kPlanes * kWords > sizeof(Queue<PV>)
             ? sizeof(uint32_t) * kPlanes * kWords
             : sizeof(Queue<PV>);
}
constexpr size_t kVertexSmem =
    warp_bytes<true>() * (kVertexThreads / 32) + sizeof(uint32_t) * kBitCols;
static_assert(kVertexSmem <= 48 * 1024, "no attribute needed");

// One work item per warp in turn: at most kBitRange partners of one group,
// however large the group is.  (Ranges of the whole partner array, with a
// walk over the groups in them, spent half of the kernel on groups without
// bitmaps.)
template <bool PV>
__global__ void __launch_bounds__(PV ? kVertexThreads : kThreads, PV ? 2 : 8)
k_count_bits(const BitArgs a) {
  grid_begin();
  constexpr int THREADS = PV ? kVertexThreads : kThreads, WARPS = THREADS / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char *s_mine = smem + warp_bytes<PV>() * (threadIdx.x >> 5);
  Queue<PV> &s_queue = *reinterpret_cast<Queue<PV> *>(s_mine);
  uint32_t *s_planes = reinterpret_cast<uint32_t *>(s_mine);  // once the queue is done with
  uint32_t *s_t = reinterpret_cast<uint32_t *>(smem + warp_bytes<PV>() * WARPS);  // PV only
  Ctrl *ctrl = a.ctrl;
  if (aborted(ctrl) || ctrl->n_bit_items == 0u) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t items = ctrl->n_bit_items;
  if (PV) {
    for (int c = threadIdx.x; c < kBitCols; c += THREADS) s_t[c] = 0u;
    __syncthreads();
  }
  unsigned long long total = 0;
  Sums sums{0u, 0u, 0u, 0ull};
  for (uint32_t i = blockIdx.x * WARPS + warp; i < items; i += gridDim.x * WARPS) {
    const int2 item = load(a.items + i);
    const uint32_t s = (uint32_t)item.y;
    const uint32_t t = min(s + kBitRange<PV>, (uint32_t)load(a.goff + item.x + 1));
    const uint32_t rh = load(a.rec + item.x);
    if constexpr (PV)
      bits_vertex(a, item.x, rh, s, t, s_queue, s_planes, s_t, total);
    else
      bits_total(a, rh, s, t, s_queue, sums);
  }
  if (PV) {
    __syncthreads();
    const int32_t base = bits_base(a.n);
    for (int c = threadIdx.x; c < kBitCols; c += THREADS)
      if (s_t[c]) atomicAdd((unsigned long long *)&a.t[base + c], (unsigned long long)s_t[c]);
  } else {
    total = 8ull * sums.eights + 4u * (unsigned)__popc(sums.fours) +
            2u * (unsigned)__popc(sums.twos) + (unsigned)__popc(sums.ones);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
  }
  if (lane == 0 && total) atomicAdd(&ctrl->total, total);
}

uint32_t sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (uint32_t)(sms > 0 ? sms : 1);
}

}  // namespace

void launch_bits_build(const int32_t *queue, int32_t n, const int2 *ldesc, const int32_t *col4,
                       const int32_t *goff, uint32_t slots, bool per_vertex, uint32_t *bits,
                       const BitItems &items, Ctrl *ctrl, cudaStream_t st, int32_t shard,
                       int32_t shards) {
  const auto kernel = per_vertex ? k_bits_build<true> : k_bits_build<false>;
  launch(kernel, sm_count() * 8u, kThreads, 0, st, queue, n, ldesc, col4, goff, slots, bits,
         items.rec, items.items, ctrl, (uint32_t)shard, (uint32_t)shards);
}

void launch_count_bits(const int2 *ldesc, const int32_t *col4, const int32_t *goff,
                       const int32_t *part, const int32_t *pskip, const BitItems &items,
                       const uint32_t *bits, int32_t n, Ctrl *ctrl, int64_t *t, cudaStream_t st) {
  const BitArgs a{goff, part, pskip, ldesc, col4, items.rec, bits, items.items, n, ctrl, t};
  if (t)
    launch(k_count_bits<true>, sm_count() * 2u, kVertexThreads, kVertexSmem, st, a);
  else
    launch(k_count_bits<false>, sm_count() * 8u, kThreads, warp_bytes<false>() * kWarps, st, a);
}

}  // namespace tc
