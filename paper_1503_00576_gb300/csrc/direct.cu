// direct.cu -- the counting sorts of the forward lists and the partner
// groups, and the vertex order they need (single-pass preprocessing).
//
// The radix passes of preprocess.cu move every 8-byte key three times per
// sort.  Both sorts only group: the order within a forward list does not
// matter (each list is sorted on its own later), nor that within a partner
// group, nor that of vertices of equal degree.  So each of them can be one
// counting sort with a counter per vertex: count by atomics, scan, scatter.
//
//   rank classes   the order of Sec. II-B up to ties: vertices by degree
//                  class (the degree itself below 256, then 32 classes per
//                  octave), counted per CTA in shared memory, so that the
//                  global counters see one atomic per CTA and class
//   orient         each key from its lower rank; the place in the owner's
//                  list comes from the atomic that counts its out-degree
//   lists          the scatter into the column array
//   groups         the scatter of the edges that the list sort emitted
//                  (group.cu) into their partner groups
//
// An atomic and a scattered write per key cost less than three passes while
// the counters and the array written to stay in L2; past that, a list's
// entries reach DRAM one 32-byte sector each (kDirectMaxPairs has both
// sides measured), and unless very many pairs share very few counters
// (kCrowdedMean).  R-MAT scale 20, 16.8M pairs: orient 244 us, lists 169,
// groups 243, classes 12; the radix passes of the three sorts took 690 and
// the group keys 89.
#include "tc_common.cuh"

namespace tc {
namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 8;

// ---------------------------------------------------------------------------
// rank classes
// ---------------------------------------------------------------------------
constexpr int kRankPer = 8;                       // vertices per thread and tile
constexpr int kRankTile = kThreads * kRankPer;
static_assert(2 * kRankClasses <= 256 * kMaxPasses, "class counters live in the histograms");
static_assert(256 + (31 - 8) * 32 <= kRankClasses, "every degree has a class");

__device__ __forceinline__ uint32_t rank_class(uint32_t d) {
  if (d < 256u) return d;
  const int e = 31 - __clz((int)d);  // >= 8
  return 256u + (uint32_t)(e - 8) * 32u + ((d >> (e - 5)) & 31u);
}

// Vertices per degree class.
__global__ void __launch_bounds__(kThreads)
k_rank_hist(const int32_t *deg, int32_t n, uint32_t *__restrict__ hist) {
  grid_begin();
  __shared__ uint32_t s_cnt[kRankClasses];
  for (int i = threadIdx.x; i < kRankClasses; i += kThreads) s_cnt[i] = 0;
  __syncthreads();
  const uint32_t stride = gridDim.x * kThreads;
  for (uint32_t v = blockIdx.x * kThreads + threadIdx.x; v < (uint32_t)n; v += stride)
    atomicAdd(&s_cnt[rank_class((uint32_t)load(deg + v))], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < kRankClasses; i += kThreads)
    if (s_cnt[i]) atomicAdd(&hist[i], s_cnt[i]);
}

// rank[v]: first rank of v's class (every CTA scans the class counts for
// itself), plus the places its tile reserved in the class, plus v's place
// within the tile.
__global__ void __launch_bounds__(kThreads)
k_rank_assign(const int32_t *deg, int32_t n, const uint32_t *hist,
              uint32_t *__restrict__ cursor, int32_t *__restrict__ rank) {
  grid_begin();
  constexpr int PER = kRankClasses / kThreads;
  __shared__ uint32_t s_start[kRankClasses], s_cnt[kRankClasses], s_warp[kThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t h[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    h[i] = load(hist + tid * PER + i);
    sum += h[i];
  }
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t run = incl - sum;
  for (int w = 0; w < warp; ++w) run += s_warp[w];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    s_start[tid * PER + i] = run;
    run += h[i];
  }
  const uint32_t tiles = ((uint32_t)n + kRankTile - 1) / kRankTile;
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    for (int i = tid; i < kRankClasses; i += kThreads) s_cnt[i] = 0;
    __syncthreads();
    uint32_t c[kRankPer], at[kRankPer];
#pragma unroll
    for (int i = 0; i < kRankPer; ++i) {
      const uint32_t v = tile * kRankTile + i * kThreads + tid;
      if (v < (uint32_t)n) {
        c[i] = rank_class((uint32_t)load(deg + v));
        at[i] = atomicAdd(&s_cnt[c[i]], 1u);
      }
    }
    __syncthreads();
    for (int i = tid; i < kRankClasses; i += kThreads) {
      const uint32_t cnt = s_cnt[i];
      if (cnt) s_cnt[i] = s_start[i] + atomicAdd(&cursor[i], cnt);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRankPer; ++i) {
      const uint32_t v = tile * kRankTile + i * kThreads + tid;
      if (v < (uint32_t)n) rank[v] = (int32_t)(s_cnt[c[i]] + at[i]);
    }
    __syncthreads();  // s_cnt is reused
  }
}

// ---------------------------------------------------------------------------
// forward lists
// ---------------------------------------------------------------------------
// Each key as (lower rank) << b | (higher rank), with its place in the
// owner's list; self-loops and dropped pairs (the sentinel) stay as holes.
__global__ void __launch_bounds__(kThreads)
k_direct_orient(const uint64_t *keys, int b, const int32_t *rank,
                uint64_t *__restrict__ okeys, int32_t *__restrict__ place,
                int32_t *__restrict__ outdeg, const Ctrl *ctrl) {
  grid_begin();
  const uint32_t m = ctrl->m_in;
  const uint64_t sentinel = (1ull << (2 * b)) - 1, mask = (1ull << b) - 1;
  const uint32_t stride = gridDim.x * kThreads;
  for (uint32_t i0 = blockIdx.x * kThreads + threadIdx.x; i0 < m; i0 += kUnroll * stride) {
    uint64_t k[kUnroll];
    uint32_t ra[kUnroll], rc[kUnroll];
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      const uint32_t i = i0 + q * stride;
      k[q] = i < m ? (uint64_t)__ldcs(reinterpret_cast<const unsigned long long *>(keys) + i)
                   : sentinel;
    }
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      ra[q] = rc[q] = 0;
      if (k[q] != sentinel) {
        ra[q] = (uint32_t)load(rank + (uint32_t)(k[q] >> b));
        rc[q] = (uint32_t)load(rank + (uint32_t)(k[q] & mask));
      }
    }
    int32_t at[kUnroll];
#pragma unroll
    for (int q = 0; q < kUnroll; ++q)
      at[q] = k[q] != sentinel ? atomicAdd(&outdeg[min(ra[q], rc[q])], 1) : 0;
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      const uint32_t i = i0 + q * stride;
      if (i >= m) break;
      const uint64_t o = k[q] == sentinel
                             ? kHole
                             : ((uint64_t)min(ra[q], rc[q]) << b) | max(ra[q], rc[q]);
      __stcs(reinterpret_cast<unsigned long long *>(okeys) + i, (unsigned long long)o);
      __stcs(place + i, at[q]);
    }
  }
}

// The column array: each entry to its place in its owner's list.
__global__ void __launch_bounds__(kThreads)
k_direct_lists(const uint64_t *okeys, const int32_t *place, int b,
               const int32_t *off, int32_t *__restrict__ col,
               const Ctrl *ctrl) {
  grid_begin();
  if (aborted(ctrl)) return;  // a wait of this call ran out: off is not complete
  const uint32_t m = ctrl->m_in;
  const uint32_t mask = (uint32_t)((1ull << b) - 1);
  const uint32_t stride = gridDim.x * kThreads;
  for (uint32_t i0 = blockIdx.x * kThreads + threadIdx.x; i0 < m; i0 += kUnroll * stride) {
    uint64_t k[kUnroll];
    int32_t at[kUnroll];
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      const uint32_t i = i0 + q * stride;
      k[q] = i < m ? (uint64_t)__ldcs(reinterpret_cast<const unsigned long long *>(okeys) + i)
                   : kHole;
      at[q] = i < m ? __ldcs(place + i) : 0;
    }
#pragma unroll
    for (int q = 0; q < kUnroll; ++q)
      if (k[q] != kHole) at[q] += load(off + (uint32_t)(k[q] >> b));
#pragma unroll
    for (int q = 0; q < kUnroll; ++q)
      if (k[q] != kHole) col[at[q]] = (int32_t)((uint32_t)k[q] & mask);
  }
}

// ---------------------------------------------------------------------------
// partner groups
// ---------------------------------------------------------------------------
// Every emitted edge to its group: the group's own edges (h the owner) at
// the places they were numbered with, from the group's start; the others
// from its end down, through the counter that counted them.  The highest
// ranks' counters are hit by every second edge of an R-MAT graph, so a tile
// counts its edges to them in shared memory and takes their places with one
// atomic per rank (R-MAT scale 16, 2.5M edges: 130 us without, 38 with).
constexpr int kHotRanks = 4096;
constexpr int kGroupTile = kThreads * kUnroll;

__global__ void __launch_bounds__(kThreads)
k_direct_groups(const uint64_t *gkeys, int b, int32_t n,
                const int32_t *goff, int32_t *__restrict__ gcnt,
                int32_t *__restrict__ part, int32_t *__restrict__ pskip,
                const int2 *ldesc, int2 *__restrict__ desc,
                const Ctrl *ctrl) {
  grid_begin();
  __shared__ int32_t s_hot[kHotRanks];  // the tile's edges per rank, then the counter's old value
  if (aborted(ctrl)) return;
  const int tid = threadIdx.x;
  const uint32_t m = ctrl->m;
  const uint32_t mask = (uint32_t)((1ull << b) - 1);
  const uint32_t hot = (uint32_t)max(n - kHotRanks, 0);  // first of the hot ranks
  for (uint32_t t0 = blockIdx.x * kGroupTile; t0 < m; t0 += gridDim.x * kGroupTile) {
    for (int i = tid; i < kHotRanks; i += kThreads) s_hot[i] = 0;
    __syncthreads();
    uint64_t k[kUnroll];
    int32_t at[kUnroll];
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      const uint32_t i = t0 + q * kThreads + tid;
      k[q] = i < m ? (uint64_t)__ldcs(reinterpret_cast<const unsigned long long *>(gkeys) + i)
                   : kHole;
    }
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      at[q] = 0;
      if (k[q] == kHole) continue;
      const uint32_t h = (uint32_t)(k[q] >> b) & mask;
      if (k[q] & kOwnEdge)
        at[q] = load(goff + h) + (int32_t)((k[q] & ~kOwnEdge) >> kSkipShift);
      else if (h >= hot)
        at[q] = atomicAdd(&s_hot[h - hot], 1);
      else
        at[q] = load(goff + h + 1) - atomicSub(&gcnt[h], 1);
    }
    __syncthreads();
    for (int i = tid; i < kHotRanks; i += kThreads) {
      const int32_t c = s_hot[i];
      if (c) s_hot[i] = atomicSub(&gcnt[hot + i], c);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kUnroll; ++q) {
      if (k[q] == kHole) continue;
      const uint32_t h = (uint32_t)(k[q] >> b) & mask;
      if (!(k[q] & kOwnEdge) && h >= hot) at[q] += load(goff + h + 1) - s_hot[h - hot];
      const uint32_t l = (uint32_t)k[q] & mask;
      const int32_t skip = k[q] & kOwnEdge ? 0 : (int32_t)(k[q] >> kSkipShift);
      part[at[q]] = (int32_t)l;
      if (desc) desc[at[q]] = stream_desc(load(ldesc + l), skip, 0xffffu);
      else pskip[at[q]] = skip;
    }
    __syncthreads();  // s_hot is emptied again
  }
}

uint32_t sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (uint32_t)(sms > 0 ? sms : 1);
}

uint32_t items_grid(uint32_t items) {
  const uint32_t want = (items + kThreads * kUnroll - 1) / (kThreads * kUnroll);
  return max(1u, min(want, sm_count() * 16u));
}

}  // namespace

void launch_rank_classes(const int32_t *deg, int32_t n, uint32_t *counters, int32_t *rank,
                         cudaStream_t st) {
  const uint32_t tiles = ((uint32_t)n + kRankTile - 1) / kRankTile;
  const uint32_t grid = max(1u, min(tiles, sm_count() * 8u));
  launch(k_rank_hist, grid, kThreads, 0, st, deg, n, counters);
  launch(k_rank_assign, grid, kThreads, 0, st, deg, n, counters, counters + kRankClasses, rank);
}

void launch_direct_orient(const uint64_t *keys, uint32_t m_in, int b, const int32_t *rank,
                          uint64_t *okeys, int32_t *place, int32_t *outdeg, Ctrl *ctrl,
                          cudaStream_t st) {
  launch(k_direct_orient, items_grid(m_in), kThreads, 0, st, keys, b, rank, okeys, place, outdeg,
         ctrl);
}

void launch_direct_lists(const uint64_t *okeys, const int32_t *place, uint32_t m_in, int b,
                         const int32_t *off, int32_t *col, Ctrl *ctrl, cudaStream_t st) {
  launch(k_direct_lists, items_grid(m_in), kThreads, 0, st, okeys, place, b, off, col, ctrl);
}

void launch_direct_groups(const uint64_t *gkeys, uint32_t m_bound, int b, int32_t n,
                          const int32_t *goff, int32_t *gcnt, int32_t *part, int32_t *pskip,
                          const int2 *ldesc, int2 *desc, Ctrl *ctrl, cudaStream_t st) {
  launch(k_direct_groups, items_grid(m_bound), kThreads, 0, st, gkeys, b, n, goff, gcnt, part,
         pskip, ldesc, desc, ctrl);
}

}  // namespace tc
