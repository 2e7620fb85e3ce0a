// Several levels of the median k-d partition (Sec. 4.1 of arXiv 2404.02826) in
// two launches, for 16-bit codes split on axis depth mod 3.
//
// A level of the level-by-level path (k_tree.cu, k_scatter.cu) moves every
// particle once and takes eight launches.  Here the split planes of up to
// kSplitMaxLevels levels are found without moving anything - a byte per
// particle holds its node below the subroot (the node of depth `depth` it lies
// in) - and then every particle moves once, straight into its node of depth +
// levels.
//
// k_split: one persistent CTA per SM, as many as start in time (join); CTA c of
// those owns the contiguous positions [c * chunk, (c + 1) * chunk), and a
// segment is what a CTA holds of one subroot.  Per level:
//   A     every particle takes its child of the level above (code against the
//         split plane) and is counted in a shared histogram of its code on the
//         level's axis, one run of bins per node; the bins of all nodes share
//         16384 counters (fewer where a small input has no room for them), so
//         a bin spans 2^shift codes with the smallest shift
//         that fits the nodes' real code ranges (0 for most of them);
//   sel1  every CTA scans the summed histogram: the bin of every node's median;
//   B     only with shift > 0: the particles of those bins are counted per code
//         (with shift 0 the counters of A already hold every code);
//   sel2  every CTA derives the split code v and, from the counts of the
//         segments before its own, how many of its particles with code v go
//         left: all, none, or (one segment per node) the first `quota` in
//         position order.  The next A lists those ties as it meets them and
//         moves the first `quota` over at its end; where they are too many for a
//         list, it counts them by warp in two more passes (count_ties).
// Then F gives every particle its final child and counts the children.  Every
// step between two grid barriers reads only what was complete before the first
// of them; a barrier costs 1.3 us.
//
// k_move: ranks each tile's particles within their children (warp ballots),
// gathers them in shared memory in runs aligned as their destinations are, and
// stores 16 bytes at a time.
// All waits are bounded.
//
// What bounds it (2^27 particles, 13-bit codes, two launches of six levels): a
// pass A reads two code arrays and the node bytes and writes those, 6 bytes a
// particle, in 115 us (7.0 TB/s, the copy rate of the memory and what L2
// keeps); level 0 reads one array in 70 us, bound by the shared-memory atomics;
// B 80 us where a level needs it.  A launch takes 1.25 to 1.35 ms from board to
// board; the move 0.53 ms (13 bytes a particle, 3.3 TB/s), bound by its
// instructions (77 a row of 32 particles) and shared-memory passes (18 a row).
// Twelve levels: 3.6 to 3.8 ms, against 5.9 ms level by level (96 launches).  At
// 2^20 particles the seven levels take 0.11 ms in two launches, against 0.28 ms
// in 42.
#include <cstddef>
#include <cstdint>

#include "pc_internal.cuh"

namespace pcx {
namespace {

constexpr int kT = 1024;
constexpr int kW = kT / 32;
constexpr uint32_t kBins = kSplitBins;
constexpr uint32_t kLow = kSplitLow;
constexpr uint32_t kHalf = 1u << (kSplitMaxLevels - 1);  // nodes that split, at most
constexpr uint32_t kNodes = 1u << kSplitMaxLevels;        // children of the last level, at most
constexpr uint32_t kStep = 8u * kT;                       // particles of one step of a pass
constexpr uint32_t kTieBins = 2048;                       // digit of the tie selection by a block
constexpr uint32_t kTieWarp = 1024;                       // a warp selects among at most this many ties
constexpr uint32_t kGridSpin = 1u << 21;                  // polls of a grid barrier before it gives up

// State of one segment's nodes.  With several segments in a CTA it is kept in
// global memory between the steps (the first kStateWords words).
struct NodeTab {
  uint32_t blo[2][3][kHalf], bhi[2][3][kHalf];  // code bounds of the nodes, by parity of the level
  uint32_t plane[kHalf];  // a particle goes right if 2 code + 1 >= plane; odd: 2 v + 1, ties at v are listed
  uint32_t quota[kHalf];  // listed ties that go left
  uint32_t mine[kHalf];   // the segment's ties
  uint32_t bk[kHalf];     // median bin (code >> shift)
  uint32_t below[kHalf];  // particles of the node in lower bins
  // derived, not kept
  int32_t off[kHalf];     // bin of code x: off + (x >> shift)
  uint32_t roff[kHalf], rcnt[kHalf];  // node's place in the subroot
  uint32_t lbase[kHalf], cursor[kHalf];  // the node's part of the tie list, and its end so far; without a
                                         // list: the warp whose ties go both ways, and how many go left
};
constexpr uint32_t kStateWords = kSplitStateWords;
static_assert(kStateWords == 17 * kHalf, "kept part of NodeTab");

struct Misc {
  uint32_t c, members;          // this CTA among those that take part
  uint32_t chunk, part;         // positions of a CTA; of one of the move
  uint32_t s0, s1;              // subroots of this CTA
  uint32_t soff, scnt;          // current subroot
  uint32_t b0, b1;              // current segment
  uint32_t clo;                 // first CTA of the current subroot
  uint32_t shift, nbins;
  uint32_t ties, many;          // ties of the segment; whether a node has more than a warp selects among
  uint32_t counted;             // whether they are counted by warp instead of listed
  uint32_t fd, fbefore;         // tie selection: digit, ties below it
  uint32_t wt[kW + 1];
  uint32_t wh[kW][32];
  uint32_t th[kTieBins];
};

struct Smem {
  Misc M;
  NodeTab N;
  alignas(16) uint32_t bins[kBins];
  // sel1: prefixes of the summed histogram; B: counts per code; A, F: the tie list or the ties by
  // warp and node
  alignas(16) uint32_t sum[kBins];
};
static_assert(kW * kHalf <= kBins, "ties by warp and node");
static_assert(sizeof(Smem) <= 232448, "shared memory of one CTA");
static_assert(offsetof(Smem, bins) % 16 == 0 && offsetof(Smem, sum) % 16 == 0, "16-byte accesses");

// Positions of a CTA when m take part, a multiple of 16, and of a CTA of the move.
__device__ __forceinline__ uint32_t chunk_of(uint64_t n, uint32_t m) { return uint32_t(((n + m - 1) / m + 15u) & ~15ull); }
__device__ __forceinline__ uint32_t part_size(uint32_t chunk) {
  return ((chunk + kSplitParts - 1) / kSplitParts + 31u) & ~31u;
}

// The CTAs wait for one another, so those that take part have to be running, and the launch
// does not ask for all of them to be placed at once: a kernel of somebody else's that stays
// on an SM would hold up such a launch, and a stream with fewer SMs than the device would
// refuse it.  Instead the CTAs count themselves as they start (join), and the first to have
// waited as long as the missing ones would save (in cycles: 0.49 a particle and level on one
// CTA, shared by the k that came instead of all; kJoinLeast to kJoinMost), or the last of
// all, closes the count: the k that came split the work, one that starts later leaves.  Nobody
// waits for a CTA that has not started, and every wait ends: each CTA closes the count itself
// when its time is up.  The count starts ahead of the wait for the kernel before, so that it
// is complete by then where all come at once, the usual case.
// A cooperative launch took as long: 2^20 particles 166.0 us a call, so 165.7; 3,000,017 with
// the permutation 265.2, so 264.8; a batch of 48 snapshots 4.32 ms, so 4.35.
constexpr uint64_t kJoinLeast = 20000;         // cycles, about 10 us
constexpr uint64_t kJoinMost = 100000000;      // about 50 ms
constexpr uint32_t kJoinClosed = 0x80000000u;  // bit of the count

__device__ __forceinline__ uint32_t join_count(const SplitLaunch &a) {
  uint32_t m;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(m) : "l"(a.sync + 2) : "memory");
  return m;
}
__device__ __forceinline__ void join_close(const SplitLaunch &a, uint32_t m) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.sync + 2), "r"(m) : "memory");
}
// Thread 0: `mine` CTAs came before this one; how many take part, if that is known soon (else 0).
__device__ __forceinline__ uint32_t join(const SplitLaunch &a, uint32_t &mine) {
  mine = atomicAdd(a.sync + 1, 1u);
  if (mine + 1u == gridDim.x) {
    join_close(a, gridDim.x);
    return gridDim.x;
  }
  uint32_t m = 0;
  for (int i = 0; i < 8 && !m && !(mine & kJoinClosed); ++i) m = join_count(a);
  return m;
}
// The same, once it is known (0: not this CTA).
__device__ __forceinline__ uint32_t join_wait(const SplitLaunch &a, uint32_t mine, uint32_t m) {
  if (mine & kJoinClosed) return 0;
  if (m) return m;
  uint32_t *const came = a.sync + 1;
  const uint32_t all = gridDim.x;
  const long long t0 = clock64();
  for (uint32_t spins = 0; spins < kGridSpin; ++spins) {
    m = join_count(a);
    if (m) return m;
    const uint64_t waited = uint64_t(clock64() - t0);
    if (waited < kJoinLeast) continue;
    uint32_t k;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(k) : "l"(came) : "memory");
    if (k & kJoinClosed) continue;  // the count follows
    if (waited >= min(kJoinMost, uint64_t(a.levels) * (a.n / 2) * (all - k) / (uint64_t(all) * k))) {
      const uint32_t was = atomicOr(came, kJoinClosed);
      if (!(was & kJoinClosed)) {
        join_close(a, was);
        return was;
      }
    }
  }
  atomicOr(a.err, kErrTimeout);
  return 0;
}

// Grid barrier in two halves: between them a CTA does what no other CTA waits
// for.  Bounded; the wait is true when it gave up or the call has failed: the
// caller leaves the kernel, as every other CTA does at its next barrier.
__device__ __forceinline__ void grid_arrive(const SplitLaunch &a) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(a.sync, 1u);
  }
}
__device__ __forceinline__ bool grid_wait(const SplitLaunch &a, const Misc &M, uint32_t &epoch) {
  bool bad = false;
  ++epoch;
  if (threadIdx.x == 0) {
    const uint32_t want = epoch * M.members;
    uint32_t spins = 0;
    for (;;) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.sync) : "memory");
      if (v >= want) break;
      ++spins;
      if (spins > kGridSpin) {
        atomicOr(a.err, kErrTimeout);
        bad = true;
        break;
      }
      if ((spins & 255u) == 0 && *reinterpret_cast<volatile uint32_t *>(a.err)) {
        bad = true;
        break;
      }
    }
    __threadfence();
  }
  return __syncthreads_or(bad) != 0;
}
__device__ __forceinline__ bool grid_sync(const SplitLaunch &a, const Misc &M, uint32_t &epoch) {
  grid_arrive(a);
  return grid_wait(a, M, epoch);
}

__device__ __forceinline__ uint32_t half_of(const uint4 &w, int e) {
  const uint32_t x = e < 2 ? w.x : (e < 4 ? w.y : (e < 6 ? w.z : w.w));
  return (e & 1) ? x >> 16 : x & 0xffffu;
}
__device__ __forceinline__ uint32_t word_of(const uint4 &w, int i) { return i == 0 ? w.x : (i == 1 ? w.y : (i == 2 ? w.z : w.w)); }
__device__ __forceinline__ uint32_t byte_of(const uint2 &w, int e) { return ((e < 4 ? w.x : w.y) >> (8 * (e & 3))) & 0xffu; }

struct Ctx {
  const SplitLaunch &a;
  Misc &M;
  NodeTab &N;
  uint32_t *const bins, *const sum;
  int lane, warp;
  Smem &P;
};

// The segment of subroot s (thread 0 fills the geometry) and its kept state when
// the CTA has several (`load`), else at level 0 the subroot's bounds.
__device__ __forceinline__ void enter_seg(const Ctx &x, uint32_t s, int l, bool load) {
  const SplitLaunch &a = x.a;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t off, cnt;
    node_range(a.n, a.depth, s, off, cnt);
    x.M.soff = uint32_t(off);
    x.M.scnt = uint32_t(cnt);
    const uint32_t r0 = x.M.c * x.M.chunk;
    const uint64_t r1 = min(uint64_t(r0) + x.M.chunk, a.n);
    x.M.b0 = max(uint32_t(off), r0);
    x.M.b1 = uint32_t(min(off + cnt, r1));
    x.M.clo = uint32_t(off) / x.M.chunk;
  }
  if (load) {
    const uint32_t *src = a.state + uint64_t(x.M.c + s) * kStateWords;
    uint32_t *dst = reinterpret_cast<uint32_t *>(&x.N);
    for (uint32_t i = threadIdx.x; i < kStateWords; i += kT) dst[i] = src[i];
  }
  if (l == 0 && !load && threadIdx.x < 3) {  // the subroot's bounds from its parent's split
    const uint32_t d = threadIdx.x;
    uint32_t lo = 0, hi = a.root_hi[d];
    if (a.depth > 0) {
      const LevelNode &p = a.parents[s >> 1];
      lo = p.blo[d];
      hi = p.bhi[d];
      if (p.v != 0xffffffffu && p.axis == d) {
        if (s & 1) lo = p.v;
        else hi = p.v;
      }
    }
    x.N.blo[0][d][0] = lo;
    x.N.bhi[0][d][0] = hi;
  }
  __syncthreads();
}

__device__ __forceinline__ void keep_seg(const Ctx &x, uint32_t s) {
  __syncthreads();
  uint32_t *dst = x.a.state + uint64_t(x.M.c + s) * kStateWords;
  const uint32_t *src = reinterpret_cast<const uint32_t *>(&x.N);
  for (uint32_t i = threadIdx.x; i < kStateWords; i += kT) dst[i] = src[i];
}

constexpr int kPerLane = int(kHalf) / 32;  // nodes of a lane

__device__ __forceinline__ uint32_t warp_excl(uint32_t v, int lane) {
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  return incl - v;
}

// Level l of the segment, by different warps: the smallest shift whose bins fit
// and every node's offset (warp 0); the tie list of the level above, a run of
// `mine` places per node with an odd plane (warp 1); the nodes' places in the
// subroot.  l == levels: the tie list alone.
__device__ __forceinline__ void level_setup(const Ctx &x, int l) {
  if (x.warp == 0 && l < x.a.levels) {
    const int ax = (x.a.depth + l) % 3, p = l & 1;
    const uint32_t nodes = 1u << l;
    uint32_t lo[kPerLane], hi[kPerLane], c[kPerLane];
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
      const uint32_t j = kPerLane * x.lane + i;
      lo[i] = j < nodes ? x.N.blo[p][ax][j] : 1;
      hi[i] = j < nodes ? x.N.bhi[p][ax][j] : 0;
    }
    uint32_t sh = 0, sum, tot;
    for (;; ++sh) {
      sum = 0;
#pragma unroll
      for (int i = 0; i < kPerLane; ++i) {
        c[i] = kPerLane * x.lane + i < nodes ? (hi[i] >> sh) - (lo[i] >> sh) + 1u : 0u;
        sum += c[i];
      }
      tot = __reduce_add_sync(0xffffffffu, sum);
      if (tot <= x.a.bins || sh >= 16) break;
    }
    uint32_t ex = warp_excl(sum, x.lane);
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
      const uint32_t j = kPerLane * x.lane + i;
      if (j < nodes) x.N.off[j] = int32_t(ex) - int32_t(lo[i] >> sh);
      ex += c[i];
    }
    if (x.lane == 0) {
      x.M.shift = sh;
      x.M.nbins = min(tot, x.a.bins);
    }
  } else if (x.warp == 1) {
    const uint32_t half = (1u << l) >> 1;
    uint32_t t[kPerLane], sum = 0, most = 0;
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
      const uint32_t j = kPerLane * x.lane + i;
      t[i] = j < half && (x.N.plane[j] & 1u) ? x.N.mine[j] : 0u;
      sum += t[i];
      most = max(most, t[i]);
    }
    uint32_t ex = warp_excl(sum, x.lane);
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
      x.N.lbase[kPerLane * x.lane + i] = x.N.cursor[kPerLane * x.lane + i] = ex;
      ex += t[i];
    }
    const bool many = __any_sync(0xffffffffu, most > kTieWarp);
    if (x.lane == 31) {
      x.M.ties = ex;
      x.M.many = many;
      // A list takes this CTA some 3 cycles a tie, counting 0.1 a position and up to 1 a tie:
      // levels of 883,024 positions a CTA with up to 16,155 ties took 50 us more counted,
      // levels of 441,512 with as many ties 600 us more listed
      x.M.counted = ex > max(2048u, (x.M.b1 - x.M.b0) / 8u);
    }
  } else if (l < x.a.levels && threadIdx.x >= 64 && threadIdx.x - 64 < (1u << l)) {
    uint64_t off, cnt;
    node_range(x.M.scnt, l, threadIdx.x - 64, off, cnt);
    x.N.roff[threadIdx.x - 64] = uint32_t(off);
    x.N.rcnt[threadIdx.x - 64] = uint32_t(cnt);
  }
  __syncthreads();
}

// The value of rank `rank` among list[0 .. m), positions in [b0, 2^bits + b0): by
// one warp, 5 bits at a time.
// Not inlined: inside the kernel it lengthened the passes' loops (2^27 particles 6030 us a call
// inlined, 5965 so; 2^20 167 and 166).
__device__ __noinline__ uint32_t select_warp(const uint32_t *list, uint32_t m, uint32_t rank, uint32_t b0, int bits,
                                                uint32_t *h, int lane) {
  if (m <= 32) {  // few: every lane counts the positions below its own
    const uint32_t v = uint32_t(lane) < m ? list[lane] : 0xffffffffu;
    uint32_t below = 0;
    for (uint32_t i = 0; i < m; ++i) below += __shfl_sync(0xffffffffu, v, int(i)) < v;
    const uint32_t hit = __ballot_sync(0xffffffffu, uint32_t(lane) < m && below == rank);
    return __shfl_sync(0xffffffffu, v, hit ? __ffs(hit) - 1 : 0);
  }
  uint32_t prefix = 0;
  for (int sh = (bits + 4) / 5 * 5 - 5; sh >= 0; sh -= 5) {
    h[lane] = 0;
    __syncwarp();
    for (uint32_t i = lane; i < m; i += 32) {
      const uint32_t v = list[i] - b0;
      if ((v >> sh >> 5) == prefix) atomicAdd(&h[(v >> sh) & 31u], 1u);
    }
    __syncwarp();
    const uint32_t c = h[lane];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t hit = __ballot_sync(0xffffffffu, incl > rank);
    const int d = hit ? __ffs(hit) - 1 : 31;
    rank -= __shfl_sync(0xffffffffu, incl - c, d);
    prefix = (prefix << 5) | uint32_t(d);
  }
  return b0 + prefix;
}

// The same by the whole block, 11 bits at a time; every thread calls it.
__device__ __noinline__ uint32_t select_block(Misc &M, const uint32_t *list, uint32_t m, uint32_t rank, uint32_t b0,
                                              int bits) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t prefix = 0;
  for (int sh = (bits + 10) / 11 * 11 - 11; sh >= 0; sh -= 11) {
    for (uint32_t i = threadIdx.x; i < kTieBins; i += kT) M.th[i] = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < m; i += kT) {
      const uint32_t v = list[i] - b0;
      if ((v >> sh >> 11) == prefix) atomicAdd(&M.th[(v >> sh) & (kTieBins - 1)], 1u);
    }
    __syncthreads();
    const uint32_t c0 = M.th[2 * threadIdx.x], c1 = M.th[2 * threadIdx.x + 1];
    uint32_t incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) M.wt[warp] = incl;
    __syncthreads();
    const uint32_t t = M.wt[lane];
    const uint32_t ex = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u) + incl - c0 - c1;
    if (c0 && ex <= rank && rank < ex + c0) {
      M.fd = 2 * threadIdx.x;
      M.fbefore = ex;
    }
    if (c1 && ex + c0 <= rank && rank < ex + c0 + c1) {
      M.fd = 2 * threadIdx.x + 1;
      M.fbefore = ex + c0;
    }
    __syncthreads();
    rank -= M.fbefore;
    prefix = (prefix << 11) | M.fd;
    __syncthreads();
  }
  return b0 + prefix;
}

// Counters of the children in F: one row per part of the chunk and warp.
__device__ __forceinline__ uint32_t part_of(const Misc &M, uint32_t pos) {
  const uint32_t q = (pos - M.c * M.chunk) / M.part;
  return min(q, uint32_t(kSplitParts - 1));
}

// The CTA of the move that holds a position.
__device__ __forceinline__ uint32_t move_part(const Misc &M, uint32_t pos) {
  const uint32_t c = pos / M.chunk;
  return c * kSplitParts + min((pos - c * M.chunk) / M.part, uint32_t(kSplitParts - 1));
}

// 8 consecutive particles: their codes on the axis of the level above and on
// this one's, and their nodes.
struct Step {
  uint4 p, c;
  uint2 n;
};
// What a pass reads.  FIRST: level 0, nothing to classify.  LAST: F, which counts
// children per part of the chunk and warp instead of codes.
struct Pass {
  const uint16_t *prev, *cur;
  uint32_t half;  // nodes of the level above
};
template <bool FIRST, bool LAST>
__device__ __forceinline__ void load_step(const Ctx &x, const Pass &a, Step &t, uint32_t pos) {
  if (!FIRST) {
    t.p = __ldcg(reinterpret_cast<const uint4 *>(a.prev + pos));
    if (a.half > 1) t.n = __ldcg(reinterpret_cast<const uint2 *>(x.a.node + pos));
    else t.n = make_uint2(0, 0);  // the subroot itself
  }
  if (!LAST) t.c = __ldcg(reinterpret_cast<const uint4 *>(a.cur + pos));
}
// The pass's first step, loaded ahead of the level's setup.
template <bool FIRST, bool LAST>
__device__ __forceinline__ void first_step(const Ctx &x, const Pass &a, Step &t) {
  const uint32_t pos = (x.M.b0 & ~7u) + 8u * threadIdx.x;
  if (pos < x.M.b1) load_step<FIRST, LAST>(x, a, t, pos);
}

// A pass over the segment, whose first step is loaded.  The ties of nodes with
// an odd plane go right and are listed; there is no variant without the list,
// since a barrier waits for the CTAs that list anyway and code that runs for the
// first time costs microseconds of instruction fetches (at 2^20 particles 104 us
// a launch with both variants, 94 with one).
template <bool FIRST, bool LAST>
__device__ __forceinline__ void pass_a(const Ctx &x, const Pass &a, Step &next, uint32_t *list) {
  NodeTab &N = x.N;
  const uint32_t b0 = x.M.b0, b1 = x.M.b1, shift = x.M.shift;
  uint8_t *const nid = x.a.node;
  const uint32_t room = x.M.ties, listed = x.M.counted ? 0u : 0xffu;
  uint32_t pos = (b0 & ~7u) + 8u * threadIdx.x;
  for (; pos < b1; pos += kStep) {
    const uint4 p = next.p, c = next.c;
    const uint2 n0 = next.n;
    if (pos + kStep < b1) load_step<FIRST, LAST>(x, a, next, pos + kStep);
    uint32_t mask = 0xffu;
    if (pos < b0) mask &= 0xffu << (b0 - pos);
    if (pos + 8u > b1) mask &= 0xffu >> (pos + 8u - b1);
    uint32_t *const bins = LAST ? x.bins + (part_of(x.M, pos) * kW + x.warp) * kNodes : x.bins;
    const int32_t off0 = FIRST ? N.off[0] : 0;
    uint32_t w0 = 0, w1 = 0, hit = 0;
    auto one = [&](int e) {
      uint32_t child = 0;
      if (!FIRST) {
        const uint32_t j = byte_of(n0, e) & (kHalf - 1);
        const uint32_t pl = N.plane[j], t = 2 * half_of(p, e) + 1;
        child = 2 * j + (t >= pl ? 1u : 0u);
        if (t == pl) hit |= 1u << e;
        if (e < 4) w0 |= child << (8 * e);
        else w1 |= child << (8 * (e - 4));
      }
      if (LAST) atomicAdd(&bins[child], 1u);
      else atomicAdd(&bins[uint32_t(int32_t(half_of(c, e) >> shift) + (FIRST ? off0 : N.off[child])) & (kBins - 1)], 1u);
    };
    if (mask == 0xffu) {
#pragma unroll
      for (int e = 0; e < 8; ++e) one(e);
      if (!FIRST) *reinterpret_cast<uint2 *>(nid + pos) = make_uint2(w0, w1);
    } else {
#pragma unroll 1
      for (int e = 0; e < 8; ++e)
        if ((mask >> e) & 1u) {
          one(e);
          if (!FIRST) nid[pos + e] = uint8_t((e < 4 ? w0 : w1) >> (8 * (e & 3)));
        }
    }
    for (hit &= listed; hit; hit &= hit - 1) {
      const int e = __ffs(hit) - 1;
      const uint32_t at = atomicAdd(&N.cursor[byte_of(n0, e) & (kHalf - 1)], 1u);
      if (at < room) {
        list[at] = pos + uint32_t(e);
        if (!LAST && room <= kBins / 2) list[at + kBins / 2] = half_of(c, e);
      }
    }
  }
}

// The listed ties, all counted as going right so far: the first `quota` of each
// node in position order go left after all.
template <bool LAST>
__device__ __forceinline__ void resolve_ties(const Ctx &x, const Pass &a, const uint32_t *list) {
  NodeTab &N = x.N;
  const uint32_t b0 = x.M.b0, shift = x.M.shift;
  const int bits = int(bit_length(x.M.b1 - b0));
  auto fix = [&](uint32_t j, uint32_t i0, uint32_t step, uint32_t limit) {
    const uint32_t *l = list + N.lbase[j];
    for (uint32_t i = i0; i < N.mine[j]; i += step) {
      const uint32_t p = l[i];
      if (p >= limit) continue;
      x.a.node[p] = uint8_t(2 * j);
      uint32_t *left, *right;
      if (LAST) {
        left = x.bins + (part_of(x.M, p) * kW + x.warp) * kNodes + 2 * j;
        right = left + 1;
      } else {  // the code lies beside a list of up to half the room
        const uint32_t c = x.M.ties <= kBins / 2 ? l[i + kBins / 2] : uint32_t(__ldcg(a.cur + p));
        left = x.bins + (uint32_t(int32_t(c >> shift) + N.off[2 * j]) & (kBins - 1));
        right = x.bins + (uint32_t(int32_t(c >> shift) + N.off[2 * j + 1]) & (kBins - 1));
      }
      atomicAdd(left, 1u);
      atomicSub(right, 1u);
    }
  };
  // a node whose list is not full (never expected) is left alone, and the call fails
  auto full = [&](uint32_t j) {
    if (N.cursor[j] - N.lbase[j] == N.mine[j]) return true;
    atomicOr(x.a.err, kErrInternal);
    return false;
  };
  for (uint32_t j = x.warp; j < a.half; j += kW) {
    if (!(N.plane[j] & 1u) || N.mine[j] > kTieWarp || !full(j)) continue;
    const uint32_t limit = select_warp(list + N.lbase[j], N.mine[j], N.quota[j], b0, bits, x.M.wh[x.warp], x.lane);
    fix(j, x.lane, 32, limit);
    __syncwarp();
  }
  if (!x.M.many) return;
  for (uint32_t j = 0; j < a.half; ++j) {
    if (!(N.plane[j] & 1u) || N.mine[j] <= kTieWarp || !full(j)) continue;
    const uint32_t limit = select_block(x.M, list + N.lbase[j], N.mine[j], N.quota[j], b0, bits);
    fix(j, threadIdx.x, kT, limit);
  }
}

// The ties of a segment with many, without a list; all are counted as going right so far.  A
// warp owns a contiguous part of the segment.  First the ties are counted by warp and node;
// then, per node, the warps before the one that holds the quota's end turn all of theirs
// left, and that one its first, in position order: two passes of 5 to 7 bytes a particle,
// whatever the ties are, bound by their instructions.  A list is appended to by one atomic a
// tie and read three times, by the one CTA that holds it while all others wait: 2^24
// particles of which half are one point took 1.75 ms in k_split with one, 0.58 so (0.36
// without ties); every other one the same point 1.52 and 0.81, all on a line 1.18 and 0.62.
template <bool LAST>
__device__ __noinline__ void count_ties(const SplitLaunch &a, Smem &P, const uint16_t *prev, const uint16_t *cur,
                                        uint32_t half) {
  Misc &M = P.M;
  NodeTab &N = P.N;
  const uint32_t b0 = M.b0, b1 = M.b1, shift = M.shift;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t g0 = b0 / 8u, rows = ((b1 + 7u) / 8u - g0 + 31u) / 32u;  // rows of 32 groups of 8 positions
  const uint32_t r0 = rows * uint32_t(warp) / kW, r1 = rows * (uint32_t(warp) + 1u) / kW;
  uint8_t *const nid = a.node;
  uint32_t *const tc = P.sum, *const mine = tc + uint32_t(warp) * kHalf;
  struct Row {
    uint4 p;
    uint2 n;
  };
  auto pos_of = [&](uint32_t r) { return 8u * (g0 + 32u * r + uint32_t(lane)); };
  auto load = [&](uint32_t r, Row &t) {
    const uint32_t pos = pos_of(r);
    t.p = make_uint4(0, 0, 0, 0);
    t.n = make_uint2(0, 0);
    if (r < r1 && pos < b1) {
      t.p = __ldcg(reinterpret_cast<const uint4 *>(prev + pos));
      t.n = __ldcg(reinterpret_cast<const uint2 *>(nid + pos));
    }
  };
  // the row's ties of this lane, by position in its group; the node of position e is its child / 2.
  // Every loop over the 8 positions is unrolled: they are what the two passes are made of.
  auto node_of = [&](const Row &t, int e) { return (byte_of(t.n, e) >> 1) & (kHalf - 1); };
  auto ties = [&](const Row &t, uint32_t pos) {
    uint32_t hit = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (2u * half_of(t.p, e) + 1u == N.plane[node_of(t, e)]) hit |= 1u << e;
    if (pos < b0) hit &= pos + 8u > b0 ? 0xffu << (b0 - pos) : 0u;
    if (pos + 8u > b1) hit &= pos < b1 ? 0xffu >> (pos + 8u - b1) : 0u;
    return hit & 0xffu;
  };
  // whether the row is 256 ties of one node (a run of one point): counted at once, since every lane's
  // atomics on one counter take their turns
  auto run_of_one = [&](const Row &t, uint32_t hit) {
    const uint32_t b = t.n.x & 0xffu;
    int all;
    __match_all_sync(0xffffffffu, hit == 0xffu && t.n.x == t.n.y && t.n.x == b * 0x01010101u ? b : 256u + uint32_t(lane), &all);
    return all != 0;
  };

  for (uint32_t j = lane; j < half; j += 32) mine[j] = 0;
  __syncwarp();
  Row nx;
  load(r0, nx);
  for (uint32_t r = r0; r < r1; ++r) {
    const Row t = nx;
    load(r + 1, nx);
    const uint32_t hit = ties(t, pos_of(r));
    if (run_of_one(t, hit)) {
      if (lane == 0) atomicAdd(&mine[node_of(t, 0)], 256u);
      continue;
    }
    if (!hit) continue;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((hit >> e) & 1u) atomicAdd(&mine[node_of(t, e)], 1u);
  }
  __syncthreads();
  for (uint32_t j = warp; j < half; j += kW) {
    if (!(N.plane[j] & 1u)) continue;
    const uint32_t v = tc[uint32_t(lane) * kHalf + j], incl = warp_excl(v, lane) + v;
    const uint32_t after = __ballot_sync(0xffffffffu, incl > N.quota[j]);
    const int cut = after ? __ffs(after) - 1 : 31;
    if (lane == cut) {
      N.lbase[j] = uint32_t(cut);
      N.cursor[j] = N.quota[j] - (incl - v);
    }
    if (lane == 31 && incl != N.mine[j]) atomicOr(a.err, kErrInternal);  // never expected
  }
  __syncthreads();
  for (uint32_t j = lane; j < half; j += 32) mine[j] = 0;  // now: the ties of a cut node met so far
  __syncwarp();
  load(r0, nx);
  for (uint32_t r = r0; r < r1; ++r) {
    const Row t = nx;
    load(r + 1, nx);
    const uint32_t pos = pos_of(r), hit = ties(t, pos);
    const bool one = run_of_one(t, hit);
    uint32_t left = 0, pend = 0;
    if (one) {
      const uint32_t cut = N.lbase[node_of(t, 0)];
      left = uint32_t(warp) < cut ? hit : 0u;
      pend = uint32_t(warp) == cut ? hit : 0u;
    } else if (hit) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t cut = N.lbase[node_of(t, e)];
        if (uint32_t(warp) < cut) left |= 1u << e;
        if (uint32_t(warp) == cut) pend |= 1u << e;
      }
      left &= hit;
      pend &= hit;
    }
    for (;;) {  // the cut nodes of the row, one by one: the first ones in position order
      const uint32_t any = __ballot_sync(0xffffffffu, pend != 0);
      if (!any) break;
      const uint32_t j = __shfl_sync(0xffffffffu, pend ? node_of(t, __ffs(pend) - 1) : 0u, __ffs(any) - 1);
      uint32_t m = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (node_of(t, e) == j) m |= 1u << e;
      m &= pend;
      const uint32_t cnt = __popc(m), ex = warp_excl(cnt, lane), seen = mine[j], quota = N.cursor[j];
      uint32_t take = seen + ex < quota ? min(cnt, quota - seen - ex) : 0u;
      pend &= ~m;
      if (take == cnt) left |= m;
      else
        for (; take; --take, m &= m - 1) left |= m & (0u - m);
      __syncwarp();
      if (lane == 31) mine[j] = seen + ex + cnt;
      __syncwarp();
    }
    const bool turn = one && __all_sync(0xffffffffu, left == 0xffu);  // all 256
    if (!left) continue;
    uint4 c = make_uint4(0, 0, 0, 0);
    if (!LAST) c = __ldcg(reinterpret_cast<const uint4 *>(cur + pos));
    int same = 0;
    if (turn) {  // of one code on the next axis too, or of one part of the chunk?
      if (!LAST)
        __match_all_sync(0xffffffffu, c.x == c.y && c.x == c.z && c.x == c.w && c.x >> 16 == (c.x & 0xffffu)
                                          ? c.x & 0xffffu
                                          : 65536u + uint32_t(lane),
                         &same);
      else __match_all_sync(0xffffffffu, part_of(M, pos), &same);
    }
    uint32_t *const row = P.bins + (part_of(M, pos) * kW + warp) * kNodes;
    uint32_t w0 = t.n.x, w1 = t.n.y;
    const uint32_t by = same ? 256u : 1u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (!((left >> e) & 1u)) continue;
      const uint32_t j = node_of(t, e);
      if (e < 4) w0 ^= 1u << (8 * e);
      else w1 ^= 1u << (8 * (e - 4));
      if (same && (e > 0 || lane > 0)) continue;
      if (LAST) {  // (a group of 8 lies in one part: parts start at multiples of 16)
        atomicAdd(row + 2 * j, by);
        atomicSub(row + 2 * j + 1, by);
      } else {
        const int32_t q = int32_t(half_of(c, e) >> shift);
        atomicAdd(P.bins + (uint32_t(q + N.off[2 * j]) & (kBins - 1)), by);
        atomicSub(P.bins + (uint32_t(q + N.off[2 * j + 1]) & (kBins - 1)), by);
      }
    }
    if (pos >= b0 && pos + 8u <= b1) {
      *reinterpret_cast<uint2 *>(nid + pos) = make_uint2(w0, w1);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if ((left >> e) & 1u) nid[pos + e] = uint8_t((e < 4 ? w0 : w1) >> (8 * (e & 3)));
    }
  }
}

template <bool FIRST, bool LAST>
__device__ __forceinline__ void run_a(const Ctx &x, const Pass &a, Step &t) {
  // the list: in shared memory when it fits, else in this segment's part of the global one
  uint32_t *const list = x.M.ties <= kBins ? x.sum : x.a.ties + x.M.b0;
  pass_a<FIRST, LAST>(x, a, t, list);
  __syncthreads();
  if (!FIRST && x.M.ties) {
    if (x.M.counted) count_ties<LAST>(x.a, x.P, a.prev, a.cur, a.half);
    else resolve_ties<LAST>(x, a, list);
    __syncthreads();
  }
}

// B: the particles in their node's median bin, counted per code.
template <bool FIRST>
__device__ __forceinline__ void pass_b(const Ctx &x, const uint16_t *__restrict__ cur) {
  const NodeTab &N = x.N;
  const uint32_t b0 = x.M.b0, b1 = x.M.b1, shift = x.M.shift, cm = (1u << shift) - 1u;
  const uint8_t *const nid = x.a.node;
  uint32_t *const low = x.sum;
  const uint32_t bk0 = N.bk[0];
  uint32_t pos = (b0 & ~7u) + 8u * threadIdx.x;
  uint4 nc = make_uint4(0, 0, 0, 0);
  uint2 nn = make_uint2(0, 0);
  auto load = [&](uint32_t p) {
    nc = __ldcg(reinterpret_cast<const uint4 *>(cur + p));
    if (!FIRST) nn = __ldcg(reinterpret_cast<const uint2 *>(nid + p));
  };
  if (pos < b1) load(pos);
  for (; pos < b1; pos += kStep) {
    const uint4 c = nc;
    const uint2 n0 = nn;
    if (pos + kStep < b1) load(pos + kStep);
    uint32_t mask = 0xffu;
    if (pos < b0) mask &= 0xffu << (b0 - pos);
    if (pos + 8u > b1) mask &= 0xffu >> (pos + 8u - b1);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t q = half_of(c, e), j = FIRST ? 0u : byte_of(n0, e) & (kHalf - 1);
      if ((q >> shift) == (FIRST ? bk0 : N.bk[j]) && ((mask >> e) & 1u))
        atomicAdd(&low[((j << shift) | (q & cm)) & (kLow - 1)], 1u);
    }
  }
}

__global__ void __launch_bounds__(kT, 1) k_split(const __grid_constant__ SplitLaunch a) {
  extern __shared__ __align__(128) unsigned char sm[];
  Smem &P = *reinterpret_cast<Smem *>(sm);
  Misc &M = P.M;
  NodeTab &N = P.N;
  uint32_t mine = 0, members = 0;
  if (threadIdx.x == 0) members = join(a, mine);  // its words were zeroed ahead of the kernel before
  dep_wait();
  if (call_failed(a.err)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Ctx x = {a, M, N, P.bins, P.sum, lane, warp, P};
  const uint32_t S = 1u << a.depth;
  const int K = a.levels;
  uint32_t epoch = 0;
  if (threadIdx.x == 0) {
    M.c = mine;
    M.members = join_wait(a, mine, members);
    M.chunk = chunk_of(a.n, max(M.members, 1u));
    M.part = part_size(M.chunk);
    const uint64_t r0 = uint64_t(M.c) * M.chunk;
    M.s0 = 1;
    M.s1 = 0;
    M.nbins = 0;
    if (M.members && r0 < a.n) {  // the subroots holding the first and the last position
      const uint64_t r1 = min(r0 + M.chunk, a.n) - 1;
      for (int e = 0; e < 2; ++e) {
        uint32_t lo = 0, hi = S - 1;
        while (lo < hi) {
          const uint32_t mid = (lo + hi + 1) >> 1;
          uint64_t off, cnt;
          node_range(a.n, a.depth, mid, off, cnt);
          if (off <= (e ? r1 : r0)) lo = mid;
          else hi = mid - 1;
        }
        if (e) M.s1 = lo;
        else M.s0 = lo;
      }
    }
  }
  __syncthreads();
  if (M.members == 0) return;
  const uint32_t c = M.c, s0 = M.s0, s1 = M.s1;
  const bool multi = s1 > s0;
  const uint32_t gthreads = M.members * kT, gtid = c * kT + threadIdx.x;

  for (int l = 0; l < K; ++l) {
    const uint32_t nodes = 1u << l, half = nodes >> 1;
    const uint16_t *const cur = a.src[(a.depth + l) % 3];
    const uint16_t *const prev = a.src[(a.depth + l + 2) % 3];
    uint32_t *const hist = a.hist + uint64_t(l & 1) * S * a.bins;
    uint32_t *const low = a.low + uint64_t(l & 1) * S * a.low_cap;
    // ---- A ----
    Step step;
    const Pass pa = {prev, cur, half};
    if (!multi && l > 0 && s0 <= s1) first_step<false, false>(x, pa, step);
    for (uint32_t s = s0; s <= s1; ++s) {
      if (multi || l == 0) enter_seg(x, s, l, multi && l > 0);
      if (multi && l > 0) first_step<false, false>(x, pa, step);
      if (l == 0) first_step<true, false>(x, pa, step);
      level_setup(x, l);
      const uint32_t nbins = M.nbins;
      if (multi || l == 0) {  // else zeroed after their last use
        for (uint32_t b = threadIdx.x; b < (multi ? nbins : kBins); b += kT) P.bins[b] = 0;
        __syncthreads();
      }
      if (l == 0) run_a<true, false>(x, pa, step);
      else run_a<false, false>(x, pa, step);
      uint32_t *const h = hist + uint64_t(s) * a.bins;
      uint32_t *const own = a.seghist + uint64_t(2 * s + (c != M.clo)) * kBins;
      for (uint32_t b = threadIdx.x; b < nbins; b += kT) {
        const uint32_t v = P.bins[b];
        if (v) atomicAdd(h + b, v);
        if (multi) own[b] = v;
      }
      if (multi) keep_seg(x, s);
    }
    grid_arrive(a);
    if (l > 0) {  // the other histogram was read by every CTA before the last barrier
      uint4 *z = reinterpret_cast<uint4 *>(a.hist + uint64_t((l + 1) & 1) * S * a.bins);
      for (uint32_t i = gtid; i < S * (a.bins / 4); i += gthreads) z[i] = make_uint4(0, 0, 0, 0);
    }
    if (grid_wait(a, M, epoch)) return;
    // ---- sel1 and B ----
    for (uint32_t s = s0; s <= s1; ++s) {
      if (multi) {
        enter_seg(x, s, l, l > 0);
        level_setup(x, l);
      }
      const uint32_t nbins = M.nbins, shift = M.shift;
      {  // exclusive prefixes within each warp's 512 bins, and the warps' totals
        const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + uint64_t(s) * a.bins);
        constexpr uint32_t kPer = kBins / kW;
        uint4 v[kPer / 128];
#pragma unroll
        for (uint32_t i = 0; i < kPer / 128; ++i) {
          const uint32_t b = warp * kPer + i * 128 + lane * 4;
          v[i] = b < nbins ? __ldcg(h4 + b / 4) : make_uint4(0, 0, 0, 0);
        }
        uint32_t run = 0;
#pragma unroll
        for (uint32_t i = 0; i < kPer / 128; ++i) {
          const uint32_t b = warp * kPer + i * 128 + lane * 4;
          const uint32_t t = v[i].x + v[i].y + v[i].z + v[i].w;
          uint32_t incl = t;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          const uint32_t ex = run + incl - t;
          *reinterpret_cast<uint4 *>(&P.sum[b]) =
              make_uint4(ex, ex + v[i].x, ex + v[i].x + v[i].y, ex + v[i].x + v[i].y + v[i].z);
          run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) M.wt[warp] = run;
        __syncthreads();
        uint32_t wb = 0;
        if (warp == 0) {
          const uint32_t t = M.wt[lane];
          uint32_t incl = t;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          wb = incl - t;
        }
        __syncthreads();
        if (warp == 0) M.wt[lane] = wb;
        __syncthreads();
        // per node, by a warp: the last of its bins whose prefix does not exceed the median's rank
        const int ax = (a.depth + l) % 3;
        for (uint32_t j = warp; j < nodes; j += kW) {
          const uint32_t target = N.roff[j] + (N.rcnt[j] >> 1);
          uint32_t lo = uint32_t(N.off[j] + int32_t(N.blo[l & 1][ax][j] >> shift));
          uint32_t hi = min(uint32_t(N.off[j] + int32_t(N.bhi[l & 1][ax][j] >> shift)), kBins - 1u);
          while (lo < hi) {
            const uint32_t by = (hi - lo) / 32u + 1u, at = lo + by * lane;
            const bool le = at <= hi && M.wt[min(at, kBins - 1u) / kPer] + P.sum[min(at, kBins - 1u)] <= target;
            const uint32_t m = __ballot_sync(0xffffffffu, le);
            lo += by * (m ? 31u - uint32_t(__clz(m)) : 0u);
            hi = min(hi, lo + by - 1u);
          }
          if (lane == 0) {
            N.bk[j] = uint32_t(int32_t(lo) - N.off[j]);
            N.below[j] = M.wt[lo / kPer] + P.sum[lo] - N.roff[j];
          }
        }
        __syncthreads();
      }
      const uint32_t nlow = min(nodes << shift, a.low_cap);
      uint32_t *const sl = a.seglow + c + s;  // counter i of this segment: sl[i * segs]
      const uint64_t segs = gridDim.x + S;
      if (shift == 0) {  // A's counters hold the ties of every node
        if (threadIdx.x < nodes) {
          const uint32_t b = uint32_t(N.off[threadIdx.x] + int32_t(N.bk[threadIdx.x])) & (kBins - 1);
          sl[threadIdx.x * segs] = multi ? __ldcg(a.seghist + uint64_t(2 * s + (c != M.clo)) * kBins + b) : P.bins[b];
        }
      } else {
        for (uint32_t i = threadIdx.x; i < nlow; i += kT) P.sum[i] = 0;
        __syncthreads();
        if (l == 0) pass_b<true>(x, cur);
        else pass_b<false>(x, cur);
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < nlow; i += kT) {
          const uint32_t v = P.sum[i];
          sl[i * segs] = v;
          if (v) atomicAdd(low + uint64_t(s) * a.low_cap + i, v);
        }
      }
      if (multi) keep_seg(x, s);
    }
    grid_arrive(a);
    if (l > 0) {  // read by every CTA before the barrier before
      uint4 *z = reinterpret_cast<uint4 *>(a.low + uint64_t((l + 1) & 1) * S * a.low_cap);
      for (uint32_t i = gtid; i < S * (a.low_cap / 4); i += gthreads) z[i] = make_uint4(0, 0, 0, 0);
    }
    if (!multi)
      for (uint32_t b = threadIdx.x; b < M.nbins; b += kT) P.bins[b] = 0;
    if (grid_wait(a, M, epoch)) return;
    // ---- sel2: a warp per node ----
    for (uint32_t s = s0; s <= s1; ++s) {
      if (multi) {
        enter_seg(x, s, l, true);
        level_setup(x, l);
      }
      const uint32_t shift = M.shift;
      const int ax = (a.depth + l) % 3;
      const bool writer = l == K - 1 && c == M.clo;
      for (uint32_t j = warp; j < nodes; j += kW) {
        const uint32_t target = (N.rcnt[j] >> 1) - N.below[j];
        uint32_t vlow = 0, less = 0;
        if (shift) {
          const uint32_t *lw = low + uint64_t(s) * a.low_cap + (j << shift);
          uint32_t run = 0;
          for (uint32_t i0 = 0; i0 < (1u << shift); i0 += 32) {
            const uint32_t v = i0 + lane < (1u << shift) ? __ldcg(lw + i0 + lane) : 0u;
            uint32_t incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += y;
            }
            const uint32_t hit = __ballot_sync(0xffffffffu, v && run + incl - v <= target && target < run + incl);
            if (hit) {
              const int src = __ffs(hit) - 1;
              vlow = i0 + src;
              less = run + __shfl_sync(0xffffffffu, incl - v, src);
              break;
            }
            run += __shfl_sync(0xffffffffu, incl, 31);
          }
        }
        const uint32_t v = (N.bk[j] << shift) | vlow;
        const uint32_t tleft = target - less, slot = min((j << shift) | vlow, a.low_cap - 1u);
        uint32_t before = 0;
        const uint32_t *const row = a.seglow + uint64_t(slot) * (gridDim.x + S) + s;
        const uint32_t mine = __ldcg(row + c);
#pragma unroll 4
        for (uint32_t k = M.clo + lane; k < c; k += 32) before += __ldcg(row + k);
        before = __reduce_add_sync(0xffffffffu, before);
        const uint32_t quota = tleft > before ? min(tleft - before, mine) : 0u;
        if (lane == 0) {
          N.plane[j] = 2 * v + (quota == 0 ? 0u : (quota == mine ? 2u : 1u));
          N.quota[j] = quota;
          N.mine[j] = mine;
          const int p = l & 1, q = p ^ 1;
          if (l + 1 < K) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const uint32_t lo = N.blo[p][d][j], hi = N.bhi[p][d][j];
              N.blo[q][d][2 * j] = lo;
              N.bhi[q][d][2 * j] = d == ax ? v : hi;
              N.blo[q][d][2 * j + 1] = d == ax ? v : lo;
              N.bhi[q][d][2 * j + 1] = hi;
            }
          }
          if (writer) {  // the record the next levels take as parent
            LevelNode nd = {};
            for (int d = 0; d < 3; ++d) {
              nd.blo[d] = N.blo[p][d][j];
              nd.bhi[d] = N.bhi[p][d][j];
            }
            nd.axis = uint32_t(ax);
            nd.lo = nd.blo[ax];
            nd.hi = nd.bhi[ax];
            nd.v = v;
            nd.less = N.below[j] + less;
            nd.tleft = tleft;
            a.out_nodes[(uint64_t(s) << l) + j] = nd;
          }
        }
      }
      if (multi) keep_seg(x, s);
      else __syncthreads();
    }
  }

  // ---- F: final children, counted per segment and part of the chunk ----
  const uint32_t half = 1u << (K - 1);
  for (uint32_t s = s0; s <= s1; ++s) {
    Step step;
    const Pass pf = {a.src[(a.depth + K + 2) % 3], nullptr, half};
    if (multi) enter_seg(x, s, K, true);
    first_step<false, true>(x, pf, step);
    level_setup(x, K);
    for (uint32_t b = threadIdx.x; b < kSplitParts * kW * kNodes; b += kT) P.bins[b] = 0;
    __syncthreads();
    run_a<false, true>(x, pf, step);
    for (uint32_t i = threadIdx.x; i < kSplitParts * kNodes; i += kT) {
      const uint32_t q = i / kNodes, b = i % kNodes;
      if (q < part_of(M, M.b0) || q > part_of(M, M.b1 - 1) || b >= 2 * half) continue;
      uint32_t v = 0;
#pragma unroll 8
      for (int w = 0; w < kW; ++w) v += P.bins[(q * kW + w) * kNodes + b];
      a.segcnt[uint64_t(b) * (gridDim.x * kSplitParts + S) + c * kSplitParts + q + s] = v;
    }
  }
  if (grid_sync(a, M, epoch)) return;
  dep_launch();
  // first place of every child for every part: exclusive sums along the parts of a
  // subroot, in place, a warp per subroot and child
  const uint64_t msegs = uint64_t(gridDim.x) * kSplitParts + S;
  for (uint32_t i = c + M.members * warp; i < S << K; i += M.members * kW) {
    const uint32_t s = i >> K, b = i & ((1u << K) - 1u);
    uint64_t soff, scnt, off, cnt;
    node_range(a.n, a.depth, s, soff, scnt);
    node_range(scnt, K, b, off, cnt);
    uint32_t run = uint32_t(soff + off);
    uint32_t *const row = a.segcnt + b * msegs + s;
    const uint32_t m0 = move_part(M, uint32_t(soff)), m1 = move_part(M, uint32_t(soff + scnt - 1));
    for (uint32_t k0 = m0; k0 <= m1; k0 += 4 * 32) {
      uint32_t v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t k = k0 + 32 * u + lane;
        v[u] = k <= m1 ? __ldcg(row + k) : 0u;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t k = k0 + 32 * u + lane;
        uint32_t incl = v[u];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        if (k <= m1) row[k] = run + incl - v[u];
        run += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
  }
  uint4 *const z = reinterpret_cast<uint4 *>(a.hist);
  for (uint64_t i = gtid; i < a.zero_next; i += gthreads) z[i] = make_uint4(0, 0, 0, 0);
}

// ---- the move ----

constexpr int kMT = 512;
constexpr int kMW = kMT / 32;

template <bool IDX, int BITS, int ROWS>
struct MoveSmem {
  static constexpr uint32_t kCh = 1u << BITS;                   // children, at most
  static constexpr int kRows = ROWS;                            // rows of 32 particles per warp and tile
  static constexpr int kRankBits = kRows == 16 ? 9 : 8;         // a warp's particles of a tile
  static constexpr uint32_t kTile = uint32_t(kRows) * kMT;
  static constexpr uint32_t kStage = kTile + kCh * 14u;         // every child's run padded to whole groups of 8
  alignas(16) uint2 st[kStage];  // x | y << 16, z; place p at stage_slot(p)
  // per warp: first the nodes of its particles, then child << kRankBits | rank of every particle
  alignas(16) uint16_t code[kMW][32 * kRows];
  alignas(16) uint32_t sti[IDX ? kStage : 4];
  // counts of a child by warp, then the place in the stage of the warp's first one; 16 bits, so
  // that the counts of 64 children span the 32 banks once
  uint16_t wcnt[kMW][kCh + 2];
  uint32_t tot[kCh], lst[kCh], lend[kCh], gof[kCh], run[kCh];
  uint8_t grp[kStage / 8 + 8];
  uint32_t s0, s1, b0, b1, ngroups;
};

// Where place p of the stage lies: the four 16-byte pieces of a group of 8 are
// permuted by the group, so that the threads reading a group each meet no bank conflict.
__device__ __forceinline__ uint32_t stage_slot(uint32_t p) { return p ^ ((p >> 3) & 6u); }

// One tile, up to its particles in the stage by child.  WHOLE: the tile lies in
// the segment.  A warp ranks rows of 32 consecutive particles: the lanes with
// the same child, and the warp's count of that child so far from shared memory.
template <bool IDX, int BITS, int ROWS, bool WHOLE>
__device__ __forceinline__ void move_tile(const SplitLaunch &a, MoveSmem<IDX, BITS, ROWS> &T, uint4 nodes, uint32_t t0, uint32_t b0,
                                          uint32_t b1, uint32_t NB, int lane, int warp) {
  using V = MoveSmem<IDX, BITS, ROWS>;
  constexpr int kRows = V::kRows;
  const uint32_t ltm = (1u << lane) - 1u;
  const uint32_t w0 = t0 + uint32_t(warp) * (32 * kRows);  // the warp's first particle
  uint16_t *const wc = T.wcnt[warp], *const cb = T.code[warp];
  auto inside = [&](uint32_t p) { return WHOLE || (p >= b0 && p < b1); };
  for (uint32_t i = lane; i < (NB + 1u) / 2u; i += 32) reinterpret_cast<uint32_t *>(wc)[i] = 0;
  if (lane < 2 * kRows) reinterpret_cast<uint4 *>(cb)[lane] = nodes;
  __syncwarp();
  {
    uint32_t nd[kRows];
    const uint8_t *const nb = reinterpret_cast<const uint8_t *>(cb);
#pragma unroll
    for (int r = 0; r < kRows; ++r) nd[r] = uint32_t(nb[32 * r + lane]) & (NB - 1u);
    // the lanes with this lane's child: one ballot per bit (with a match instruction, which
    // takes as long as the row has different children, the move took 1.07 ms at 2^27)
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      uint32_t peers = WHOLE ? 0xffffffffu : __ballot_sync(0xffffffffu, inside(w0 + 32 * r + lane));
#pragma unroll
      for (int k = 0; k < BITS; ++k) {
        uint32_t v;  // the lanes whose bit k is this lane's
        asm(
            "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t"
            "vote.sync.ballot.b32 %0, p, 0xffffffff;\n\t@!p not.b32 %0, %0;\n\t}"
            : "=r"(v)
            : "r"(nd[r]), "r"(1u << k));
        peers &= v;
      }
      nd[r] |= (__popc(peers & ltm) << 8) | (__popc(peers) << 16);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const uint32_t b = nd[r] & 0xffu, old = wc[b];
      __syncwarp();
      if (inside(w0 + 32 * r + lane)) wc[b] = uint16_t(old + (nd[r] >> 16));  // every lane of the child: the same
      cb[32 * r + lane] = uint16_t((b << V::kRankBits) | (old + ((nd[r] >> 8) & 0xffu)));
      __syncwarp();
    }
  }
  // from here on a lane holds 8 consecutive particles of every 256: its codes
  constexpr int kOct = kRows / 8;
  uint4 x[kOct], y[kOct], z[kOct], ix[IDX ? 2 * kOct : 1];
#pragma unroll
  for (int i = 0; i < kOct; ++i) {
    const uint32_t p = w0 + 256u * i + 8u * lane;
    x[i] = y[i] = z[i] = make_uint4(0, 0, 0, 0);
    if (WHOLE || p < b1) {
      x[i] = __ldcg(reinterpret_cast<const uint4 *>(a.src[0] + p));
      y[i] = __ldcg(reinterpret_cast<const uint4 *>(a.src[1] + p));
      z[i] = __ldcg(reinterpret_cast<const uint4 *>(a.src[2] + p));
      if (IDX) {
        ix[2 * i] = __ldcg(reinterpret_cast<const uint4 *>(a.src_idx + p));
        ix[2 * i + 1] = __ldcg(reinterpret_cast<const uint4 *>(a.src_idx + p) + 1);
      }
    }
  }
  __syncthreads();
  // per child the warps' counts summed up, a half-warp per child
  for (uint32_t b = 2 * warp + (lane >> 4); b < NB; b += 2 * kMW) {
    const uint32_t v = T.wcnt[lane & 15][b];
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const uint32_t w = __shfl_up_sync(0xffffffffu, incl, o, 16);
      if ((lane & 15) >= o) incl += w;
    }
    T.wcnt[lane & 15][b] = uint16_t(incl - v);
    if ((lane & 15) == 15) T.tot[b] = incl;
  }
  __syncthreads();
  // the children's runs in the stage: whole groups of 8, aligned as their destinations
  if (warp == 0) {
    constexpr int kPer = int(V::kCh + 31) / 32;
    uint32_t sz[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const uint32_t b = lane * kPer + i;
      const uint32_t tot = b < NB ? T.tot[b] : 0u;
      sz[i] = tot ? ((T.run[b] & 7u) + tot + 7u) & ~7u : 0u;
      sum += sz[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t w = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += w;
    }
    uint32_t at = incl - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const uint32_t b = lane * kPer + i;
      if (b < NB) {
        const uint32_t g = T.run[b], l0 = at + (g & 7u), tot = T.tot[b];
        T.lst[b] = l0;
        T.lend[b] = l0 + tot;
        T.gof[b] = g - l0;
        T.run[b] = g + tot;
      }
      at += sz[i];
    }
    if (lane == 31) T.ngroups = incl / 8u;
  }
  __syncthreads();
  for (uint32_t b = lane; b < NB; b += 32) wc[b] = uint16_t(wc[b] + T.lst[b]);
  __syncwarp();
  for (uint32_t b = warp; b < NB; b += kMW) {
    const uint32_t l0 = T.lst[b], l1 = T.lend[b];
    if (l1 > l0)
      for (uint32_t g = l0 / 8u + lane; g < (l1 + 7u) / 8u; g += 32) T.grp[g] = uint8_t(b);
  }
#pragma unroll
  for (int i = 0; i < kOct; ++i) {
    const uint4 cd = reinterpret_cast<const uint4 *>(cb)[32 * i + lane];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (inside(w0 + 256u * i + 8u * lane + e)) {
        const uint32_t c = half_of(cd, e);
        const uint32_t at = wc[c >> V::kRankBits] + (c & ((1u << V::kRankBits) - 1u));
        const uint32_t xw = word_of(x[i], e >> 1), yw = word_of(y[i], e >> 1), zw = word_of(z[i], e >> 1);
        T.st[stage_slot(at)] = make_uint2(__byte_perm(xw, yw, (e & 1) ? 0x7632 : 0x5410), (e & 1) ? zw >> 16 : zw);
        if (IDX) T.sti[at] = word_of(ix[2 * i + (e >> 2)], e & 3);
      }
    }
  }
  __syncthreads();
}

// CTA m takes part m % kSplitParts of the chunk m / kSplitParts, tile by tile in
// position order.  A tile's particles are gathered in shared memory by child,
// every child's run starting at the same offset modulo 8 as its destination,
// so that whole groups of 8 leave as 16-byte stores.  BITS: at least `levels`,
// the bits of a child.
template <bool IDX, int BITS, int ROWS>
__global__ void __launch_bounds__(kMT, 2) k_move(const __grid_constant__ SplitLaunch a) {
  extern __shared__ __align__(128) unsigned char sm[];
  using V = MoveSmem<IDX, BITS, ROWS>;
  V &T = *reinterpret_cast<V *>(sm);
  constexpr uint32_t kTile = V::kTile;
  dep_launch();
  dep_wait();
  if (call_failed(a.err)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t m = blockIdx.x, S = 1u << a.depth;
  const int K = a.levels;
  const uint32_t NB = 1u << K;
  const uint32_t members = __ldcg(a.sync + 2);  // the CTAs that found the planes
  if (m >= members * kSplitParts) return;
  const uint32_t chunk = chunk_of(a.n, members), part = part_size(chunk);
  const uint64_t c0 = uint64_t(m / kSplitParts) * chunk, c1 = min(c0 + chunk, a.n);
  const uint64_t q0 = c0 + uint64_t(m % kSplitParts) * part;
  const uint64_t q1 = m % kSplitParts == kSplitParts - 1 ? c1 : min(q0 + part, c1);
  if (q0 >= q1) return;
  if (threadIdx.x < 2) {  // the subroots holding the first and the last position
    const uint64_t p = threadIdx.x ? q1 - 1 : q0;
    uint32_t lo = 0, hi = S - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      uint64_t off, cnt;
      node_range(a.n, a.depth, mid, off, cnt);
      if (off <= p) lo = mid;
      else hi = mid - 1;
    }
    if (threadIdx.x) T.s1 = lo;
    else T.s0 = lo;
  }
  __syncthreads();
  const uint32_t s0 = T.s0, s1 = T.s1;
  for (uint32_t s = s0; s <= s1; ++s) {
    __syncthreads();
    if (threadIdx.x == 0) {
      uint64_t off, cnt;
      node_range(a.n, a.depth, s, off, cnt);
      T.b0 = uint32_t(max(off, q0));
      T.b1 = uint32_t(min(off + cnt, q1));
    }
    if (threadIdx.x < NB) T.run[threadIdx.x] = __ldcg(a.segcnt + uint64_t(threadIdx.x) * (gridDim.x + S) + m + s);
    __syncthreads();
    const uint32_t b0 = T.b0, b1 = T.b1;
    // 16 consecutive particles' nodes of the tile at t0, loaded a tile ahead
    uint4 nodes = make_uint4(0, 0, 0, 0);
    auto load_nodes = [&](uint32_t t0) {
      const uint32_t p = t0 + uint32_t(warp) * (32 * V::kRows) + 16u * lane;
      if (lane < 2 * V::kRows && p < b1) nodes = __ldcg(reinterpret_cast<const uint4 *>(a.node + p));
    };
    load_nodes(b0 & ~31u);
    for (uint32_t t0 = b0 & ~31u; t0 < b1; t0 += kTile) {
      if (t0 >= b0 && t0 + kTile <= b1) move_tile<IDX, BITS, ROWS, true>(a, T, nodes, t0, b0, b1, NB, lane, warp);
      else move_tile<IDX, BITS, ROWS, false>(a, T, nodes, t0, b0, b1, NB, lane, warp);
      if (t0 + kTile < b1) load_nodes(t0 + kTile);
      const uint32_t ngroups = T.ngroups;
      for (uint32_t g = threadIdx.x; g < ngroups; g += kMT) {
        const uint32_t b = T.grp[g], li = 8u * g, gi = li + T.gof[b];
        if (li >= T.lst[b] && li + 8u <= T.lend[b] && uint64_t(gi) + 8u <= a.n) {
          uint32_t u[8], w[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 v = *reinterpret_cast<const uint4 *>(&T.st[stage_slot(li + 2 * i)]);
            u[2 * i] = v.x;
            w[2 * i] = v.y;
            u[2 * i + 1] = v.z;
            w[2 * i + 1] = v.w;
          }
          uint32_t ox[4], oy[4], oz[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ox[i] = __byte_perm(u[2 * i], u[2 * i + 1], 0x5410);
            oy[i] = __byte_perm(u[2 * i], u[2 * i + 1], 0x7632);
            oz[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
          }
          __stcg(reinterpret_cast<uint4 *>(a.dst[0] + gi), make_uint4(ox[0], ox[1], ox[2], ox[3]));
          __stcg(reinterpret_cast<uint4 *>(a.dst[1] + gi), make_uint4(oy[0], oy[1], oy[2], oy[3]));
          __stcg(reinterpret_cast<uint4 *>(a.dst[2] + gi), make_uint4(oz[0], oz[1], oz[2], oz[3]));
          if (IDX) {
            const uint4 *q = reinterpret_cast<const uint4 *>(&T.sti[li]);
            __stcg(reinterpret_cast<uint4 *>(a.dst_idx + gi), q[0]);
            __stcg(reinterpret_cast<uint4 *>(a.dst_idx + gi) + 1, q[1]);
          }
        }
      }
      // the groups at the two ends of every run, a lane per particle
      for (uint32_t i = threadIdx.x; i < NB * 16u; i += kMT) {
        const uint32_t b = i >> 4, l0 = T.lst[b], l1 = T.lend[b];
        const uint32_t g0 = l0 & ~7u, g1 = (l1 - 1u) & ~7u;
        const uint32_t g = (i & 8u) ? g1 : g0, li = g | (i & 7u);
        const bool mine = l1 > l0 && li >= l0 && li < l1 && (g < l0 || g + 8u > l1) && !((i & 8u) && g1 == g0);
        if (mine) {
          const uint32_t gi = li + T.gof[b];
          if (gi < a.n) {
            const uint2 v = T.st[stage_slot(li)];
            __stcg(a.dst[0] + gi, uint16_t(v.x));
            __stcg(a.dst[1] + gi, uint16_t(v.x >> 16));
            __stcg(a.dst[2] + gi, uint16_t(v.y));
            if (IDX) __stcg(a.dst_idx + gi, T.sti[li]);
          } else {
            atomicOr(a.err, kErrInternal);
          }
        }
      }
      // the next tile writes these tables and the stage after its first barriers
    }
  }
}

template <bool IDX, int BITS, int ROWS>
cudaError_t move_launch(const SplitLaunch &a, cudaStream_t st) {
  constexpr size_t smem = sizeof(MoveSmem<IDX, BITS, ROWS>);
  int per_sm = 0;
  cudaError_t e = resident_blocks<k_move<IDX, BITS, ROWS>>(kMT, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  TraceScope ts("k_move", st);
  return launch_dependent(a.alone, k_move<IDX, BITS, ROWS>, dim3(unsigned(a.grid) * kSplitParts), dim3(kMT), smem, st, a);
}
// Tiles of 8192 particles (16 rows a warp) carry their fixed work over twice as many
// (its barriers, scans and tables are half of the instructions with 8); of 4096 where a CTA holds no more, since then
// every warp has rows, and with indices or 256 children, whose stages fill the SM.
template <bool IDX, int BITS>
cudaError_t move_rows(const SplitLaunch &a, cudaStream_t st) {
  if constexpr (!IDX && BITS <= 7) {
    if (a.n / (uint64_t(a.grid) * kSplitParts) > 8u * kMT) return move_launch<IDX, BITS, 16>(a, st);
  }
  return move_launch<IDX, BITS, 8>(a, st);
}
template <bool IDX>
cudaError_t move_dispatch(const SplitLaunch &a, cudaStream_t st) {
  if (a.levels <= 4) return move_rows<IDX, 4>(a, st);
  if (a.levels == 5) return move_rows<IDX, 5>(a, st);
  if (a.levels == 6) return move_rows<IDX, 6>(a, st);
  return a.levels == 7 ? move_rows<IDX, 7>(a, st) : move_rows<IDX, 8>(a, st);
}

}  // namespace

cudaError_t launch_split(const SplitLaunch &a, cudaStream_t st) {
  constexpr size_t smem = sizeof(Smem);
  int per_sm = 0;
  cudaError_t e = resident_blocks<k_split>(kT, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1 || a.grid < 1) return cudaErrorInvalidConfiguration;
  {
    TraceScope ts("k_split", st);
    e = launch_dependent(a.alone, k_split, dim3(unsigned(a.grid)), dim3(kT), smem, st, a);
    if (e != cudaSuccess) return e;
  }
  return a.src_idx ? move_dispatch<true>(a, st) : move_dispatch<false>(a, st);
}

}  // namespace pcx
