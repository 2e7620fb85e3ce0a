// The deep levels of the median k-d partition, the leaves' bit boxes and the
// packed sequences in one kernel (Sec. 4.1 and 4.2, Fig. 4 of arXiv 2404.02826).
//
// Once every node of a level fits in shared memory, a CTA takes one node (in
// ticket order), copies its code arrays in with bulk copies and finishes its
// subtree on chip, without returning to HBM:
//   - every remaining level (the median rule of Sec. 4.1: code < v, then the
//     first `tleft` codes equal to v in index order, go left).  With 16-bit
//     codes and the depth-mod-3 axis nothing moves until the last level is
//     split: a thread keeps its particles' subnodes beside their codes, a histogram
//     of the split axis over all subnodes gives every median, and one stable
//     partition then takes the particles to their leaves (Multi).
//     Otherwise (32-bit codes, widest-cell axis, the leaf-size search's pass,
//     which needs the arrangement of every level): per level and subnode a
//     radix select, then a stable two-way partition in place through tensor
//     memory;
//   - the leaves' bit boxes (AABB, the particle closest to its centre, Eq. 2);
//   - the CTA's first payload word, from the payload sizes of the CTAs before
//     it (decoupled look-back over one status word per node, bounded waits);
//   - the leaf records and the packed payload (Fig. 4), straight from shared
//     memory, and the optional permutation.
// The subnodes of a level are served by equal groups of warps: at relative
// depth k there are 2^k subnodes and 32 / 2^k warps each, and a thread takes
// positions row * (1024 / 2^k) + its index in the group, so it always holds at
// most kRows positions whatever k is.
#include <cstdint>

#include "pc_internal.cuh"
#include "pc_mbar.cuh"

namespace pcx {
namespace {

constexpr int kT = 1024;  // threads of a CTA
constexpr int kLgWarps = 5;
constexpr int kWarps = 1 << kLgWarps;
constexpr int kSubMaxLevels = kLgWarps + 1;  // splits inside a CTA: at least one warp per splitting subnode
constexpr uint32_t kSubBins = 2048;  // radix bins of a level, shared by its subnodes
constexpr uint32_t kMultiBins = 3072;  // the same where levels are split without moving
constexpr uint32_t kLookSpin = 1u << 20;  // polls of a predecessor's status before giving up
constexpr uint32_t kTmemCols = 512;       // tensor-memory columns of a CTA (one CTA per SM)

// One subnode of the CTA's subtree at the current level.
struct SubNode {
  uint32_t off, cnt;        // position in the CTA's node, particles
  uint32_t blo[3], bhi[3];  // cell: code bounds on every axis, from the ancestors' splits
  uint32_t axis, split;     // split axis; 1 if the subnode splits (more than r particles)
  uint32_t lo, prefix, below, width;  // radix select: lowest code, chosen digits, count below them, digit bits
  int32_t shift;
  uint32_t v, tleft;        // split code; particles equal to v that go left
};

struct SubLeaf {
  uint32_t off, cnt, centre, m;
  int32_t qref[3];
  uint32_t words;
  unsigned long long word_off;
  uint32_t lo[3], hi[3];
};

struct SubMisc {
  uint32_t shift, narrow;       // bins of a level; whether codes outside the subnodes' ranges are skipped
  unsigned long long bar;
  unsigned long long prefix;    // payload words of the nodes before this one
  unsigned long long wd[kWarps][2];
  uint32_t wp[kWarps][2];
  unsigned long long off, cnt;  // the node: first particle, particles
  uint32_t j, nl, lead, ilead, tmem;
  uint32_t skip;                // an earlier kernel of the call failed: the node is not worked
  uint32_t wt[kWarps];          // warp totals of the scans
  uint32_t gb[kWarps];          // scan value at the first entry of each group
  uint32_t fb[kWarps], fbefore[kWarps];
};

// Warps per leaf in the leaf phase: kWarps >> lgwl slots of 2^lgwl warps;
// more leaves than warps: a warp per leaf, in turns.
struct LeafSlots {
  uint32_t lgwl, WL, slots, lw, lt, lstep;
};
__device__ __forceinline__ LeafSlots leaf_slots(uint32_t nl, int warp, int lane) {
  LeafSlots q;
  uint32_t lgwl = kLgWarps;
  while (lgwl > 0 && (uint32_t(kWarps) >> lgwl) < nl) --lgwl;
  q.lgwl = lgwl;
  q.WL = 1u << lgwl;
  q.slots = uint32_t(kWarps) >> lgwl;
  q.lw = uint32_t(warp) & (q.WL - 1u);  // warp within its leaf group
  q.lt = q.lw * 32 + uint32_t(lane);
  q.lstep = q.WL * 32;
  return q;
}

constexpr uint32_t kTiesLeft = 0xffffffffu, kTiesRight = 0xfffffffeu;

// Tables of the levels split without moving (an entry per subnode).
struct MultiTab {
  union {
    uint32_t tc[kWarps][kWarps];            // by warp: ties of its particles, then where they go: all
                                            // left, all right, or the subnode's ties before them
    uint16_t wcnt[kWarps][2 * kWarps + 2];  // the move: a warp's particles of a child, then its first place
  };
  uint32_t plane[kWarps];  // right if 2 code + 1 >= plane
  int32_t off[kWarps];     // bin of code x: off + (x >> shift)
  uint32_t range[kWarps];  // codes that can hold the median: lowest | how many << 16 (none: a leaf)
  uint32_t tleft[kWarps];  // ties that go left
};

__host__ __device__ constexpr uint32_t al128(uint32_t x) { return (x + 127u) & ~127u; }

// Shared-memory layout of one CTA: the code arrays of a node of up to
// kRows * 1024 particles (each with room for the lead and tail of a 16-byte
// aligned window), the optional index array, the radix bins, the partition's
// masks and scan (reused as the packing's word staging), the subnode and leaf
// records.  All offsets are compile-time constants.
// MULTI: the levels are split without moving, and with input indices the
// particles' places in the node are kept (16 bits) instead of the indices, so
// that a CTA holds half as many more.
template <typename C, bool IDX, bool MULTI>
struct SubL {
  static constexpr int R =
      sizeof(C) == 2 ? (IDX ? (MULTI ? 24 : 16) : 32) : (IDX ? 12 : 16);  // positions per thread
  // tensor-memory columns of one thread: every array's values of its positions, 32 bits per column
  static constexpr int kCodeCols = sizeof(C) == 2 ? R / 2 : R;
  static constexpr int kCols = 3 * kCodeCols + (MULTI ? R / 2 : (IDX ? R : 0));
  static_assert(kCodeCols % 4 == 0 && (kWarps / 4) * kCols <= 512, "tensor-memory columns");
  static constexpr uint32_t kCap = uint32_t(R) * kT;
  static constexpr uint32_t kSlots = kCap + 16;
  static constexpr uint32_t kCodeStride = al128(kSlots * uint32_t(sizeof(C)));
  static constexpr uint32_t kIdx = 3 * kCodeStride;
  static constexpr uint32_t kBins = kIdx + (IDX ? al128(kSlots * (MULTI ? 2 : 4)) : 0u);
  static constexpr uint32_t kStage = kBins + al128((MULTI ? kMultiBins : kSubBins) * 4);
  static constexpr uint32_t kPart = MULTI ? sizeof(MultiTab) : uint32_t(R) * kWarps * 16, kPack = kWarps * 96u * 4;
  static constexpr uint32_t kSn0 = kStage + al128(kPart > kPack ? kPart : kPack);
  static constexpr uint32_t kSn1 = kSn0 + al128(kWarps * sizeof(SubNode));
  static constexpr uint32_t kLeaf = kSn1 + al128(kWarps * sizeof(SubNode));
  static constexpr uint32_t kMisc = kLeaf + al128(2 * kWarps * sizeof(SubLeaf));
  static constexpr uint32_t kTotal = kMisc + al128(sizeof(SubMisc));
  static_assert(kTotal <= 232448, "shared memory of one CTA");
};

constexpr unsigned long long kStAgg = 1ull << 62, kStIncl = 2ull << 62, kStVal = (1ull << 62) - 1;

__device__ __forceinline__ void st_release_u64(unsigned long long *p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint32_t widest_axis(const uint32_t *blo, const uint32_t *bhi) {
  uint32_t ax = 0;
  for (uint32_t d = 1; d < 3; ++d)
    if (bhi[d] - blo[d] > bhi[ax] - blo[ax]) ax = d;
  return ax;
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Radix-select state of a splitting subnode from its cell (k_prep's rule):
// all codes equal on the axis decides at once, else digits of at most hb bits.
__device__ __forceinline__ void sub_select_init(SubNode &s, uint32_t hb) {
  s.lo = s.blo[s.axis];
  const uint32_t B = bit_length(s.bhi[s.axis] - s.lo);
  s.prefix = 0;
  s.below = 0;
  if (!s.split) {
    s.width = 0;
  } else if (B == 0) {
    s.width = 0;
    s.v = s.lo;
    s.tleft = s.cnt >> 1;
  } else {
    s.width = B < hb ? B : hb;
    s.shift = int32_t(B - s.width);
  }
}

// ---- tensor memory (TMEM): where each thread keeps its rows between levels ----
// Between two levels a thread's positions (its rows of its group's subnode)
// live in its own TMEM lane (tcgen05.st / tcgen05.ld, shape 32x32b: a warp
// reaches the 32 lanes of its lane quarter, 32 bits per column).  Shared
// memory only serves the exchange of a level's move: every thread writes its
// values to their destinations, the block synchronises, and every thread reads
// its rows of the next level back into TMEM.  One warp allocates the columns
// at the start and frees them at the end.  Every tcgen05 instruction is
// .sync.aligned, so each helper first reconverges the warp.
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {
  __syncwarp();
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  __syncwarp();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 4 consecutive columns of this thread's lane; completes by tmem_wait_st()
__device__ __forceinline__ void tmem_st4(uint32_t t, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  __syncwarp();
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(t), "r"(a), "r"(b), "r"(c),
               "r"(d)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  __syncwarp();
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// 8 consecutive columns, complete when the call returns
__device__ __forceinline__ void tmem_ld8(uint32_t t, uint32_t *v) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(t)
      : "memory");
}
// 4 columns from each of three places (the x, y, z values of the same rows), one wait
__device__ __forceinline__ void tmem_ld4x3(uint32_t t0, uint32_t t1, uint32_t t2, uint32_t *v) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%12];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [%13];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [%14];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11])
      : "r"(t0), "r"(t1), "r"(t2)
      : "memory");
}
// 4 columns from one place and 2 from another, one wait
__device__ __forceinline__ void tmem_ld4_2(uint32_t t0, uint32_t t1, uint32_t *v, uint32_t *n) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%6];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4, %5}, [%7];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(n[0]), "=r"(n[1])
      : "r"(t0), "r"(t1)
      : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t t, uint32_t *v) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1])
      : "r"(t)
      : "memory");
}
// 2 consecutive columns; complete by tmem_wait_st()
__device__ __forceinline__ void tmem_st2(uint32_t t, uint32_t a, uint32_t b) {
  __syncwarp();
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(t), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t t, uint32_t *v) {
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
      : "r"(t)
      : "memory");
}

// Up to 8 columns (`left` of them remain in the array; a compile-time value
// after unrolling), the rest zero.
__device__ __forceinline__ void tmem_ld_cols(uint32_t t, uint32_t *v, int left) {
  if (left >= 8) {
    tmem_ld8(t, v);
  } else {
    tmem_ld4(t, v);
    v[4] = v[5] = v[6] = v[7] = 0;
  }
}

// Value of row r of a thread's array from its columns: 16-bit values two rows
// per column (rows 2c and 2c + 1 in column c), 32-bit values one row each.
template <typename E>
__device__ __forceinline__ uint32_t row_of(const uint32_t *cols, int r) {
  if constexpr (sizeof(E) == 2) return (cols[r >> 1] >> (16 * (r & 1))) & 0xffffu;
  else return cols[r];
}

// Reads the rows p = r * Tg + ltid (r < nv) of one array of a subnode from
// shared memory into the thread's columns from `taddr` (completion:
// tmem_wait_st).
template <int R, typename E>
__device__ __forceinline__ void load_rows(const E *A, uint32_t nv, uint32_t Tg, uint32_t ltid, uint32_t taddr) {
  constexpr int NC = sizeof(E) == 2 ? R / 2 : R;
  constexpr int RPC = sizeof(E) == 2 ? 2 : 1;  // rows per column
#pragma unroll
  for (int c0 = 0; c0 < NC; c0 += 4) {
    uint32_t v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[c] = 0;
#pragma unroll
      for (int h = 0; h < RPC; ++h) {
        const int r = RPC * (c0 + c) + h;
        if (uint32_t(r) < nv) v[c] |= uint32_t(A[uint32_t(r) * Tg + ltid]) << (16 * h);
      }
    }
    tmem_st4(taddr + uint32_t(c0), v[0], v[1], v[2], v[3]);
  }
}

// All levels of a CTA's node, then one move (16-bit codes, depth-mod-3 axis).
// Warp w owns the positions [w Rn 32, (w + 1) Rn 32) in rows of 32.  A thread's
// rows stay in its tensor-memory columns, 8 rows a chunk: the codes of array d
// from tcol + d NC, from kRk on first a byte per row with 4 x its subnode (the
// byte offset into the tables), at the end child << 10 | rank.  On entry cur[0]
// is the node; on exit X0 (and, with IDX, the places P) are in leaf order and
// cur holds the subnodes of the last level.  bins: zero on entry and on exit.
// Chunks whose rows all hold particles take unguarded code: with a guard per
// row the guards cost more than the work.
// A CTA of 32768 particles and three levels takes 119 K cycles (2^27 particles:
// 1.58 ms a launch, 1.94 with a move per level and a particle per lane in the
// packing, 148 K): copy 5, rows into tensor memory 4, per level histogram 6
// (bound by the shared-memory atomics), search 1.5, split 7, ties 3, then ranks 9,
// move 10, boxes 11, look-back 10 (waiting for the slowest node before), packing 15.
template <bool IDX, typename L>
struct Multi {
  static constexpr int R = L::R, NC = L::kCodeCols;
  static constexpr uint32_t kRk = 3u * NC, kNid = kRk + R / 4;  // rank columns: R / 2; nodes: their second half
  static constexpr uint32_t S = L::kCodeStride / 2;
  const SubtreeLaunch &a;
  uint16_t *const X0, *const P;
  uint32_t *const bins;
  MultiTab &T;
  SubMisc &M;
  const uint32_t tcol;
  const int lane, warp;
  uint32_t cnt, Rn, w0, nv, nvw, chunks;  // nv: this thread's rows, nvw: the least of the warp

  template <typename V>
  static __device__ __forceinline__ V at4(const V *t, uint32_t byte) {
    return *reinterpret_cast<const V *>(reinterpret_cast<const char *>(t) + byte);
  }
  static __device__ __forceinline__ uint32_t byte_at(const uint32_t *n, int i) {
    return __byte_perm(n[i >> 2], 0u, 0x4440u | uint32_t(i & 3));
  }

  // NARROW: only codes that can hold their subnode's median
  template <bool FULL, bool NARROW>
  __device__ __forceinline__ void hist_chunk(uint32_t ch, uint32_t ax, uint32_t shift) {
    uint32_t v[4], n[2];
    tmem_ld4_2(tcol + ax * NC + 4u * ch, tcol + kNid + 2u * ch, v, n);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t c = row_of<uint16_t>(v, i), j4 = byte_at(n, i);
      const uint32_t b = min(uint32_t(int32_t(c >> shift) + at4(T.off, j4)), kMultiBins - 1u);
      bool in = FULL || 8u * ch + i < nv;
      if (NARROW) {
        const uint32_t rg = at4(T.range, j4);
        in = in && c - (rg & 0xffffu) < (rg >> 16);
      }
      if (in) atomicAdd(&bins[b], 1u);
    }
  }
  // to the children, ties right; the ties are counted by warp and subnode, their rows kept
  template <bool FULL>
  __device__ __forceinline__ uint32_t split_chunk(uint32_t ch, uint32_t ax) {
    uint32_t v[4], n[2], o[2] = {0, 0}, hit = 0;
    tmem_ld4_2(tcol + ax * NC + 4u * ch, tcol + kNid + 2u * ch, v, n);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t t = 2u * row_of<uint16_t>(v, i) + 1u, j4 = byte_at(n, i);
      const uint32_t p = at4(T.plane, j4);
      o[i >> 2] |= (2u * j4 + (t >= p ? 4u : 0u)) << (8 * (i & 3));
      if (t == p && (FULL || 8u * ch + i < nv)) hit |= 1u << i;
    }
    tmem_st2(tcol + kNid + 2u * ch, o[0], o[1]);
    if (__any_sync(0xffffffffu, hit != 0)) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((hit >> i) & 1u) atomicAdd(&T.tc[warp][byte_at(n, i) >> 2], 1u);
    }
    return hit;
  }
  // the ties of a chunk whose subnode's ties in this warp all go left
  __device__ __forceinline__ void left_chunk(uint32_t ch, uint32_t hit) {
    uint32_t n[2];
    tmem_ld2(tcol + kNid + 2u * ch, n);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t how = T.tc[warp][(byte_at(n, i) >> 3) & 31u];  // 4 x child = 8 x node + 4
      if (((hit >> i) & 1u) && how == kTiesLeft) n[i >> 2] -= 4u << (8 * (i & 3));
    }
    tmem_st2(tcol + kNid + 2u * ch, n[0], n[1]);
  }
  // the first `quota` ties of subnode j in position order
  __device__ __forceinline__ void cut_node(uint32_t j, uint32_t quota, uint32_t hits) {
    const uint32_t ltm = (1u << lane) - 1u;
    uint32_t seen = 0;
    for (uint32_t ch = 0; ch < chunks && seen < quota; ++ch) {
      const uint32_t hit = (hits >> (8u * ch)) & 0xffu;
      if (!__any_sync(0xffffffffu, hit != 0)) continue;
      uint32_t n[2];
      tmem_ld2(tcol + kNid + 2u * ch, n);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool mine = ((hit >> i) & 1u) && ((byte_at(n, i) >> 3) & 31u) == j;
        const uint32_t m = __ballot_sync(0xffffffffu, mine);
        if (mine && seen + __popc(m & ltm) < quota) n[i >> 2] -= 4u << (8 * (i & 3));
        seen += __popc(m);
      }
      tmem_st2(tcol + kNid + 2u * ch, n[0], n[1]);
    }
  }
  // ranks among the warp's particles of the same child
  template <bool FULL, int BITS>
  __device__ __forceinline__ void rank_chunk(uint32_t ch) {
    const uint32_t ltm = (1u << lane) - 1u;
    uint16_t *const wc = T.wcnt[warp];
    uint32_t n[2], rk[4];
    tmem_ld2(tcol + kNid + 2u * ch, n);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t b = byte_at(n, i) >> 2;
      uint32_t peers = FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, 8u * ch + i < nv);
#pragma unroll
      for (int q = 0; q < BITS; ++q) {
        uint32_t m;  // the lanes whose bit q is this lane's
        asm(
            "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t"
            "vote.sync.ballot.b32 %0, p, 0xffffffff;\n\t@!p not.b32 %0, %0;\n\t}"
            : "=r"(m)
            : "r"(b), "r"(1u << q));
        peers &= m;
      }
      const uint32_t old = wc[b];
      __syncwarp();
      if (FULL || 8u * ch + i < nv) wc[b] = uint16_t(old + __popc(peers));  // the same from every lane of the child
      __syncwarp();
      const uint32_t cd = (b << 10) | (old + __popc(peers & ltm));
      if (i & 1) rk[i >> 1] |= cd << 16;
      else rk[i >> 1] = cd;
    }
    tmem_st4(tcol + kRk + 4u * ch, rk[0], rk[1], rk[2], rk[3]);
  }
  template <bool FULL>
  __device__ __forceinline__ void move_chunk(uint32_t ch) {
    const uint16_t *const wc = T.wcnt[warp];
    uint32_t v[12], rk[4];
    tmem_ld4x3(tcol + 4u * ch, tcol + NC + 4u * ch, tcol + 2 * NC + 4u * ch, v);
    tmem_ld4(tcol + kRk + 4u * ch, rk);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t cd = row_of<uint16_t>(rk, i);
      const uint32_t dst = min(uint32_t(wc[cd >> 10]) + (cd & 1023u), uint32_t(L::kCap) - 1u);
      if (FULL || 8u * ch + i < nv) {
        X0[dst] = uint16_t(row_of<uint16_t>(v, i));
        X0[S + dst] = uint16_t(row_of<uint16_t>(v + 4, i));
        X0[2 * S + dst] = uint16_t(row_of<uint16_t>(v + 8, i));
        if (IDX) P[dst] = uint16_t(w0 + 32u * (8u * ch + i));
      }
    }
  }

  __device__ __forceinline__ void run(SubNode *&cur, SubNode *&nxt) {
    cnt = cur[0].cnt;
    Rn = (cnt + kT - 1u) / kT;
    chunks = (Rn + 7u) / 8u;
    w0 = uint32_t(warp) * Rn * 32u + uint32_t(lane);
    nv = w0 < cnt ? min((cnt - w0 + 31u) / 32u, Rn) : 0u;
    nvw = __reduce_min_sync(0xffffffffu, nv);
#pragma unroll
    for (int d = 0; d < 3; ++d) load_rows<R>(X0 + d * S + uint32_t(warp) * Rn * 32u, nv, 32u, uint32_t(lane), tcol + d * NC);
    for (uint32_t ch = 0; ch < chunks; ++ch) tmem_st2(tcol + kNid + 2u * ch, 0u, 0u);
    tmem_wait_st();

    for (int k = 0; k < a.levels; ++k) {
      const uint32_t G = 1u << k, ax = uint32_t(a.depth + k) % 3u;
      if (threadIdx.x < G) {
        SubNode &u = cur[threadIdx.x];
        u.lo = u.blo[ax];
        u.prefix = u.bhi[ax];  // the codes that can hold the median: lo .. prefix
        u.below = 0;
      }
      __syncthreads();
      // the medians: bins of 2^shift codes over all subnodes' ranges, narrowed until shift is 0
      for (bool first = true;; first = false) {
        if (warp == 0) {
          const bool in = uint32_t(lane) < G && cur[lane].split;
          const uint32_t lo = in ? cur[lane].lo : 1u, hi = in ? cur[lane].prefix : 0u;
          uint32_t sh = 0, nb, tot;
          for (;; ++sh) {
            nb = in ? (hi >> sh) - (lo >> sh) + 1u : 0u;
            tot = __reduce_add_sync(0xffffffffu, nb);
            if (tot <= kMultiBins || sh >= 16) break;
          }
          uint32_t incl = nb;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          T.off[lane] = int32_t(incl - nb) - int32_t(lo >> sh);
          T.range[lane] = in ? (lo & 0xffffu) | (min(hi - lo + 1u, 0xffffu) << 16) : 0u;
          const bool all = __all_sync(0xffffffffu, in || uint32_t(lane) >= G);
          if (lane == 0) {
            M.shift = sh;
            M.narrow = !(first && all);
          }
        }
        __syncthreads();
        const uint32_t shift = M.shift;
        const bool narrow = M.narrow != 0;
        for (uint32_t ch = 0; ch < chunks; ++ch) {
          const bool full = 8u * ch + 8u <= nvw;
          if (!narrow) {
            if (full) hist_chunk<true, false>(ch, ax, shift);
            else hist_chunk<false, false>(ch, ax, shift);
          } else {
            if (full) hist_chunk<true, true>(ch, ax, shift);
            else hist_chunk<false, true>(ch, ax, shift);
          }
        }
        __syncthreads();
        {  // exclusive prefixes in place, three bins per thread
          static_assert(kMultiBins == 3 * kT, "bins per thread");
          const uint32_t b = 3u * threadIdx.x, h0 = bins[b], h1 = bins[b + 1], h2 = bins[b + 2];
          uint32_t incl = h0 + h1 + h2;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          if (lane == 31) M.wt[warp] = incl;
          __syncthreads();
          const uint32_t t = M.wt[lane];
          const uint32_t ex = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u) + incl - h0 - h1 - h2;
          bins[b] = ex;
          bins[b + 1] = ex + h0;
          bins[b + 2] = ex + h0 + h1;
        }
        __syncthreads();
        if (uint32_t(warp) < G && cur[warp].split) {  // a warp per subnode: its last bin whose prefix is not above the rank
          SubNode &u = cur[warp];
          const int32_t off = T.off[warp];
          uint32_t lo = uint32_t(int32_t(u.lo >> shift) + off);
          uint32_t hi = min(uint32_t(int32_t(u.prefix >> shift) + off), kMultiBins - 1u);
          const uint32_t s0 = bins[min(lo, kMultiBins - 1u)], target = (u.cnt >> 1) - u.below + s0;
          while (lo < hi) {
            const uint32_t by = (hi - lo) / 32u + 1u, at = lo + by * lane;
            const uint32_t m = __ballot_sync(0xffffffffu, at <= hi && bins[min(at, kMultiBins - 1u)] <= target);
            lo += by * (m ? 31u - uint32_t(__clz(m)) : 0u);
            hi = min(hi, lo + by - 1u);
          }
          __syncwarp();
          if (lane == 0) {
            const uint32_t q = uint32_t(int32_t(lo) - off);  // the bin's codes: q << shift ..
            u.below += bins[min(lo, kMultiBins - 1u)] - s0;
            u.lo = max(u.lo, q << shift);
            u.prefix = min(u.prefix, ((q + 1u) << shift) - 1u);
          }
        }
        __syncthreads();
        for (uint32_t b = threadIdx.x; b < kMultiBins; b += kT) bins[b] = 0;
        if (shift == 0) break;
      }
      // the planes (an odd one: 2 v + 1, its ties are listed) and the children
      T.tc[warp][lane] = 0;
      if (threadIdx.x < G) {
        SubNode &u = cur[threadIdx.x];
        const uint32_t v = u.lo, kk = u.cnt >> 1;
        u.v = v;
        u.tleft = kk - u.below;
        T.plane[threadIdx.x] = u.split ? 2u * v + 1u : 0x7ffffffeu;
        if (k + 1 < a.levels) {
          if (!u.split) atomicOr(a.err, kErrInternal);
          for (uint32_t h = 0; h < 2; ++h) {
            SubNode &w = nxt[2 * threadIdx.x + h];
            for (int d = 0; d < 3; ++d) {
              w.blo[d] = u.blo[d];
              w.bhi[d] = u.bhi[d];
            }
            if (h) w.blo[ax] = v;
            else w.bhi[ax] = v;
            w.off = u.off + (h ? kk : 0u);
            w.cnt = h ? u.cnt - kk : kk;
            w.axis = uint32_t(a.depth + k + 1) % 3u;
            w.split = w.cnt > a.leaf_size;
          }
        }
      }
      __syncthreads();
      uint32_t hits = 0;  // a bit per row
      for (uint32_t ch = 0; ch < chunks; ++ch) {
        const uint32_t h = 8u * ch + 8u <= nvw ? split_chunk<true>(ch, ax) : split_chunk<false>(ch, ax);
        hits |= h << (8u * ch);
      }
      tmem_wait_st();
      __syncthreads();
      // where each warp's ties start among its subnode's: the first `tleft` of all go left
      if (uint32_t(warp) < G) {
        const uint32_t mine = T.tc[lane][warp];
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        const uint32_t tleft = cur[warp].split ? cur[warp].tleft : 0u;
        T.tc[lane][warp] = incl <= tleft ? kTiesLeft : (incl - mine >= tleft ? kTiesRight : incl - mine);
        if (lane == 0) T.tleft[warp] = tleft;
      }
      __syncthreads();
      {
        const uint32_t how = uint32_t(lane) < G ? T.tc[warp][lane] : kTiesRight;
        if (__any_sync(0xffffffffu, how == kTiesLeft)) {
          for (uint32_t ch = 0; ch < chunks; ++ch) {
            const uint32_t h = (hits >> (8u * ch)) & 0xffu;
            if (__any_sync(0xffffffffu, h != 0)) left_chunk(ch, h);
          }
          tmem_wait_st();
        }
        for (uint32_t cut = __ballot_sync(0xffffffffu, how < kTiesRight); cut; cut &= cut - 1u) {
          const uint32_t j = uint32_t(__ffs(cut)) - 1u;
          cut_node(j, T.tleft[j] - __shfl_sync(0xffffffffu, how, j), hits);
          tmem_wait_st();
        }
        tmem_wait_st();
      }
      if (k + 1 < a.levels) {
        SubNode *t = cur;
        cur = nxt;
        nxt = t;
      }
      __syncthreads();
    }

    // ---- the move ----
    const uint32_t NB = 1u << a.levels;
    uint16_t *const wc = T.wcnt[warp];
    for (uint32_t b = lane; b < 2u * kWarps; b += 32) wc[b] = 0;
    __syncwarp();
    for (uint32_t ch = 0; ch < chunks; ++ch) {
      const bool full = 8u * ch + 8u <= nvw;
      if (a.levels <= 3) {
        if (full) rank_chunk<true, 3>(ch);
        else rank_chunk<false, 3>(ch);
      } else {
        if (full) rank_chunk<true, 6>(ch);
        else rank_chunk<false, 6>(ch);
      }
    }
    tmem_wait_st();
    __syncthreads();
    // first place of every warp's particles of a child: the child's place from the median rule
    for (uint32_t b = warp; b < NB; b += kWarps) {
      const SubNode &u = cur[b >> 1];
      const uint32_t base = u.off + ((b & 1u) ? (u.split ? u.cnt >> 1 : u.cnt) : 0u);
      const uint32_t v = T.wcnt[lane][b];
      uint32_t incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      T.wcnt[lane][b] = uint16_t(base + incl - v);
    }
    __syncthreads();
    for (uint32_t ch = 0; ch < chunks; ++ch) {
      if (8u * ch + 8u <= nvw) move_chunk<true>(ch);
      else move_chunk<false>(ch);
    }
    __syncthreads();
  }
};

// 128 particles of a leaf (block `blk` of its non-centre particles) packed by a
// warp, 8 <= w <= 32: a lane forms 4 consecutive particles' 4 w bits, shifted to
// their place in the words, and takes the word it shares with the next lane's
// first bits.  128 particles fill 4 w whole words.  24 instructions per 32
// particles, against 80 with a particle per lane whose words are put together
// by shuffles.
template <typename C>
__device__ __forceinline__ void pack_block(const C *x0, const C *x1, const C *x2, uint32_t b0, uint32_t b1, uint32_t b2,
                                           uint32_t m0, uint32_t m1, uint32_t w, uint32_t blk, uint32_t centre,
                                           uint32_t nsl, uint32_t words, uint32_t *payload, int lane) {
  uint32_t v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t sl = blk * 128u + 4u * lane + i;
    const uint32_t p = min(sl, nsl - 1u) + (sl >= centre ? 1u : 0u);
    const uint32_t q = min(p, nsl);  // nsl + 1 particles with the centre
    const uint32_t y = uint32_t(x0[q]) - b0 | ((uint32_t(x1[q]) - b1) << (m0 & 31u)) |
                       ((uint32_t(x2[q]) - b2) << ((m0 + m1) & 31u));
    v[i] = sl < nsl ? y : 0u;
  }
  const unsigned long long lo = v[0] | ((unsigned long long)v[1] << w), hi = v[2] | ((unsigned long long)v[3] << w);
  const unsigned long long a0 = w < 32u ? lo | (hi << (2u * w)) : lo, a1 = w < 32u ? hi >> (64u - 2u * w) : hi;
  const uint32_t bit = 4u * w * uint32_t(lane), k0 = bit >> 5, sh = bit & 31u, end = sh + 4u * w;
  const uint32_t t0 = uint32_t(a0), t1 = uint32_t(a0 >> 32), t2 = uint32_t(a1), t3 = uint32_t(a1 >> 32);
  uint32_t W[5] = {t0 << sh, __funnelshift_l(t0, t1, sh), __funnelshift_l(t1, t2, sh), __funnelshift_l(t2, t3, sh),
                   __funnelshift_l(t3, 0u, sh)};
  const uint32_t nx = __shfl_down_sync(0xffffffffu, W[0], 1);
  const uint32_t last = (end - 1u) >> 5, gw0 = blk * 4u * w + k0;
#pragma unroll
  for (uint32_t i = 0; i < 5; ++i) {
    if ((i > 0 || sh == 0) && i <= last && gw0 + i < words) {
      uint32_t word = W[i];
      if (i == last && (end & 31u) != 0) word |= nx;
      __stcs(payload + gw0 + i, word);
    }
  }
}

// COST: the leaf-size search's pass.  Every subnode splits at every level;
// before the first level and after each one the leaves at that depth get their
// bit boxes, and their payload words are added to cost_words[level]; nothing
// is written to the stream.
template <typename C, bool IDX, bool WIDEST, bool COST>
__global__ void __launch_bounds__(kT, 1) k_subtree(const __grid_constant__ SubtreeLaunch a) {
  constexpr bool MULTI = sizeof(C) == 2 && !WIDEST && !COST;
  using L = SubL<C, IDX, MULTI>;
  constexpr int R = L::R;
  extern __shared__ __align__(128) unsigned char sm[];
  uint32_t *bins = reinterpret_cast<uint32_t *>(sm + L::kBins);
  // per (row, warp): scan of the packed counts, mask of code < v, mask of code == v
  uint4 *S4 = reinterpret_cast<uint4 *>(sm + L::kStage);
  SubNode *cur = reinterpret_cast<SubNode *>(sm + L::kSn0);
  SubNode *nxt = reinterpret_cast<SubNode *>(sm + L::kSn1);
  SubLeaf *LF = reinterpret_cast<SubLeaf *>(sm + L::kLeaf);
  SubMisc &M = *reinterpret_cast<SubMisc *>(sm + L::kMisc);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ltm = (1u << lane) - 1u;

  dep_launch();
  dep_wait();
  // ---- the node: ticket order, so every node before it has started ----
  if (threadIdx.x == 0) {
    M.j = atomicAdd(a.ticket, 1u);
    mbar_init(&M.bar, 1);
    mbar_fence_init();
  }
  constexpr uint32_t kV = 16 / sizeof(C);  // codes per 16 bytes
  if (threadIdx.x == 0) {
    const uint32_t j = M.j;
    uint64_t off64, cnt64;
    node_range(a.n, a.depth, j, off64, cnt64);
    M.off = off64;
    M.cnt = cnt64;
    const uint32_t lead = uint32_t(off64) & (kV - 1u), ilead = uint32_t(off64) & 3u;
    M.lead = lead;
    M.ilead = ilead;
    const uint32_t noff = uint32_t(off64), ncnt = uint32_t(cnt64);
    const uint32_t nwin = (lead + ncnt + kV - 1u) & ~(kV - 1u);
    const uint32_t niw = (ilead + ncnt + 3u) & ~3u;
    const bool dead = *reinterpret_cast<const volatile uint32_t *>(a.err) != 0u;
    M.skip = dead ? 1u : 0u;
    const bool ok = ncnt <= L::kCap && !dead;
    const uint32_t bytes = ok ? 3 * nwin * uint32_t(sizeof(C)) + (IDX && !MULTI ? 4 * niw : 0u) : 0u;
    if (!ok && !dead) atomicOr(a.err, kErrInternal);
    mbar_expect_tx(&M.bar, bytes);
    if (bytes) {
      for (int d = 0; d < 3; ++d)
        bulk_g2s(sm + d * L::kCodeStride, static_cast<const C *>(a.codes[d]) + (noff - lead),
                 nwin * uint32_t(sizeof(C)), &M.bar);
      if (IDX && !MULTI) bulk_g2s(sm + L::kIdx, a.idx + (noff - ilead), 4 * niw, &M.bar);
    }
    // the root of the subtree: its cell from the parent's split (k_prep's rule);
    // in a failed call the parents' records were never written and are not read
    SubNode &s = cur[0];
    if (a.depth == 0 || dead) {
      for (int d = 0; d < 3; ++d) {
        s.blo[d] = 0;
        s.bhi[d] = a.root_hi[d];
      }
    } else {
      const LevelNode &p = a.parents[j >> 1];
      for (int d = 0; d < 3; ++d) {
        s.blo[d] = p.blo[d];
        s.bhi[d] = p.bhi[d];
      }
      if (p.v != 0xffffffffu && p.axis < 3u) {
        if (j & 1) s.blo[p.axis] = p.v;
        else s.bhi[p.axis] = p.v;
      }
    }
    s.off = 0;
    s.cnt = ok ? ncnt : 0u;
    s.axis = WIDEST ? widest_axis(s.blo, s.bhi) : uint32_t(a.depth % 3);
    s.split = s.cnt > a.leaf_size;
  }
  // the radix bins start at zero (every select pass leaves them zero again)
  for (uint32_t b = threadIdx.x; b < (MULTI ? kMultiBins : kSubBins); b += kT) bins[b] = 0;
  if (warp == 0) tmem_alloc(&M.tmem, kTmemCols);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  // this thread's tensor-memory columns: lane quarter warp % 4, columns by warpgroup
  const uint32_t tcol = M.tmem + ((32u * (uint32_t(warp) & 3u)) << 16) + (uint32_t(warp) >> 2) * uint32_t(L::kCols);
  // A failed call (an earlier kernel, or this copy's wait giving up): the
  // node's status is published as complete, so that no later node waits for
  // it, and the CTA leaves.
  const bool late = wait_buffer(&M.bar, 0, a.err);
  if (__syncthreads_or(late || M.skip != 0u)) {
    if (!COST && threadIdx.x == 0) st_release_u64(a.status + M.j, kStIncl);
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
      tmem_fence_after();
      tmem_dealloc(M.tmem, kTmemCols);
    }
    return;
  }
  // element i of the node (any array) sits at slot lead + i
  C *const X0 = reinterpret_cast<C *>(sm) + M.lead;

  // ---- the levels inside the CTA ----
  constexpr int NC = L::kCodeCols;                 // TMEM columns of one code array
  constexpr int RPC = sizeof(C) == 2 ? 2 : 1;      // rows per column
  constexpr uint32_t S = L::kCodeStride / sizeof(C);
  uint32_t *const XI = reinterpret_cast<uint32_t *>(sm + L::kIdx) + M.ilead;
  if (!MULTI && a.levels > 0) {  // the root's rows into TMEM (level 0: one group of all warps)
    const uint32_t cnt0 = cur[0].cnt;
    const uint32_t nv0 = cnt0 > threadIdx.x ? (cnt0 - threadIdx.x + kT - 1u) / kT : 0u;
    load_rows<R>(X0, nv0, kT, threadIdx.x, tcol);
    load_rows<R>(X0 + S, nv0, kT, threadIdx.x, tcol + NC);
    load_rows<R>(X0 + 2 * S, nv0, kT, threadIdx.x, tcol + 2 * NC);
    if (IDX) load_rows<R>(XI, nv0, kT, threadIdx.x, tcol + 3 * NC);
    tmem_wait_st();
  }
  const C *const Y0 = X0, *const Y1 = X0 + S, *const Y2 = X0 + 2 * S;
  // Leaves below the subnodes cur[0..G): the two halves of a splitting subnode
  // (with `halves`), else the subnode itself; their AABBs, centres (first
  // position on ties), widths (Eq. 2) and payload words, in LF.  Returns
  // their number.  Every thread calls it.
  auto leaf_boxes = [&](uint32_t G, bool halves) -> uint32_t {
    if (threadIdx.x == 0) {
      uint32_t nl = 0;
      for (uint32_t t = 0; t < G; ++t) {
        const SubNode &u = cur[t];
        if (halves && u.split) {
          const uint32_t kk = u.cnt >> 1;
          LF[nl].off = u.off;
          LF[nl++].cnt = kk;
          LF[nl].off = u.off + kk;
          LF[nl++].cnt = u.cnt - kk;
        } else {
          LF[nl].off = u.off;
          LF[nl++].cnt = u.cnt;
        }
      }
      M.nl = nl;
    }
    __syncthreads();
    const uint32_t nl = M.nl;
    if (threadIdx.x < nl) {
      for (int d = 0; d < 3; ++d) {
        LF[threadIdx.x].lo[d] = 0xffffffffu;
        LF[threadIdx.x].hi[d] = 0;
      }
    }
    const LeafSlots q = leaf_slots(nl, warp, lane);
    const uint32_t lgwl = q.lgwl, WL = q.WL, slots = q.slots, lt = q.lt, lstep = q.lstep;
    __syncthreads();
    // bit boxes: AABB
    for (uint32_t f = uint32_t(warp) >> lgwl; f < nl; f += slots) {
      const uint32_t off = LF[f].off, cnt = LF[f].cnt;
      uint32_t mn0 = 0xffffffffu, mn1 = 0xffffffffu, mn2 = 0xffffffffu, mx0 = 0, mx1 = 0, mx2 = 0;
      if (sizeof(C) == 2) {  // eight codes a load, two a minimum; the ends one by one
        const uint32_t e0 = uint32_t(X0 - reinterpret_cast<C *>(sm)) + off, e1 = e0 + cnt;  // slots of the leaf
        const uint32_t g0 = min((e0 + 7u) & ~7u, e1), g1 = max(g0, e1 & ~7u);
        uint32_t n2[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, x2[3] = {0, 0, 0};
        for (uint32_t g = g0 + 8u * lt; g < g1; g += 8u * lstep) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const uint4 q = *reinterpret_cast<const uint4 *>(sm + d * L::kCodeStride + 2u * g);
            n2[d] = min_u16x2(n2[d], min_u16x2(min_u16x2(q.x, q.y), min_u16x2(q.z, q.w)));
            x2[d] = max_u16x2(x2[d], max_u16x2(max_u16x2(q.x, q.y), max_u16x2(q.z, q.w)));
          }
        }
        const uint32_t e = lt < 8u ? (e0 + lt < g0 ? e0 + lt : e1) : (lt < 16u ? g1 + lt - 8u : e1);
        if (e < e1) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const uint32_t c = *reinterpret_cast<const C *>(sm + d * L::kCodeStride + 2u * e) * 0x10001u;
            n2[d] = min_u16x2(n2[d], c);
            x2[d] = max_u16x2(x2[d], c);
          }
        }
        mn0 = min(n2[0] & 0xffffu, n2[0] >> 16);
        mn1 = min(n2[1] & 0xffffu, n2[1] >> 16);
        mn2 = min(n2[2] & 0xffffu, n2[2] >> 16);
        mx0 = max(x2[0] & 0xffffu, x2[0] >> 16);
        mx1 = max(x2[1] & 0xffffu, x2[1] >> 16);
        mx2 = max(x2[2] & 0xffffu, x2[2] >> 16);
      } else {
        for (uint32_t i = lt; i < cnt; i += lstep) {
          const uint32_t c0 = Y0[off + i], c1 = Y1[off + i], c2 = Y2[off + i];
          mn0 = min(mn0, c0);
          mx0 = max(mx0, c0);
          mn1 = min(mn1, c1);
          mx1 = max(mx1, c1);
          mn2 = min(mn2, c2);
          mx2 = max(mx2, c2);
        }
      }
      mn0 = __reduce_min_sync(0xffffffffu, mn0);
      mn1 = __reduce_min_sync(0xffffffffu, mn1);
      mn2 = __reduce_min_sync(0xffffffffu, mn2);
      mx0 = __reduce_max_sync(0xffffffffu, mx0);
      mx1 = __reduce_max_sync(0xffffffffu, mx1);
      mx2 = __reduce_max_sync(0xffffffffu, mx2);
      if (lane == 0) {
        atomicMin(&LF[f].lo[0], mn0);
        atomicMin(&LF[f].lo[1], mn1);
        atomicMin(&LF[f].lo[2], mn2);
        atomicMax(&LF[f].hi[0], mx0);
        atomicMax(&LF[f].hi[1], mx1);
        atomicMax(&LF[f].hi[2], mx2);
      }
    }
    __syncthreads();
    // centre: least squared distance to the AABB centre, first position on ties.
    // When every side of the box is below 2^15 codes, |2q - lo - hi| < 2^15 and
    // the squared distance is exact in 32 bits; otherwise it is formed in 64.
    {
      int it = 0;
      for (uint32_t f = uint32_t(warp) >> lgwl; f < nl; f += slots, ++it) {
        const uint32_t off = LF[f].off, cnt = LF[f].cnt;
        const uint32_t l0 = LF[f].lo[0], l1 = LF[f].lo[1], l2 = LF[f].lo[2];
        const uint32_t u0 = LF[f].hi[0], u1 = LF[f].hi[1], u2 = LF[f].hi[2];
        unsigned long long bd;
        uint32_t bp;
        if (max(u0 - l0, max(u1 - l1, u2 - l2)) < 32768u) {
          const int s0 = int(l0 + u0), s1 = int(l1 + u1), s2 = int(l2 + u2);
          uint32_t md = 0xffffffffu, mp = 0xffffffffu;
          for (uint32_t i = lt; i < cnt; i += lstep) {
            const int e0 = 2 * int(Y0[off + i]) - s0, e1 = 2 * int(Y1[off + i]) - s1, e2 = 2 * int(Y2[off + i]) - s2;
            const uint32_t d2 = uint32_t(e0 * e0) + uint32_t(e1 * e1) + uint32_t(e2 * e2);
            if (d2 < md) {  // positions rise within a thread: the first minimum is the lowest
              md = d2;
              mp = i;
            }
          }
          const uint32_t wmd = __reduce_min_sync(0xffffffffu, md);
          bp = __reduce_min_sync(0xffffffffu, md == wmd ? mp : 0xffffffffu);
          bd = wmd;
        } else {
          const long long s0 = (long long)l0 + u0, s1 = (long long)l1 + u1, s2 = (long long)l2 + u2;
          bd = ~0ull;
          bp = 0xffffffffu;
          for (uint32_t i = lt; i < cnt; i += lstep) {
            const long long e0 = 2ll * Y0[off + i] - s0, e1 = 2ll * Y1[off + i] - s1, e2 = 2ll * Y2[off + i] - s2;
            const unsigned long long d2 =
                (unsigned long long)(e0 * e0) + (unsigned long long)(e1 * e1) + (unsigned long long)(e2 * e2);
            if (d2 < bd) {
              bd = d2;
              bp = i;
            }
          }
  #pragma unroll
          for (int o = 16; o; o >>= 1) {
            const unsigned long long od = __shfl_xor_sync(0xffffffffu, bd, o);
            const uint32_t op = __shfl_xor_sync(0xffffffffu, bp, o);
            if (od < bd || (od == bd && op < bp)) {
              bd = od;
              bp = op;
            }
          }
        }
        if (lane == 0) {
          M.wd[warp][it] = bd;
          M.wp[warp][it] = bp;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < nl) {
      const uint32_t f = threadIdx.x;
      unsigned long long bd = ~0ull;
      uint32_t bp = 0xffffffffu;
      const bool turns = nl > uint32_t(kWarps);
      const uint32_t w0 = turns ? (f % kWarps) : (f << lgwl), wn = turns ? 1u : WL, it = turns ? (f / kWarps) : 0u;
      for (uint32_t w = w0; w < w0 + wn; ++w) {
        const unsigned long long od = M.wd[w][it];
        const uint32_t op = M.wp[w][it];
        if (od < bd || (od == bd && op < bp)) {
          bd = od;
          bp = op;
        }
      }
      SubLeaf &lf = LF[f];
      const uint32_t c = bp < lf.cnt ? bp : 0u;
      const uint32_t q0 = Y0[lf.off + c], q1 = Y1[lf.off + c], q2 = Y2[lf.off + c];
      const uint32_t m0 = bits_for_range(max(q0 - lf.lo[0], lf.hi[0] - q0));
      const uint32_t m1 = bits_for_range(max(q1 - lf.lo[1], lf.hi[1] - q1));
      const uint32_t m2 = bits_for_range(max(q2 - lf.lo[2], lf.hi[2] - q2));
      lf.qref[0] = int32_t(q0);
      lf.qref[1] = int32_t(q1);
      lf.qref[2] = int32_t(q2);
      lf.centre = c;
      lf.m = m0 | (m1 << 8) | (m2 << 16);
      lf.words = uint32_t((uint64_t(m0 + m1 + m2) * (lf.cnt ? lf.cnt - 1 : 0) + 31) >> 5);
    }
    __syncthreads();
    return nl;
  };
  // the leaf-size search: payload words of the leaves at in-CTA depth k
  auto add_cost = [&](uint32_t nl, int k) {
    if (warp == 0) {
      unsigned long long w = 0;
      for (uint32_t f = lane; f < nl; f += 32) w += LF[f].words;
#pragma unroll
      for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
      if (lane == 0) atomicAdd(a.cost_words + k, w);
    }
  };
  if (COST) add_cost(leaf_boxes(1, false), 0);  // the node itself as one leaf
  uint16_t *const PL = reinterpret_cast<uint16_t *>(sm + L::kIdx);  // MULTI: places of the input indices in the node
  if constexpr (MULTI) {
    if (a.levels > 0)
      Multi<IDX, L>{a, X0, PL, bins, *reinterpret_cast<MultiTab *>(sm + L::kStage), M, tcol, lane, warp}.run(cur, nxt);
    else if (IDX)
      for (uint32_t i = threadIdx.x; i < cur[0].cnt; i += kT) PL[i] = uint16_t(i);
  }
  for (int k = 0; !MULTI && k < a.levels; ++k) {
    const int lgW = kLgWarps - k;  // log2 of the warps per group
    const uint32_t G = 1u << k;
    const int g = warp >> lgW;
    const uint32_t Tg = uint32_t(kT) >> k;
    const uint32_t ltid = threadIdx.x & (Tg - 1u);
    const uint32_t BPG = kSubBins >> k, hb = 11u - uint32_t(k);
    const uint32_t soff = cur[g].off, scnt = cur[g].cnt;
    const uint32_t nv = scnt > ltid ? (scnt - ltid + Tg - 1u) / Tg : 0u;  // rows of this thread in its subnode
    const uint32_t tax = tcol + cur[g].axis * NC;                           // columns of the split axis
    if (threadIdx.x < G) sub_select_init(cur[threadIdx.x], hb);
    // radix select of every splitting subnode, one digit per pass, from the rows in TMEM
    bool any = __syncthreads_or(threadIdx.x < G && cur[threadIdx.x].width != 0);
    while (any) {
      const uint32_t width = cur[g].width;
      const bool act = width != 0;
      if (act) {
        const uint32_t lo = cur[g].lo, prefix = cur[g].prefix, shift = uint32_t(cur[g].shift);
        const uint32_t mask = (1u << width) - 1u;
        uint32_t *hg = bins + uint32_t(g) * BPG;
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 8) {
          uint32_t v[8];
          tmem_ld_cols(tax + uint32_t(c0), v, NC - c0);
#pragma unroll
          for (int i = 0; i < 8 * RPC; ++i) {
            const int r = RPC * c0 + i;
            if (r < R && uint32_t(r) < nv) {
              const uint32_t hbk = (row_of<C>(v, i) - lo) >> shift;
              if ((hbk >> width) == prefix) atomicAdd(&hg[hbk & mask], 1u);
            }
          }
        }
      }
      __syncthreads();
      // the bucket holding rank cnt/2 - below: kBinsPer bins per thread, scanned within the group
      constexpr uint32_t kBinsPer = kSubBins / kT;
      const uint32_t b0 = kBinsPer * threadIdx.x;  // bins of this thread (in its own group's region)
      uint32_t h[kBinsPer], x = 0;
#pragma unroll
      for (uint32_t e = 0; e < kBinsPer; ++e) {
        h[e] = bins[b0 + e];
        bins[b0 + e] = 0;
        x += h[e];
      }
      if (!act) x = 0;
      uint32_t incl = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) M.wt[warp] = incl;
      __syncthreads();
      if (act) {
        uint32_t base = 0;
        for (int w = g << lgW; w < warp; ++w) base += M.wt[w];
        uint32_t ex = base + incl - x;
        const uint32_t target = (scnt >> 1) - cur[g].below;
        if (x && ex <= target && target < ex + x) {
          uint32_t e = 0;
          while (e + 1 < kBinsPer && target >= ex + h[e]) ex += h[e++];
          M.fb[g] = b0 - uint32_t(g) * BPG + e;
          M.fbefore[g] = ex;
        }
      }
      __syncthreads();
      bool still = false;
      if (act && ltid == 0) {
        SubNode &u = cur[g];
        u.below += M.fbefore[g];
        u.prefix = (u.prefix << u.width) | M.fb[g];
        if (u.shift == 0) {
          u.v = u.lo + u.prefix;
          u.tleft = (u.cnt >> 1) - u.below;
          u.width = 0;
        } else {
          const uint32_t w = uint32_t(u.shift) < hb ? uint32_t(u.shift) : hb;
          u.shift -= int32_t(w);
          u.width = w;
          still = true;
        }
      }
      any = __syncthreads_or(still);
    }

    const bool split = cur[g].split != 0;
    // classification: masks of code < v and code == v per (row, warp)
    {
      const uint32_t v = cur[g].v;
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 8) {
        uint32_t cv[8];
        tmem_ld_cols(tax + uint32_t(c0), cv, NC - c0);
#pragma unroll
        for (int i = 0; i < 8 * RPC; ++i) {
          const int r = RPC * c0 + i;
          if (r >= R) break;
          const bool valid = split && uint32_t(r) < nv;
          const uint32_t c = row_of<C>(cv, i);
          const uint32_t lm = __ballot_sync(0xffffffffu, valid && c < v);
          const uint32_t tm = __ballot_sync(0xffffffffu, valid && c == v);
          if (lane == 0) {
            S4[r * kWarps + warp].y = lm;
            S4[r * kWarps + warp].z = tm;
          }
        }
      }
    }
    __syncthreads();
    // one block-wide exclusive scan over the entries (group, row, warp of the group),
    // the order of the positions within each subnode; kEPT consecutive entries per thread
    {
      constexpr uint32_t kE = uint32_t(R) * kWarps, kEPT = (kE + kT - 1) / kT;
      const uint32_t per_group = uint32_t(R) << lgW;
      uint32_t cx[kEPT], slot[kEPT], sum = 0;
#pragma unroll
      for (uint32_t e = 0; e < kEPT; ++e) {
        const uint32_t i = threadIdx.x * kEPT + e;
        cx[e] = 0;
        slot[e] = 0;
        if (i < kE) {
          const uint32_t gi = i / per_group;
          const uint32_t rem = i - gi * per_group;
          const uint32_t row = rem >> lgW, w = rem & ((1u << lgW) - 1u);
          slot[e] = row * kWarps + (gi << lgW) + w;
          cx[e] = (uint32_t(__popc(S4[slot[e]].y)) << 16) | uint32_t(__popc(S4[slot[e]].z));
        }
        sum += cx[e];
      }
      uint32_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) M.wt[warp] = inc;
      __syncthreads();
      if (warp == 0) {
        const uint32_t t = lane < kWarps ? M.wt[lane] : 0u;
        uint32_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, ti, o);
          if (lane >= o) ti += y;
        }
        if (lane < kWarps) M.wt[lane] = ti - t;
      }
      __syncthreads();
      uint32_t ex = M.wt[warp] + inc - sum;
#pragma unroll
      for (uint32_t e = 0; e < kEPT; ++e) {
        const uint32_t i = threadIdx.x * kEPT + e;
        if (i < kE) {
          S4[slot[e]].x = ex;
          if (i % per_group == 0) M.gb[i / per_group] = ex;
        }
        ex += cx[e];
      }
    }
    __syncthreads();
    // the move: every row from TMEM to its destination in shared memory
    {
      const uint32_t kk = scnt >> 1, gbase = M.gb[g], tleft = cur[g].tleft;
      C *const A0 = X0 + soff, *const A1 = X0 + S + soff, *const A2 = X0 + 2 * S + soff;
      uint32_t *const AI = XI + soff;
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 4) {
        uint32_t v[12];
        tmem_ld4x3(tcol + uint32_t(c0), tcol + uint32_t(NC + c0), tcol + uint32_t(2 * NC + c0), v);
        uint32_t vi[4 * RPC];
        if (IDX) {
          tmem_ld4(tcol + uint32_t(3 * NC + RPC * c0), vi);
          if (RPC == 2) tmem_ld4(tcol + uint32_t(3 * NC + RPC * c0 + 4), vi + 4);
        }
#pragma unroll
        for (int i = 0; i < 4 * RPC; ++i) {
          const int r = RPC * c0 + i;
          if (uint32_t(r) < nv) {
            const uint32_t p = uint32_t(r) * Tg + ltid;
            uint32_t dst = p;
            if (split) {
              const uint4 e = S4[r * kWarps + warp];
              const uint32_t P = e.x - gbase;
              const uint32_t lb = (P >> 16) + uint32_t(__popc(e.y & ltm));
              uint32_t gl;
              bool left;
              if (e.z == 0) {  // no code of this warp's row equals v
                gl = lb + min(P & 0xffffu, tleft);
                left = (e.y >> lane) & 1u;
              } else {
                const uint32_t tb = (P & 0xffffu) + uint32_t(__popc(e.z & ltm));
                left = ((e.y >> lane) & 1u) || (((e.z >> lane) & 1u) && tb < tleft);
                gl = lb + min(tb, tleft);
              }
              dst = left ? gl : kk + p - gl;
              if (dst >= scnt) {
                atomicOr(a.err, kErrInternal);
                dst = p;
              }
            }
            A0[dst] = C(row_of<C>(v, i));
            A1[dst] = C(row_of<C>(v + 4, i));
            A2[dst] = C(row_of<C>(v + 8, i));
            if (IDX) AI[dst] = vi[i];
          }
        }
      }
    }
    // children of every subnode (every subnode above the last level splits)
    if (k + 1 < a.levels && threadIdx.x < G) {
      const SubNode &u = cur[threadIdx.x];
      if (!u.split) atomicOr(a.err, kErrInternal);
      const uint32_t kk = u.cnt >> 1;
      SubNode &cl = nxt[2 * threadIdx.x], &cr = nxt[2 * threadIdx.x + 1];
      for (int d = 0; d < 3; ++d) {
        cl.blo[d] = cr.blo[d] = u.blo[d];
        cl.bhi[d] = cr.bhi[d] = u.bhi[d];
      }
      cl.bhi[u.axis] = u.v;
      cr.blo[u.axis] = u.v;
      cl.off = u.off;
      cl.cnt = kk;
      cr.off = u.off + kk;
      cr.cnt = u.cnt - kk;
      const uint32_t ax = uint32_t((a.depth + k + 1) % 3);
      cl.axis = WIDEST ? widest_axis(cl.blo, cl.bhi) : ax;
      cr.axis = WIDEST ? widest_axis(cr.blo, cr.bhi) : ax;
      cl.split = cl.cnt > a.leaf_size;
      cr.split = cr.cnt > a.leaf_size;
    }
    __syncthreads();  // the level's arrangement is complete in shared memory
    if (COST) add_cost(leaf_boxes(G, true), k + 1);
    if (k + 1 < a.levels) {
      SubNode *t = cur;
      cur = nxt;
      nxt = t;
      // this thread's rows of the next level back into TMEM
      const int g2 = warp >> (lgW - 1);
      const uint32_t Tg2 = Tg >> 1, ltid2 = threadIdx.x & (Tg2 - 1u);
      const uint32_t off2 = cur[g2].off, cnt2 = cur[g2].cnt;
      const uint32_t nv2 = cnt2 > ltid2 ? (cnt2 - ltid2 + Tg2 - 1u) / Tg2 : 0u;
      load_rows<R>(X0 + off2, nv2, Tg2, ltid2, tcol);
      load_rows<R>(X0 + S + off2, nv2, Tg2, ltid2, tcol + NC);
      load_rows<R>(X0 + 2 * S + off2, nv2, Tg2, ltid2, tcol + 2 * NC);
      if (IDX) load_rows<R>(XI + off2, nv2, Tg2, ltid2, tcol + 3 * NC);
      tmem_wait_st();
      // the next level's moves overwrite shared memory only after its selection's barriers
    }
  }

  if (COST) {
    // the search pass: the deepest in-CTA arrangement back to HBM when asked
    // (a deeper search continues there); no leaf records, look-back or packing
    if (a.wb_codes[0]) {
      const uint64_t o = M.off;
      const uint32_t cnt = uint32_t(M.cnt);
      for (uint32_t i = threadIdx.x; i < cnt; i += kT) {
        static_cast<C *>(a.wb_codes[0])[o + i] = X0[i];
        static_cast<C *>(a.wb_codes[1])[o + i] = X0[S + i];
        static_cast<C *>(a.wb_codes[2])[o + i] = X0[2 * S + i];
        if (IDX) a.wb_idx[o + i] = XI[i];
      }
      // and the records of the last in-CTA level (depth + levels - 1), the parents of the
      // level over HBM that continues from there: their cells and splits (k_prep's fields)
      if (a.wb_nodes && a.levels > 0) {
        const uint32_t G = 1u << (a.levels - 1);
        if (threadIdx.x < G) {
          const SubNode &u = cur[threadIdx.x];
          LevelNode nd = {};
          for (int d = 0; d < 3; ++d) {
            nd.blo[d] = u.blo[d];
            nd.bhi[d] = u.bhi[d];
          }
          nd.axis = u.axis;
          nd.v = u.split ? u.v : 0xffffffffu;
          a.wb_nodes[(uint64_t(M.j) << (a.levels - 1)) + threadIdx.x] = nd;
        }
      }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
      tmem_fence_after();
      tmem_dealloc(M.tmem, kTmemCols);
    }
    return;
  }
  // ---- leaves: the last level's subnodes, split or not, in order ----
  const uint32_t nl = leaf_boxes(a.levels > 0 ? 1u << (a.levels - 1) : 1u, true);
  const LeafSlots q = leaf_slots(nl, warp, lane);
  const uint32_t lgwl = q.lgwl, WL = q.WL, slots = q.slots, lw = q.lw, lt = q.lt, lstep = q.lstep;
  // ---- payload words before this node: decoupled look-back ----
  const uint32_t j = M.j;
  if (warp == 0) {
    unsigned long long agg = 0;
    for (uint32_t f = lane; f < nl; f += 32) agg += LF[f].words;
#pragma unroll
    for (int o = 16; o; o >>= 1) agg += __shfl_xor_sync(0xffffffffu, agg, o);
    if (lane == 0) st_release_u64(a.status + j, (j == 0 ? kStIncl : kStAgg) | agg);
    unsigned long long prefix = 0;
    if (j > 0) {
      long long i = (long long)j - 1;
      uint32_t spins = 0;
      for (;;) {
        const long long q = i - lane;
        const unsigned long long st = q >= 0 ? ld_acquire_u64(a.status + q) : kStIncl;
        const unsigned long long flag = st >> 62;
        const uint32_t incl = __ballot_sync(0xffffffffu, flag == 2), zero = __ballot_sync(0xffffffffu, flag == 0);
        const int fi = incl ? __ffs(incl) - 1 : 32;
        const uint32_t rel = fi >= 31 ? 0xffffffffu : ((2u << fi) - 1u);
        if (zero & rel) {
          if (++spins > kLookSpin) {
            if (lane == 0) atomicOr(a.err, kErrTimeout);
            break;
          }
          __nanosleep(64);
          continue;
        }
        unsigned long long v = lane <= fi ? (st & kStVal) : 0ull;
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        prefix += v;
        if (fi < 32) break;
        i -= 32;
      }
      if (lane == 0) st_release_u64(a.status + j, kStIncl | (prefix + agg));
    }
    if (lane == 0) {
      if (uint64_t(j) + 1 == (1ull << a.depth)) *a.total_words = prefix + agg;
      unsigned long long run = prefix;
      for (uint32_t f = 0; f < nl; ++f) {
        LF[f].word_off = run;
        run += LF[f].words;
      }
    }
  }
  __syncthreads();

  // ---- leaf records, permutation and packed payload ----
  const uint64_t off64 = M.off;
  const uint64_t leaf0 =
      uint64_t(j) * a.leaves_small + (off64 - uint64_t(j) * (a.n >> a.depth)) * (a.leaves_big - a.leaves_small);
  uint32_t *sw = reinterpret_cast<uint32_t *>(sm + L::kStage) + warp * 96;
  uint32_t *payload0 = reinterpret_cast<uint32_t *>(a.out + kHeaderBytes + uint64_t(kLeafBytes) * a.num_leaves);
  for (uint32_t f = uint32_t(warp) >> lgwl; f < nl; f += slots) {
    const uint32_t foff = LF[f].off, fcnt = LF[f].cnt, centre = LF[f].centre, fm = LF[f].m, words = LF[f].words;
    const unsigned long long word_off = LF[f].word_off;
    const uint64_t gl = leaf0 + f, goff = off64 + foff;
    if (gl >= a.num_leaves || goff + fcnt > a.n || word_off + words > a.payload_cap) {
      if (lt == 0) atomicOr(a.err, kErrInternal);
      continue;
    }
    const uint32_t r0 = uint32_t(LF[f].qref[0]), r1 = uint32_t(LF[f].qref[1]), r2 = uint32_t(LF[f].qref[2]);
    if (lt == 0) {
      uint4 *rec = reinterpret_cast<uint4 *>(a.out + kHeaderBytes + uint64_t(kLeafBytes) * gl);
      rec[0] = make_uint4(uint32_t(goff), uint32_t(goff >> 32), uint32_t(word_off), uint32_t(word_off >> 32));
      rec[1] = make_uint4(r0, r1, r2, fm);
    }
    if (IDX && a.perm) {
      const uint32_t *XI = reinterpret_cast<const uint32_t *>(sm + L::kIdx) + M.ilead + foff;
      for (uint32_t i = lt; i < fcnt; i += lstep) {
        const uint32_t src = i == 0 ? centre : (i - 1 < centre ? i - 1 : i);
        if (MULTI) a.perm[goff + i] = __ldg(a.idx + off64 + PL[foff + src]);
        else a.perm[goff + i] = XI[src];
      }
    }
    const uint32_t m0 = fm & 0xffu, m1 = (fm >> 8) & 0xffu, m2 = (fm >> 16) & 0xffu;
    const uint32_t w = m0 + m1 + m2;
    if (w == 0 || fcnt < 2) continue;
    uint32_t *payload = payload0 + word_off;
    const uint32_t h0 = m0 ? (1u << (m0 - 1)) - 1u : 0u;
    const uint32_t h1 = m1 ? (1u << (m1 - 1)) - 1u : 0u;
    const uint32_t h2 = m2 ? (1u << (m2 - 1)) - 1u : 0u;
    const uint32_t nsl = fcnt - 1, chunks = (nsl + 31) / 32;
    if (w >= 8 && w <= 32) {
      const C *x0 = Y0 + foff, *x1 = Y1 + foff, *x2 = Y2 + foff;
      for (uint32_t blk = lw; blk * 128u < nsl; blk += WL)
        pack_block(x0, x1, x2, r0 - h0, r1 - h1, r2 - h2, m0, m1, w, blk, centre, nsl, words, payload, lane);
      continue;
    }
    // w <= 32: word k of a chunk takes bits from lanes i0 = 32k / w on (at most nit of them)
    const uint32_t i0 = w <= 32 ? (32u * lane) / w : 0u;
    const int sh0 = int(i0 * w) - int(32u * lane);
    const uint32_t nit = w <= 32 ? (31u + w) / w + 1u : 0u;
    const C *x0 = Y0 + foff, *x1 = Y1 + foff, *x2 = Y2 + foff;
    for (uint32_t ch = lw; ch < chunks; ch += WL) {
      // this lane's particle as one w-bit value c_x | c_y << m_x | c_z << (m_x + m_y), in three limbs
      const uint32_t sl = ch * 32 + lane;
      uint32_t v0 = 0, v1 = 0, v2 = 0;
      if (sl < nsl) {
        const uint32_t p = sl < centre ? sl : sl + 1;
        const uint32_t cx = m0 ? uint32_t(x0[p]) - r0 + h0 : 0u;
        const uint32_t cy = m1 ? uint32_t(x1[p]) - r1 + h1 : 0u;
        const uint32_t cz = m2 ? uint32_t(x2[p]) - r2 + h2 : 0u;
        const unsigned long long y = (unsigned long long)cy << m0;
        v0 = cx | uint32_t(y);
        v1 = uint32_t(y >> 32);
        const uint32_t s2 = m0 + m1;
        const unsigned long long z = (unsigned long long)cz << (s2 & 31);
        if (s2 < 32) {
          v0 |= uint32_t(z);
          v1 |= uint32_t(z >> 32);
        } else {
          v1 |= uint32_t(z);
          v2 = uint32_t(z >> 32);
        }
      }
      if (w <= 32) {
        // lane k assembles word k of the chunk from the lanes whose values overlap it
        uint32_t word = 0;
        for (uint32_t t = 0; t < nit; ++t) {
          const uint32_t i = i0 + t;
          const uint32_t vi = __shfl_sync(0xffffffffu, v0, i & 31u);
          const int sh = sh0 + int(t * w);
          if (i < 32 && sh < 32) word |= sh >= 0 ? (vi << sh) : (vi >> -sh);
        }
        const uint32_t gw = ch * w + lane;
        if (lane < w && gw < words) __stcs(payload + gw, word);
      } else {
        for (uint32_t t = lane; t < w; t += 32) sw[t] = 0;
        __syncwarp();
        if (sl < nsl) {
          const uint32_t b = lane * w, k0 = b >> 5, sh = b & 31;
          const uint32_t nwd = (sh + w + 31) >> 5;
          atomicOr(&sw[k0], v0 << sh);
          if (nwd > 1) atomicOr(&sw[k0 + 1], __funnelshift_l(v0, v1, sh));
          if (nwd > 2) atomicOr(&sw[k0 + 2], __funnelshift_l(v1, v2, sh));
          if (nwd > 3) atomicOr(&sw[k0 + 3], __funnelshift_l(v2, 0u, sh));
        }
        __syncwarp();
        for (uint32_t t = lane; t < w; t += 32) {
          const uint32_t gw = ch * w + t;
          if (gw < words) __stcs(payload + gw, sw[t]);
        }
        __syncwarp();
      }
    }
  }
  // every warp is done with tensor memory before warp 0 frees it
  tmem_fence_before();
  __syncthreads();
  if (warp == 0) {
    tmem_fence_after();
    tmem_dealloc(M.tmem, kTmemCols);
  }
}

template <typename C, bool IDX, bool WIDEST, bool COST>
cudaError_t subtree_launch_as(const SubtreeLaunch &a, cudaStream_t st) {
  const uint32_t smem = SubL<C, IDX, sizeof(C) == 2 && !WIDEST && !COST>::kTotal;
  int per_sm = 0;
  cudaError_t e = resident_blocks<k_subtree<C, IDX, WIDEST, COST>>(kT, smem, &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  TraceScope ts(COST ? "k_subtree_cost" : "k_subtree", st);
  return launch_dependent(a.alone, k_subtree<C, IDX, WIDEST, COST>, dim3(unsigned(1ull << a.depth)), dim3(kT), smem, st, a);
}
template <typename C, bool IDX, bool WIDEST>
cudaError_t subtree_launch(const SubtreeLaunch &a, cudaStream_t st) {
  return a.cost_words ? subtree_launch_as<C, IDX, WIDEST, true>(a, st) : subtree_launch_as<C, IDX, WIDEST, false>(a, st);
}

}  // namespace

uint32_t subtree_capacity(int code_bytes, bool with_idx, bool multi) {
  if (code_bytes == 2 && multi)
    return with_idx ? SubL<uint16_t, true, true>::kCap : SubL<uint16_t, false, true>::kCap;
  return code_bytes == 2 ? (with_idx ? SubL<uint16_t, true, false>::kCap : SubL<uint16_t, false, false>::kCap)
                         : (with_idx ? SubL<uint32_t, true, false>::kCap : SubL<uint32_t, false, false>::kCap);
}

cudaError_t launch_subtree(const SubtreeLaunch &a, cudaStream_t st) {
  if (a.code_bytes == 2) {
    if (a.idx) return a.widest ? subtree_launch<uint16_t, true, true>(a, st) : subtree_launch<uint16_t, true, false>(a, st);
    return a.widest ? subtree_launch<uint16_t, false, true>(a, st) : subtree_launch<uint16_t, false, false>(a, st);
  }
  if (a.idx) return a.widest ? subtree_launch<uint32_t, true, true>(a, st) : subtree_launch<uint32_t, true, false>(a, st);
  return a.widest ? subtree_launch<uint32_t, false, true>(a, st) : subtree_launch<uint32_t, false, false>(a, st);
}

}  // namespace pcx
