// Bottom-up voxel sampling (Section 4.2 of the paper).
//
// The paper processes one node per workgroup with one 128^3 grid per SM in
// global memory (8 MB / 33 MB per workgroup, Sections 4.2.2-4.2.3).  Here a
// CTA handles one (parent, child octant) pair, an "item": the child's
// samples (its leaf points, or the voxels the child itself received one
// level below) all fall into one 64^3 octant of the parent's 128^3 grid
// (the observation of Section 4.2).  Sampling an item takes two passes over
// its samples, both in shared memory:
//
//  1. mark: every sample sets its cell's bit in a 32 KB occupancy bitmap of
//     the octant (the item's samples were asked into L2 when it started); a
//     block scan of the bitmap's population counts then stores, beside
//     every 32-cell word of the bitmap, the rank of its first occupied
//     cell, which numbers the item's D occupied cells 0..D-1 in cell order;
//  2. accumulate: every sample finds its cell's rank (two reads and one
//     population count) and updates the dense entry of that rank.
//
// No hashing and no probing: every lookup costs the same, D is exact before
// anything is accumulated (so the item's staging block is reserved to the
// record), and the voxels come out sorted by cell.  The dense entries of
// one pass hold 4688 to 17817 cells, depending on the layout; an item with
// more occupied cells takes its ranks in consecutive ranges, one accumulate
// pass each, and may hand ranges to other SMs.  Colour sums are exact
// integers in 32-bit words (16-bit fields whose wraps are listed, 32-bit
// sums while they provably cannot overflow, low and high words otherwise),
// because only 32-bit shared atomic adds are native; the single-sample modes
// (minimal-hash pick, first come of Section 4.2.1, random with the key of
// Listing 1) keep, per cell, the smallest key by a 64-bit atomicMin, which is
// native, and the colour of the sample that holds it.
//
// What bounds it: the shared-memory data pipe (0.43 wavefronts per active SM
// cycle in the largest level of 20M indoor points, 43 % of them the atomics'),
// instruction issue (40 % of the slots) and the barriers between an item's
// phases; levels of uneven items leave SMs idle at their end.  Measured against
// 64-bit atomic sums merged over equal lanes and 128-bit compare-and-swap picks
// (all levels of one build, GB300): 500M indoor points filtered 11.5 -> 8.2 ms,
// 50M aerial filtered 1.14 -> 0.72 ms, 200M indoor points picked 5.9 -> 5.4 ms.
//
// Every octant's voxels go to a staging area; a level scan then assigns
// each parent one contiguous voxel range (children are consecutive in node
// order), and the next level up copies the records to that range while it
// reads them (so each record is read once).
#include <cstddef>

#include "common.cuh"
#include "kernels.h"
#include "wgrid.cuh"

namespace lodk {

namespace {

// One CTA per SM with all of its shared memory.  (Two CTAs of 512 threads and
// 113 KB each hide each other's serial steps, but hold half the cells a pass
// and double the samples in flight, which then miss L2: 500M-point filtered
// build 9.6 against 8.3 ms per SM.)
constexpr int kVoxThreads = 1024;
constexpr int kVoxWarps = kVoxThreads / 32;
constexpr int kVoxCtasPerSm = 1;
constexpr uint32_t kSharedOff = 225 * 1024;       // VoxShared lies behind the arrays
constexpr int kSmemBytes = 226 * 1024;
constexpr uint32_t kBatch = 4u * kVoxThreads;  // samples of one CTA iteration
// 32 KB of occupancy bits (one word per 32 cells along x) and, per word, the
// 16-bit rank of its first occupied cell
constexpr uint32_t kWords = kOctCells / 32u;  // 8192
constexpr uint32_t kRankOff = kWords * 4u;
constexpr uint32_t kDenseOff = kRankOff + kWords * 2u;
// 16-bit field wraps of one accumulate pass (see update16): a leaf of at most
// 65,535 points has at most 254 + 255 + 254
constexpr uint32_t kMaxWraps = 768u;
constexpr uint32_t kWrapOff = kSharedOff - kMaxWraps * 4u;
constexpr uint32_t kDenseBytes = kWrapOff - kDenseOff;
// cells one accumulate pass holds; every layout is 32-bit words (64-bit keys
// first) followed by the 16-bit cell of each rank.  All updates are native
// 32-bit shared atomics: a 64-bit shared atomicAdd is a compare-and-swap loop
// here (measured, 32 lanes on random entries: 18.7 clocks per warp and SM
// against 2.8 for a 32-bit one, and 125 against 2.6 when the lanes share 32
// entries; a 64-bit atomicMin is native, 5.2).
constexpr uint32_t kCapLeaf = kDenseBytes / 10;    // filtered leaf, <= 65535 points: {R:16 G:16}, {B:16 n:16}
constexpr uint32_t kCapNarrow = kDenseBytes / 18;  // filtered, 32-bit sums: R, G, B, n
constexpr uint32_t kCapWide = kDenseBytes / 30;    // filtered, 64-bit sums: R, G, B (low and high words), n
constexpr uint32_t kCapPick = kDenseBytes / 22;    // single sample: u64 {key high word, index}, {index, rgba}, n
constexpr uint32_t kCapWeighted = kDenseBytes / 38;  // weighted: w R, w G, w B, w (low and high words), n
constexpr uint64_t kNarrowMaxSamples = 0xFFFFFFFFull / 255;  // 32-bit channel sums cannot overflow
constexpr uint64_t kLeafMaxSamples = 0xFFFFu;                // a 16-bit count cannot
constexpr uint64_t kMask40 = (1ull << 40) - 1;
constexpr uint32_t kNoRank = 0xFFFFFFFFu;
constexpr int kScan = (int)(kWords / 4u / kVoxThreads);  // 4-word groups of a thread in the rank scan
// Filtered staging records of cells of fewer than kPackMaxCount points carry
// their exact sums in the record's last word (10 bits per channel), so that
// neither the extraction nor the next level up touches the 16-byte sums
// array for them; larger cells keep the last word kNone and their sums in
// that array.
constexpr uint64_t kPackMaxCount = 1024;

// A channel's exact sum s over n < 1024 points and its rounded mean
// m = floor((s + floor(n/2)) / n) determine the remainder
// s + floor(n/2) - m n, which lies in [0, n); the three remainders, 10 bits
// each, fit below bit 30 (so the word never equals kNone).
__device__ __forceinline__ uint32_t pack_remainders(uint64_t sr, uint64_t sg, uint64_t sb, uint64_t n, uint32_t m) {
  const uint32_t nn = (uint32_t)n, h = nn >> 1;
  const uint32_t rr = (uint32_t)sr + h - (m & 255u) * nn;
  const uint32_t rg = (uint32_t)sg + h - ((m >> 8) & 255u) * nn;
  const uint32_t rb = (uint32_t)sb + h - ((m >> 16) & 255u) * nn;
  return rr | (rg << 10) | (rb << 20);
}

// The sums of a packed record {cell, mean rgba, n, remainders} in the
// layout of the sums array: {R | G << 40, G >> 24 | B << 16}.
__device__ __forceinline__ ulonglong2 unpack_sums(const int4& rec) {
  const uint32_t m = (uint32_t)rec.y, nn = (uint32_t)rec.z, w = (uint32_t)rec.w, h = nn >> 1;
  const uint64_t sr = (m & 255u) * nn + (w & 1023u) - h;
  const uint64_t sg = ((m >> 8) & 255u) * nn + ((w >> 10) & 1023u) - h;
  const uint64_t sb = ((m >> 16) & 255u) * nn + ((w >> 20) & 1023u) - h;
  return make_ulonglong2(sr | (sg << 40), (sg >> 24) | (sb << 16));
}

// an item's samples prefetched into L2 when it starts: at most this many
// bytes (152 SMs x 256 KB stays well inside the 126 MB L2)
constexpr uint64_t kPrefetchBytes = 256u * 1024u;

// Ask the bulk-copy unit to bring [p, p + bytes) into L2 (p 16-byte
// aligned, bytes a multiple of 16; nothing waits on it).
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Ranks, among the item's occupied cells (cell order), of a thread's four
// samples' cells, minus lo; kNoRank for samples without ok[k] (ALL: every
// sample counts) or outside [lo, lo + span).  Cells are always valid.  The bitmap is read-only during an accumulate pass, so
// the reads are issued together.  Word ranks are 16 bits: items of 65,536
// occupied cells and more (qbase != nullptr) store them relative to the
// first cell of their quarter of the octant (2048 words).
template <bool ALL>
__device__ __forceinline__ void cell_ranks4(const uint32_t* bits, const uint16_t* wrank, const uint32_t* qbase,
                                            const uint32_t (&cell)[4], const bool* ok, uint32_t lo, uint32_t span,
                                            uint32_t (&rk)[4]) {
  uint32_t w[4], b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    w[k] = bits[cell[k] >> 5];
    b[k] = wrank[cell[k] >> 5];
  }
  if (qbase) {
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] += qbase[cell[k] >> 16];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t r = b[k] + __popc(w[k] & ((1u << (cell[k] & 31u)) - 1u)) - lo;
    rk[k] = (ALL || ok[k]) && r < span ? r : kNoRank;
  }
}

struct ItemInfo {
  uint32_t tile;
  uint64_t g;        // absolute node id of the item (the child)
  uint32_t kx, ky, kz;
  uint32_t Lp;       // parent log2 edge
  int32_t pmin[3];
  bool leaf;
  uint64_t n;        // samples
  uint64_t npts;     // original points in the child's cube
};

__device__ __forceinline__ uint32_t find_tile(const uint32_t* prefix, uint32_t n_tiles, uint32_t it) {
  uint32_t lo = 0, hi = n_tiles;  // largest t with prefix[t] <= it
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (prefix[mid] <= it) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Local cell (x | y << 6 | z << 12) of a point in the item's octant: bits
// L - 7 .. L - 2 of each offset from the parent's corner (edge 2^L), moved to
// their place by one rotation per axis.  Bits that a rotation wraps around
// are masked off, or zero (L < 7: the offset has no more than L bits).
struct CellMap {
  uint32_t mx, my, mz, s;
  __device__ __forceinline__ explicit CellMap(const ItemInfo& I)
      : mx((uint32_t)I.pmin[0]), my((uint32_t)I.pmin[1]), mz((uint32_t)I.pmin[2]), s(I.Lp - 7u) {}
  __device__ __forceinline__ uint32_t operator()(const int4& q) const {
    const uint32_t dx = (uint32_t)q.x - mx, dy = (uint32_t)q.y - my, dz = (uint32_t)q.z - mz;
    return (__funnelshift_r(dx, dx, s) & 63u) | (__funnelshift_r(dy, dy, s - 6u) & 0xFC0u) |
           (__funnelshift_r(dz, dz, s - 12u) & 0x3F000u);
  }
};

// Local cell of a child's voxel (its cell in the child's 128^3 grid).
__device__ __forceinline__ uint32_t voxel_cell(uint32_t cell) {
  const uint32_t x = (cell & 127u) >> 1, y = ((cell >> 7) & 127u) >> 1, z = ((cell >> 14) & 127u) >> 1;
  return x | (y << 6) | (z << 12);
}

// Cell of the parent's 128^3 grid of a local cell.
__device__ __forceinline__ uint32_t parent_cell(uint32_t l, const ItemInfo& I) {
  return ((I.kx << 6) | (l & 63u)) | (((I.ky << 6) | ((l >> 6) & 63u)) << 7) | (((I.kz << 6) | (l >> 12)) << 14);
}

}  // namespace

// Shared state of one voxel CTA.
struct VoxShared {
  uint32_t D;                  // occupied cells of the item
  uint32_t r0, r1;             // rank interval this CTA accumulates
  uint32_t nch;                // inner items: children
  unsigned long long stage;    // first staging record of the item (rank 0)
  int32_t cmin[3];             // header: the child's min corner
  uint32_t n_wraps;            // 16-bit field wraps listed by the pass
  unsigned long long cparent, cfirst;  // header: parent node, first child (absolute)
  unsigned long long nbase;    // header: the tile's first node
  unsigned long long pfirst;   // header: the parent's first child (absolute)
  unsigned long long pbase;    // header: the child's first leaf point (absolute)
  uint32_t cpre[9];            // inner items: prefix of the children's record counts
  uint32_t settle;             // single sample: the pass needs settle_pick
  unsigned long long cstage[8];  // ... their first staging records
  unsigned long long cdense[8];  // ... their places in the voxel array
  uint32_t wsum[kVoxWarps];
  uint32_t qbase[4];           // rank of the first cell of each quarter of the octant
  uint4 border[8];             // weighted: the border lists of the parent's children, in octant order
  uint32_t pmask;              // ... and which octants they are
  uint32_t pick_level, idx_bound;  // header: level of the parent, bound of the tile's input indices
  uint32_t next;               // the item or unit taken next
  ItemInfo I;
};
static_assert(sizeof(VoxShared) <= kSmemBytes - kSharedOff, "VoxShared fits behind the arrays");

// Reserve `n` consecutive slots of the unit queue; false when it is full
// (the reservation is all or nothing, so no slot is left unwritten).
__device__ __forceinline__ bool reserve_units(unsigned int* count, uint32_t cap, uint32_t n, uint32_t* first) {
  uint32_t old = *((volatile unsigned int*)count);
  for (int tries = 0; tries < 4096; ++tries) {
    if (old + n > cap) return false;
    const uint32_t prev = atomicCAS(count, old, old + n);
    if (prev == old) {
      *first = old;
      return true;
    }
    old = prev;
  }
  return false;
}

// Everything a voxel CTA keeps in shared memory is one dynamic array, so that
// the phases below address it as shared memory.
extern __shared__ __align__(16) unsigned char vox_smem[];

namespace {

__device__ __forceinline__ uint32_t* vox_bits() { return reinterpret_cast<uint32_t*>(vox_smem); }
__device__ __forceinline__ uint16_t* vox_wrank() { return reinterpret_cast<uint16_t*>(vox_smem + kRankOff); }
__device__ __forceinline__ uint32_t* vox_fields() { return reinterpret_cast<uint32_t*>(vox_smem + kDenseOff); }
__device__ __forceinline__ uint32_t* vox_wraps() { return reinterpret_cast<uint32_t*>(vox_smem + kWrapOff); }
__device__ __forceinline__ VoxShared& vox_shared() { return *reinterpret_cast<VoxShared*>(vox_smem + kSharedOff); }

// The dense entries: one array of `cap` words per field (64-bit keys first),
// then the 16-bit cell of each rank.
template <uint32_t WORDS, uint32_t CAP>
__device__ __forceinline__ uint16_t* vox_cells() {
  return reinterpret_cast<uint16_t*>(vox_fields() + WORDS * CAP);
}

// Empty dense entries: all zero bytes in the averaging modes (whatever the
// layout), ~0 keys and zero counts in the single-sample modes.
template <int MODE>
__device__ __forceinline__ void vox_clear_dense() {
  if (MODE == LOD_FILTER || MODE == LOD_WEIGHTED) {
    uint4* z = reinterpret_cast<uint4*>(vox_smem + kDenseOff);
    for (uint32_t i = threadIdx.x; i < kDenseBytes / 16u; i += kVoxThreads) z[i] = make_uint4(0, 0, 0, 0);
  } else {
    unsigned long long* E = reinterpret_cast<unsigned long long*>(vox_smem + kDenseOff);
    for (uint32_t i = threadIdx.x; i < kCapPick; i += kVoxThreads) {
      E[i] = ~0ull;
      vox_fields()[4u * kCapPick + i] = 0u;
    }
  }
}

// Set the occupancy bits of a thread's four samples (cells with ok[k]).
// The four words are read first, back to back, and only bits found clear are
// set: most samples find theirs set already, and samples that share a word
// (32 cells in a row, often a whole warp's) then cost one broadcast read
// where their atomics would be taken one after another.  A read that misses
// a concurrent update only costs a redundant atomic.
template <bool ALL>
__device__ __forceinline__ void mark4(const uint32_t (&cell)[4], const bool* ok) {
  uint32_t cur[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) cur[k] = ALL || ok[k] ? *((volatile uint32_t*)&vox_bits()[cell[k] >> 5]) : ~0u;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (!((cur[k] >> (cell[k] & 31u)) & 1u)) atomicOr(&vox_bits()[cell[k] >> 5], 1u << (cell[k] & 31u));
}

__device__ __forceinline__ int4 ld_if(const int4* p, uint32_t tid, int k, uint32_t rem) {
  int4 q = make_int4(0, 0, 0, 0);
  if (tid + k * kVoxThreads < rem) q = __ldcg(p + k * kVoxThreads);
  return q;
}

// A thread's samples of a contiguous array are p[tid + k * kVoxThreads] for
// k = 0..3, then the next kBatch: its next four are loaded before its current
// four are worked on (the item's samples were asked into L2 when it started,
// so a load is an L2 latency that the other work covers).  `rem` counts the
// samples from p on, so offsets stay small whatever the item's size.  While
// two whole batches are left (FULL) no bound is checked.

// Pass 1 (mark the occupied cells) of a leaf's points.
__device__ __forceinline__ void mark_leaf(const int4* p, uint32_t rem) {
  const CellMap cm(vox_shared().I);
  const uint32_t tid = threadIdx.x;
  p += tid;
  int4 q0 = ld_if(p, tid, 0, rem), q1 = ld_if(p, tid, 1, rem), q2 = ld_if(p, tid, 2, rem), q3 = ld_if(p, tid, 3, rem);
  while (rem >= 2 * kBatch) {
    const uint32_t cell[4] = {cm(q0), cm(q1), cm(q2), cm(q3)};
    p += kBatch;
    rem -= kBatch;
    q0 = __ldcg(p), q1 = __ldcg(p + kVoxThreads), q2 = __ldcg(p + 2 * kVoxThreads), q3 = __ldcg(p + 3 * kVoxThreads);
    mark4<true>(cell, nullptr);
  }
  for (;;) {
    const uint32_t cell[4] = {cm(q0), cm(q1), cm(q2), cm(q3)};
    const bool ok[4] = {tid < rem, tid + kVoxThreads < rem, tid + 2 * kVoxThreads < rem, tid + 3 * kVoxThreads < rem};
    const bool more = rem > kBatch;
    if (more) {
      p += kBatch;
      rem -= kBatch;
      q0 = ld_if(p, tid, 0, rem), q1 = ld_if(p, tid, 1, rem), q2 = ld_if(p, tid, 2, rem), q3 = ld_if(p, tid, 3, rem);
    }
    mark4<false>(cell, ok);
    if (!more) break;
  }
}

// The same with kept indices: the leaf is read from the 32-byte staging
// records and, when out is given, published to the point / index arrays,
// contiguously (idempotent: a retried build writes the same values).
__device__ __forceinline__ void mark_wide(const int4* w, uint32_t rem, int4* out, uint32_t* out_idx) {
  const CellMap cm(vox_shared().I);
  const uint32_t tid = threadIdx.x;
  const bool publish = out != nullptr;
  w += 2u * tid;
  out += tid;
  out_idx += tid;
  auto load = [&](uint32_t off, int4& q, uint32_t& x) {
    q = make_int4(0, 0, 0, 0);
    x = 0u;
    if (tid + off < rem) ld_wide(w + 2u * off, q, x);
  };
  int4 q0, q1, q2, q3;
  uint32_t x0, x1, x2, x3;
  load(0, q0, x0), load(kVoxThreads, q1, x1), load(2 * kVoxThreads, q2, x2), load(3 * kVoxThreads, q3, x3);
  for (;;) {
    uint32_t cell[4];
    bool ok[4];
    auto take = [&](int k, int4& q, uint32_t& x) {
      ok[k] = tid + k * kVoxThreads < rem;
      cell[k] = cm(q);
      if (ok[k] && publish) {
        out[k * kVoxThreads] = q;
        out_idx[k * kVoxThreads] = x;
      }
      load(kBatch + k * kVoxThreads, q, x);
    };
    take(0, q0, x0), take(1, q1, x1), take(2, q2, x2), take(3, q3, x3);
    mark4<false>(cell, ok);
    if (rem <= kBatch) break;
    rem -= kBatch;
    w += 2u * kBatch;
    out += kBatch;
    out_idx += kBatch;
  }
}

// The children's voxels, one flat sequence of `total` staged records: child
// ci of sample f, walking forward.
__device__ __forceinline__ uint64_t child_record(const VoxShared& S, uint32_t f, uint32_t& ci) {
  while (f >= S.cpre[ci + 1]) ++ci;
  return S.cstage[ci] + (f - S.cpre[ci]);
}

// Pass 1 of an inner child: mark its voxels [first, total) and, with `dense`,
// publish them there (idempotent; an array found too small makes the build rerun with the
// exact size).  Filtered records are published without their packed sums.
template <bool FILT>
__device__ __forceinline__ void mark_inner(const int4* stage_in, uint32_t first, uint32_t total, int4* dense, uint64_t dense_cap) {
  const VoxShared& S = vox_shared();
  uint32_t cl = 0, cp = 0;  // children of the samples being loaded and marked
  auto load = [&](uint32_t f, int4& q) {
    q = make_int4(0, 0, 0, 0);
    if (f < total) q = __ldcg(stage_in + child_record(S, f, cl));
  };
  uint32_t f = first + threadIdx.x;
  int4 q0, q1, q2, q3;
  load(f, q0), load(f + kVoxThreads, q1), load(f + 2 * kVoxThreads, q2), load(f + 3 * kVoxThreads, q3);
  for (; f < total; f += kBatch) {
    uint32_t cell[4];
    bool ok[4];
    auto take = [&](int k, int4& q) {
      const uint32_t fk = f + k * kVoxThreads;
      ok[k] = fk < total;
      cell[k] = voxel_cell((uint32_t)q.x);
      if (ok[k] && dense) {
        while (fk >= S.cpre[cp + 1]) ++cp;
        const uint64_t dst = S.cdense[cp] + (fk - S.cpre[cp]);
        if (dst < dense_cap) dense[dst] = FILT ? make_int4(q.x, q.y, q.z, (int)kNone) : q;
      }
      load(fk + kBatch, q);
    };
    take(0, q0), take(1, q1), take(2, q2), take(3, q3);
    mark4<false>(cell, ok);
  }
}

// Pass 2 of a filtered leaf of at most kLeafMaxSamples points: {R:16 G:16}
// and {B:16 n:16}, two atomics per point.  A 16-bit field that wraps is seen
// by exactly one of them (in the value it gets back); those wraps, at most
// kMaxWraps per pass, are listed and put back at extraction.
template <bool ALL>
__device__ __forceinline__ void add16x4(const uint32_t (&cell)[4], const uint32_t (&col)[4], const bool* ok, const uint32_t* qbase,
                                        uint32_t lo, uint32_t span) {
  VoxShared& S = vox_shared();
  uint32_t* const W0 = vox_fields();
  uint32_t* const W1 = W0 + kCapLeaf;
  uint32_t rk[4], o0[4], o1[4];
  cell_ranks4<ALL>(vox_bits(), vox_wrank(), qbase, cell, ok, lo, span, rk);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    o0[k] = 0u;
    o1[k] = 1u;
    if (rk[k] < span) {
      o0[k] = atomicAdd(&W0[rk[k]], __byte_perm(col[k], 0u, 0x4140));  // R | G << 16
      o1[k] = atomicAdd(&W1[rk[k]], __byte_perm(col[k], 1u, 0x5452));  // B | 1 << 16
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (o1[k] == 0u) vox_cells<2, kCapLeaf>()[rk[k]] = (uint16_t)cell[k];
    if (((o0[k] | o1[k]) & 0x80008000u) == 0u) continue;  // every field below 2^15: nothing wraps
    const uint32_t r = col[k] & 255u, g = (col[k] >> 8) & 255u, b = (col[k] >> 16) & 255u;
    const uint32_t wr = ((o0[k] & 0xFFFFu) + r) >> 16, wb = ((o1[k] & 0xFFFFu) + b) >> 16;
    const uint32_t wg = o0[k] + (r | (g << 16)) < o0[k] ? 1u : 0u;
    if (wr | wg | wb) {
      const uint32_t e = atomicAdd(&S.n_wraps, 1u);
      if (e < kMaxWraps) vox_wraps()[e] = rk[k] | (wr << 16) | (wg << 17) | (wb << 18);
    }
  }
}

__device__ __forceinline__ void acc_leaf16(const int4* p, uint32_t rem, uint32_t lo, uint32_t span) {
  const CellMap cm(vox_shared().I);
  const uint32_t* const qbase = vox_shared().D > 0xFFFFu ? vox_shared().qbase : nullptr;
  const uint32_t tid = threadIdx.x;
  p += tid;
  int4 q0 = ld_if(p, tid, 0, rem), q1 = ld_if(p, tid, 1, rem), q2 = ld_if(p, tid, 2, rem), q3 = ld_if(p, tid, 3, rem);
  while (rem >= 2 * kBatch) {
    const uint32_t cell[4] = {cm(q0), cm(q1), cm(q2), cm(q3)};
    const uint32_t col[4] = {(uint32_t)q0.w, (uint32_t)q1.w, (uint32_t)q2.w, (uint32_t)q3.w};
    p += kBatch;
    rem -= kBatch;
    q0 = __ldcg(p), q1 = __ldcg(p + kVoxThreads), q2 = __ldcg(p + 2 * kVoxThreads), q3 = __ldcg(p + 3 * kVoxThreads);
    add16x4<true>(cell, col, nullptr, qbase, lo, span);
  }
  for (;;) {
    const uint32_t cell[4] = {cm(q0), cm(q1), cm(q2), cm(q3)};
    const uint32_t col[4] = {(uint32_t)q0.w, (uint32_t)q1.w, (uint32_t)q2.w, (uint32_t)q3.w};
    const bool ok[4] = {tid < rem, tid + kVoxThreads < rem, tid + 2 * kVoxThreads < rem, tid + 3 * kVoxThreads < rem};
    const bool more = rem > kBatch;
    if (more) {
      p += kBatch;
      rem -= kBatch;
      q0 = ld_if(p, tid, 0, rem), q1 = ld_if(p, tid, 1, rem), q2 = ld_if(p, tid, 2, rem), q3 = ld_if(p, tid, 3, rem);
    }
    add16x4<false>(cell, col, ok, qbase, lo, span);
    if (!more) break;
  }
}

// One filtered update with full sums: four 32-bit fields (WIDE false), or low
// and high words (the add that wraps a low word carries) and the count.
template <bool WIDE>
__device__ __forceinline__ void add_sums(uint32_t rk, uint32_t cell, uint64_t r, uint64_t g, uint64_t b, uint32_t n) {
  uint32_t* const F = vox_fields() + rk;
  if (!WIDE) {
    atomicAdd(F, (uint32_t)r);
    atomicAdd(F + kCapNarrow, (uint32_t)g);
    atomicAdd(F + 2u * kCapNarrow, (uint32_t)b);
    if (atomicAdd(F + 3u * kCapNarrow, n) == 0u) vox_cells<4, kCapNarrow>()[rk] = (uint16_t)cell;
  } else {
    auto add64 = [&](uint32_t f, uint64_t s) {
      const uint32_t l = (uint32_t)s, old = atomicAdd(F + f * kCapWide, l);
      const uint32_t h = (uint32_t)(s >> 32) + (old + l < old ? 1u : 0u);
      if (h) atomicAdd(F + (f + 1u) * kCapWide, h);
    };
    add64(0u, r);
    add64(2u, g);
    add64(4u, b);
    if (atomicAdd(F + 6u * kCapWide, n) == 0u) vox_cells<7, kCapWide>()[rk] = (uint16_t)cell;
  }
}

// Pass 2 of a filtered leaf of more points.
template <bool WIDE>
__device__ __forceinline__ void acc_leaf_sums(const int4* p, uint32_t rem, uint32_t lo, uint32_t span) {
  VoxShared& S = vox_shared();
  const CellMap cm(S.I);
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  p += threadIdx.x;
  for (;;) {
    uint32_t cell[4], rk[4], col[4];
    bool ok[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ok[k] = threadIdx.x + k * kVoxThreads < rem;
      int4 q = make_int4(0, 0, 0, 0);
      if (ok[k]) q = __ldcg(p + k * kVoxThreads);
      cell[k] = ok[k] ? cm(q) : 0u;
      col[k] = (uint32_t)q.w;
    }
    cell_ranks4<false>(vox_bits(), vox_wrank(), qbase, cell, ok, lo, span, rk);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (rk[k] != kNoRank) add_sums<WIDE>(rk[k], cell[k], col[k] & 255u, (col[k] >> 8) & 255u, (col[k] >> 16) & 255u, 1u);
    if (rem <= kBatch) break;
    rem -= kBatch;
    p += kBatch;
  }
}

// Pass 2 of a filtered inner child: its voxels with their exact sums, which
// travel in the record (cells of fewer than 1024 points) or lie in the sums
// array.
template <bool WIDE>
__device__ __forceinline__ void acc_inner_sums(const int4* stage_in, const ulonglong2* sums_in, uint32_t total, uint32_t lo,
                                            uint32_t span) {
  VoxShared& S = vox_shared();
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  uint32_t cl = 0, cs = 0;
  auto load = [&](uint32_t f, int4& q) {
    q = make_int4(0, 0, 0, 0);
    if (f < total) q = __ldcg(stage_in + child_record(S, f, cl));
  };
  uint32_t f = threadIdx.x;
  int4 q0, q1, q2, q3;
  load(f, q0), load(f + kVoxThreads, q1), load(f + 2 * kVoxThreads, q2), load(f + 3 * kVoxThreads, q3);
  for (; f < total; f += kBatch) {
    ulonglong2 sm[4];
    uint32_t cell[4], rk[4], n[4];
    bool ok[4];
    auto take = [&](int k, int4& q) {
      const uint32_t fk = f + k * kVoxThreads;
      ok[k] = fk < total;
      if ((uint32_t)q.w != kNone) sm[k] = unpack_sums(q);
      else sm[k] = __ldcg(sums_in + child_record(S, fk, cs));
      cell[k] = voxel_cell((uint32_t)q.x);
      n[k] = (uint32_t)q.z;
      load(fk + kBatch, q);
    };
    take(0, q0), take(1, q1), take(2, q2), take(3, q3);
    cell_ranks4<false>(vox_bits(), vox_wrank(), qbase, cell, ok, lo, span, rk);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (rk[k] != kNoRank)
        add_sums<WIDE>(rk[k], cell[k], sm[k].x & kMask40, (sm[k].x >> 40) | ((sm[k].y & 0xFFFFull) << 24), sm[k].y >> 16, n[k]);
  }
}

// Single-sample modes.  Each cell keeps the smallest {high word of the key,
// input index} (one native 64-bit atomicMin).  A sample that lowered it, and
// still holds it on a second look, leaves {index, colour} beside it; the
// extraction takes them when the index is the one kept.  Two things make the
// pass settle its cells once more by whole keys (settle_pick): two keys of
// one cell that share their high word (the later update of the two finds the
// other's word), and a slower sample's {index, colour} written over the
// winner's.  (Reading the winner back from its position instead of keeping
// its colour cost more: extraction 1.65 against 0.30 ms per SM on a 200M-point
// build.)
struct PickArgs {
  uint32_t lo, span, level, idx_bound;
  unsigned long long out_at;  // extraction: staging record of rank lo
  int4* stage_out;
  uint64_t stage_cap;
  unsigned int* error;
};

__device__ __forceinline__ unsigned long long* pick_keys() { return reinterpret_cast<unsigned long long*>(vox_fields()); }
__device__ __forceinline__ uint2* pick_pays() { return reinterpret_cast<uint2*>(vox_fields()) + kCapPick; }
__device__ __forceinline__ uint32_t* pick_counts() { return vox_fields() + 4u * kCapPick; }

// The upper word of a sample's key (first come: the key is the 32-bit index
// itself, unique, so it takes the upper word's place).
template <int MODE>
__device__ __forceinline__ uint32_t pick_high(uint32_t ix, uint32_t level) {
  return MODE == LOD_FIRST ? ix : (uint32_t)(pick_key<MODE>(ix, level) >> 32);
}

template <int MODE>
__device__ __forceinline__ void pick_sample(const PickArgs& P, uint32_t rk, uint32_t cell, uint32_t ix, uint32_t rgba, uint32_t n) {
  const uint32_t h = pick_high<MODE>(ix, P.level);
  const unsigned long long mine = ((unsigned long long)h << 32) | ix;
  const unsigned long long old = atomicMin(&pick_keys()[rk], mine);
  if (atomicAdd(&pick_counts()[rk], n) == 0u) vox_cells<5, kCapPick>()[rk] = (uint16_t)cell;
  if (old > mine) {
    if (*((volatile unsigned long long*)&pick_keys()[rk]) == mine) pick_pays()[rk] = make_uint2(ix, rgba);
  }
  if ((uint32_t)(old >> 32) == h) vox_shared().settle = 1u;
}

// A leaf's points and input indices.
template <int MODE>
__device__ __forceinline__ void pick_leaf(const PickArgs& P, const int4* p, const uint32_t* pidx, uint32_t total) {
  VoxShared& S = vox_shared();
  const CellMap cm(S.I);
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  const uint32_t tid = threadIdx.x;
  uint32_t rem = total;
  p += tid;
  pidx += tid;
  auto load = [&](uint32_t off, int4& q, uint32_t& x) {
    q = make_int4(0, 0, 0, 0);
    x = 0u;
    if (tid + off < rem) {
      q = __ldcg(p + off);
      x = __ldcg(pidx + off);
    }
  };
  int4 q0, q1, q2, q3;
  uint32_t x0, x1, x2, x3;
  load(0, q0, x0), load(kVoxThreads, q1, x1), load(2 * kVoxThreads, q2, x2), load(3 * kVoxThreads, q3, x3);
  for (;;) {
    uint32_t cell[4], rk[4], ix[4], col[4];
    bool ok[4];
    auto take = [&](int k, int4& q, uint32_t& x) {
      ok[k] = tid + k * kVoxThreads < rem;
      cell[k] = cm(q);
      ix[k] = x;
      col[k] = (uint32_t)q.w;
      load(kBatch + k * kVoxThreads, q, x);
    };
    take(0, q0, x0), take(1, q1, x1), take(2, q2, x2), take(3, q3, x3);
    cell_ranks4<false>(vox_bits(), vox_wrank(), qbase, cell, ok, P.lo, P.span, rk);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (rk[k] != kNoRank) pick_sample<MODE>(P, rk[k], cell[k], ix[k], col[k], 1u);
    if (rem <= kBatch) break;
    rem -= kBatch;
    p += kBatch;
    pidx += kBatch;
  }
}

template <int MODE>
__device__ __forceinline__ void pick_inner(const PickArgs& P, const int4* stage_in, uint32_t total) {
  VoxShared& S = vox_shared();
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  uint32_t cl = 0;
  auto load = [&](uint32_t f, int4& q) {
    q = make_int4(0, 0, 0, 0);
    if (f < total) q = __ldcg(stage_in + child_record(S, f, cl));
  };
  uint32_t f = threadIdx.x;
  int4 q0, q1, q2, q3;
  load(f, q0), load(f + kVoxThreads, q1), load(f + 2 * kVoxThreads, q2), load(f + 3 * kVoxThreads, q3);
  for (; f < total; f += kBatch) {
    uint32_t cell[4], rk[4], ix[4], n[4], col[4];
    bool ok[4];
    auto take = [&](int k, int4& q) {
      const uint32_t fk = f + k * kVoxThreads;
      ok[k] = fk < total;
      cell[k] = voxel_cell((uint32_t)q.x);
      ix[k] = (uint32_t)q.w;
      n[k] = (uint32_t)q.z;
      col[k] = (uint32_t)q.y;
      load(fk + kBatch, q);
    };
    take(0, q0), take(1, q1), take(2, q2), take(3, q3);
    cell_ranks4<false>(vox_bits(), vox_wrank(), qbase, cell, ok, P.lo, P.span, rk);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (rk[k] != kNoRank) pick_sample<MODE>(P, rk[k], cell[k], ix[k], col[k], n[k]);
  }
}

// Settles an extracted pass by whole keys: the smallest key of every cell
// first, then the sample that holds it (keys of distinct samples differ)
// writes colour and index of the cell's record.  Rare, so it is one sample at
// a time and keeps its registers to itself.  Every thread of the CTA calls
// it; the entries are empty before and after.
template <int MODE>
__device__ __noinline__ void settle_pick(PickArgs P, const int4* src, const uint32_t* pidx, bool leaf, uint32_t total) {
  VoxShared& S = vox_shared();
  unsigned long long* const E = pick_keys();
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  const CellMap cm(S.I);
  for (int step = 0; step < 2; ++step) {
    __syncthreads();
    uint32_t ci = 0;
    for (uint32_t i0 = threadIdx.x; i0 < total; i0 += kVoxThreads) {
      uint32_t cell, rgba, ix;
      if (leaf) {
        const int4 q = __ldcg(src + i0);
        cell = cm(q);
        rgba = (uint32_t)q.w;
        ix = __ldcg(pidx + i0);
      } else {
        const int4 q = __ldcg(src + child_record(S, i0, ci));
        cell = voxel_cell((uint32_t)q.x);
        rgba = (uint32_t)q.y;
        ix = (uint32_t)q.w;
      }
      const uint32_t word = cell >> 5;
      const uint32_t rk = vox_wrank()[word] + (qbase ? qbase[cell >> 16] : 0u) +
                          __popc(vox_bits()[word] & ((1u << (cell & 31u)) - 1u)) - P.lo;
      if (rk < P.span) {
        const unsigned long long key = pick_key<MODE>(ix, P.level);
        if (step == 0) {
          atomicMin(&E[rk], key);
        } else if (E[rk] == key) {
          if (ix >= P.idx_bound) atomicOr(P.error, kErrInternal);
          if (P.out_at + rk < P.stage_cap) {
            P.stage_out[P.out_at + rk].y = (int)rgba;
            P.stage_out[P.out_at + rk].w = (int)ix;
          }
        }
      }
      if (total - i0 <= kVoxThreads) break;  // (i0 + kVoxThreads may not fit 32 bits)
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < P.span; i += kVoxThreads) E[i] = ~0ull;
  if (threadIdx.x == 0) S.settle = 0;
}

// Neighbourhood-weighted average (Section 4.2.4; see k_weighted.cu): a sample
// adds its weight and weighted colours to those of its 2x2x2 cells that lie in
// the item's octant, are occupied and have a rank of the pass.  Sums are exact
// 64-bit integers in low and high words (a weighted colour has at most 32
// bits, so the high word only counts the low word's wraps).
__device__ __forceinline__ void add_weighted(const WBlock& b, uint32_t rgba, const uint32_t* qbase, uint32_t lo, uint32_t span) {
  const ItemInfo& I = vox_shared().I;
  const uint32_t oct[3] = {I.kx, I.ky, I.kz};
  float sq[3][2];
  bool in[3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float e1 = __fsub_rn(b.e0[a], 1.0f);
    sq[a][0] = __fmul_rn(b.e0[a], b.e0[a]);
    sq[a][1] = __fmul_rn(e1, e1);
    in[a][0] = ((b.j1[a] - 1) >> 6) == (int32_t)oct[a];
    in[a][1] = (b.j1[a] >> 6) == (int32_t)oct[a];
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int kx = (k >> 2) & 1, ky = (k >> 1) & 1, kz = k & 1;
    if (!(in[0][kx] && in[1][ky] && in[2][kz])) continue;
    const uint32_t w = w_weight(__fadd_rn(__fadd_rn(sq[0][kx], sq[1][ky]), sq[2][kz]));
    if (!w) continue;
    const uint32_t cell = ((uint32_t)(b.j1[0] - 1 + kx) & 63u) | (((uint32_t)(b.j1[1] - 1 + ky) & 63u) << 6) |
                          (((uint32_t)(b.j1[2] - 1 + kz) & 63u) << 12);
    const uint32_t word = vox_bits()[cell >> 5], bit = cell & 31u;
    if (!((word >> bit) & 1u)) continue;
    const uint32_t rk = vox_wrank()[cell >> 5] + (qbase ? qbase[cell >> 16] : 0u) + __popc(word & ((1u << bit) - 1u)) - lo;
    if (rk >= span) continue;
    uint32_t* const F = vox_fields() + rk;
    const uint32_t v[4] = {w * (rgba & 255u), w * ((rgba >> 8) & 255u), w * ((rgba >> 16) & 255u), w};
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const uint32_t old = atomicAdd(F + 2u * f * kCapWeighted, v[f]);
      if (old + v[f] < old) atomicAdd(F + (2u * f + 1u) * kCapWeighted, 1u);
    }
  }
}

// The sample's own cell takes its count.
__device__ __forceinline__ void add_weighted_own(uint32_t cell, uint32_t n, const uint32_t* qbase, uint32_t lo, uint32_t span) {
  const uint32_t word = vox_bits()[cell >> 5];
  const uint32_t rk = vox_wrank()[cell >> 5] + (qbase ? qbase[cell >> 16] : 0u) + __popc(word & ((1u << (cell & 31u)) - 1u)) - lo;
  if (rk < span && atomicAdd(vox_fields() + 8u * kCapWeighted + rk, n) == 0u) vox_cells<9, kCapWeighted>()[rk] = (uint16_t)cell;
}

// Pass 2 of the weighted mode: the item's own samples, then its siblings'
// border lists.  Issue-bound (up to eight weights a sample), so the samples
// are taken one at a time.
__device__ __forceinline__ void acc_weighted(const int4* src, const int4* border_list, bool leaf, uint32_t total, uint32_t lo,
                                             uint32_t span) {
  VoxShared& S = vox_shared();
  const uint32_t* const qbase = S.D > 0xFFFFu ? S.qbase : nullptr;
  const CellMap cm(S.I);
  const uint32_t oct = (S.I.kx << 2) | (S.I.ky << 1) | S.I.kz;
  uint32_t ci = 0;
  for (uint32_t i = threadIdx.x; i < total; i += kVoxThreads) {
    if (leaf) {
      const int4 q = __ldcg(src + i);
      add_weighted_own(cm(q), 1u, qbase, lo, span);
      add_weighted(w_point_block(q, S.I.pmin, S.I.Lp), (uint32_t)q.w, qbase, lo, span);
    } else {
      const int4 q = __ldcg(src + child_record(S, i, ci));
      add_weighted_own(voxel_cell((uint32_t)q.x), (uint32_t)q.z, qbase, lo, span);
      add_weighted(w_voxel_block((uint32_t)q.x, oct), (uint32_t)q.y, qbase, lo, span);
    }
    if (total - i <= kVoxThreads) break;  // (i + kVoxThreads may not fit 32 bits)
  }
  for (uint32_t k = 0, r = 0; k < 8; ++k) {
    if (!((S.pmask >> k) & 1u)) continue;
    const uint4 L = S.border[r++];
    if (k == oct) continue;
    const int4* const e = border_list + (L.x | ((uint64_t)L.y << 32));
    for (uint32_t i = threadIdx.x; i < L.z; i += kVoxThreads) {
      const int4 q = __ldcg(e + i);
      if (L.w) add_weighted(w_point_block(q, S.I.pmin, S.I.Lp), (uint32_t)q.w, qbase, lo, span);
      else add_weighted(w_voxel_block((uint32_t)q.x & 0x1FFFFFu, k), (uint32_t)q.y, qbase, lo, span);
      if (L.z - i <= kVoxThreads) break;
    }
  }
}

// The cell of rank r (its lower 16 bits are kept beside the entry): the
// upper two bits are the quarter of the octant the rank lies in.
__device__ __forceinline__ uint32_t rank_cell(const VoxShared& S, uint32_t low, uint32_t r) {
  return low | (((r >= S.qbase[1] ? 1u : 0u) + (r >= S.qbase[2] ? 1u : 0u) + (r >= S.qbase[3] ? 1u : 0u)) << 16);
}

enum SumLayout { kLeaf16, kNarrow, kWide };

// Extraction: rank lo + i goes to staging record at + i (cell order; `at`
// beyond stage_cap: the reservation reported it), and the entry is left empty
// for the next pass or item (the next item's layout may put an accumulator
// where a cell is kept now).
template <SumLayout LAYOUT>
__device__ __forceinline__ void extract_sums(int4* stage_out, ulonglong2* sums_out, uint64_t stage_cap, uint64_t at,
                                          uint32_t lo, uint32_t span) {
  VoxShared& S = vox_shared();
  uint32_t* const F = vox_fields();
  uint16_t* const K = LAYOUT == kLeaf16 ? vox_cells<2, kCapLeaf>() : (LAYOUT == kNarrow ? vox_cells<4, kCapNarrow>() : vox_cells<7, kCapWide>());
  const uint32_t n_wraps = LAYOUT == kLeaf16 ? min(S.n_wraps, kMaxWraps) : 0u;
  for (uint32_t i = threadIdx.x; i < span; i += kVoxThreads) {
    const uint32_t cell = rank_cell(S, K[i], lo + i);
    K[i] = 0;
    uint64_t sr, sg, sb, n;
    if (LAYOUT == kLeaf16) {
      const uint32_t w0 = F[i], w1 = F[kCapLeaf + i];
      F[i] = 0u;
      F[kCapLeaf + i] = 0u;
      uint32_t cr = 0, cg = 0, cb = 0;
      for (uint32_t e = 0; e != n_wraps; ++e) {
        const uint32_t w = vox_wraps()[e];
        if ((w & 0xFFFFu) == i) {
          cr += (w >> 16) & 1u;
          cg += (w >> 17) & 1u;
          cb += (w >> 18) & 1u;
        }
      }
      // a wrap of a word's lower field has carried into its upper one
      sr = (w0 & 0xFFFFu) + (cr << 16);
      sg = (w0 >> 16) + (cg << 16) - cr;
      sb = (w1 & 0xFFFFu) + (cb << 16);
      n = ((w1 >> 16) - cb) & 0xFFFFu;
    } else if (LAYOUT == kNarrow) {
      sr = F[i];
      sg = F[kCapNarrow + i];
      sb = F[2u * kCapNarrow + i];
      n = F[3u * kCapNarrow + i];
#pragma unroll
      for (uint32_t f = 0; f < 4u; ++f) F[f * kCapNarrow + i] = 0u;
    } else {
      sr = F[i] | ((uint64_t)F[kCapWide + i] << 32);
      sg = F[2u * kCapWide + i] | ((uint64_t)F[3u * kCapWide + i] << 32);
      sb = F[4u * kCapWide + i] | ((uint64_t)F[5u * kCapWide + i] << 32);
      n = F[6u * kCapWide + i];
#pragma unroll
      for (uint32_t f = 0; f < 7u; ++f) F[f * kCapWide + i] = 0u;
    }
    const uint32_t m = mean_rgba(sr, sg, sb, n);
    const bool packed = n < kPackMaxCount;  // the sums travel in the record itself
    if (at + i < stage_cap) {
      stage_out[at + i] = make_int4((int)parent_cell(cell, S.I), (int)m, (int)n,
                                    packed ? (int)pack_remainders(sr, sg, sb, n, m) : (int)kNone);
      if (!packed) sums_out[at + i] = make_ulonglong2(sr | (sg << 40), (sg >> 24) | (sb << 16));
    }
  }
}

// Extraction of the weighted mode.
__device__ __forceinline__ void extract_weighted(int4* stage_out, uint64_t stage_cap, uint64_t at, uint32_t lo, uint32_t span) {
  VoxShared& S = vox_shared();
  uint32_t* const F = vox_fields();
  uint16_t* const K = vox_cells<9, kCapWeighted>();
  for (uint32_t i = threadIdx.x; i < span; i += kVoxThreads) {
    const uint32_t cell = rank_cell(S, K[i], lo + i), n = F[8u * kCapWeighted + i];
    unsigned long long s[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) s[f] = F[2u * f * kCapWeighted + i] | ((unsigned long long)F[(2u * f + 1u) * kCapWeighted + i] << 32);
#pragma unroll
    for (uint32_t f = 0; f < 9u; ++f) F[f * kCapWeighted + i] = 0u;
    const uint32_t rgba = w_round(s[0], s[3]) | (w_round(s[1], s[3]) << 8) | (w_round(s[2], s[3]) << 16) | 0xFF000000u;
    if (at + i < stage_cap) stage_out[at + i] = make_int4((int)parent_cell(cell, S.I), (int)rgba, (int)n, (int)kNone);
  }
}

// Extraction of the single-sample modes.
template <int MODE>
__device__ __forceinline__ void extract_pick(const PickArgs& P) {
  VoxShared& S = vox_shared();
  uint16_t* const K = vox_cells<5, kCapPick>();
  for (uint32_t i = threadIdx.x; i < P.span; i += kVoxThreads) {
    const unsigned long long e = pick_keys()[i];
    const uint2 pay = pick_pays()[i];
    const uint32_t best = (uint32_t)e, n = pick_counts()[i], cell = rank_cell(S, K[i], P.lo + i);
    pick_keys()[i] = ~0ull;
    pick_counts()[i] = 0u;
    if (pay.x != best) S.settle = 1u;
    else if (best >= P.idx_bound || pick_high<MODE>(best, P.level) != (uint32_t)(e >> 32))
      atomicOr(P.error, kErrInternal);  // cannot happen for a cell that received a sample
    if (P.out_at + i < P.stage_cap)
      P.stage_out[P.out_at + i] = make_int4((int)parent_cell(cell, S.I), (int)pay.y, (int)n, (int)best);
  }
}

}  // namespace

namespace {

// The item's header, read by warp 0 in two dependent steps: lane 0 reads the
// child node; then lane 8 reads the parent node while lanes 0..7 read the
// children's records (inner items), all at once.
__device__ __forceinline__ void vox_header(const BuildArgs& a, const VoxLevel& v, uint32_t it) {
  VoxShared& S = vox_shared();
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  if (tid < 32) {
    if (lane == 0) {
      const uint32_t t = find_tile(v.item_prefix, a.n_tiles, it);
      const uint32_t* ls = v.lvl_start + (uint64_t)t * (kMaxLevels + 1);
      const TileDesc& td = a.tiles[t];
      const uint64_t g = td.node_base + ls[v.level + 1] + (it - v.item_prefix[t]);
      const lod_node_t c = v.nodes[g];
      S.I.tile = t;
      S.I.g = g;
      S.cmin[0] = c.min[0];
      S.cmin[1] = c.min[1];
      S.cmin[2] = c.min[2];
      S.I.leaf = (c.flags & LOD_NODE_LEAF) != 0;
      S.I.n = S.I.leaf ? c.point_count : c.voxel_count;
      S.I.npts = c.point_count;
      S.nbase = td.node_base;
      S.cparent = td.node_base + c.parent;
      S.cfirst = td.node_base + c.first_child;
      S.pbase = td.pt_base + c.point_offset;
      S.nch = S.I.leaf ? 0u : (uint32_t)__popc(c.child_mask);
      S.pick_level = td.level0 + v.level;
      S.idx_bound = td.idx_bound;
    }
    __syncwarp();
    const uint32_t nch = S.nch;
    if (S.I.leaf) {
      // the leaf's points (32-byte records where indices are kept), in
      // 64 KB pieces, one per lane
      const bool wsrc = a.wide != nullptr;
      const char* base = wsrc ? (const char*)(a.wide + 2 * S.pbase) : (const char*)(a.out + S.pbase);
      const uint64_t bytes = umin64(S.I.n * (wsrc ? 32u : 16u), kPrefetchBytes);
      const uint64_t off = (uint64_t)lane << 16;
      if (off < bytes) prefetch_l2(base + off, (uint32_t)umin64(bytes - off, 1u << 16));
    }
    if (lane == 8) {
      const lod_node_t p = v.nodes[S.cparent];
      S.I.Lp = p.log2_size;
      S.pmask = p.child_mask;
      S.pfirst = S.nbase + p.first_child;
      S.I.pmin[0] = p.min[0];
      S.I.pmin[1] = p.min[1];
      S.I.pmin[2] = p.min[2];
      S.I.kx = S.cmin[0] != p.min[0];
      S.I.ky = S.cmin[1] != p.min[1];
      S.I.kz = S.cmin[2] != p.min[2];
    }
    // the children's staged records, one flat sample sequence
    uint32_t occ = 0;
    if (lane < nch) {
      const NodeAux ca = v.aux[S.cfirst + lane];
      S.cstage[lane] = ca.stage;
      S.cdense[lane] = ca.dense;
      occ = ca.occ;
      if (occ) prefetch_l2(v.stage_in + ca.stage, (uint32_t)umin64((uint64_t)occ * 16u, 1u << 16));
    }
    if (lane < 8) {
      uint32_t incl = occ;  // prefix over lanes 0..7
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFu, incl, o);
        if ((int)lane >= o) incl += y;
      }
      if (lane == 0) S.cpre[0] = 0;
      S.cpre[lane + 1] = incl;
    }
  }
}

// Ranks the occupied cells: an exclusive scan of the words' counts.  Every
// warp ranks 32 kScan consecutive groups of four words by coalesced 16-byte
// loads: lane l holds groups l, l + 32, ...  Returns their number.
__device__ __forceinline__ uint32_t vox_rank_cells() {
  VoxShared& S = vox_shared();
  const uint4* const bits4 = reinterpret_cast<const uint4*>(vox_smem);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t D;
  {
    uint32_t pre[kScan], tot = 0;
#pragma unroll
    for (int m = 0; m < kScan; ++m) {
      const uint4 e = bits4[warp * (32u * kScan) + lane + 32u * (uint32_t)m];
      const uint32_t c = __popc(e.x) + __popc(e.y) + __popc(e.z) + __popc(e.w);
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += y;
      }
      pre[m] = tot + incl - c;
      tot += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (lane == 0) S.wsum[warp] = tot;
    __syncthreads();
    // every warp adds up the warps before it
    const uint32_t ws = lane < kVoxWarps ? S.wsum[lane] : 0u;
    uint32_t wi = ws;
#pragma unroll
    for (int o = 1; o < kVoxWarps; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if ((int)lane >= o) wi += y;
    }
    const uint32_t excl = wi - ws;
    D = __shfl_sync(0xFFFFFFFFu, wi, kVoxWarps - 1);
    uint32_t base = __shfl_sync(0xFFFFFFFFu, excl, warp);
    const uint32_t quarter = __shfl_sync(0xFFFFFFFFu, excl, warp & ~(kVoxWarps / 4u - 1u));
    if (D > 0xFFFFu) base -= quarter;  // word ranks relative to their quarter
    if (warp == 0 && lane < kVoxWarps && lane % (kVoxWarps / 4u) == 0) S.qbase[lane / (kVoxWarps / 4u)] = excl;
#pragma unroll
    for (int m = 0; m < kScan; ++m) {
      const uint32_t at = warp * (32u * kScan) + lane + 32u * (uint32_t)m;
      const uint4 e = bits4[at];
      const uint32_t r0 = base + pre[m], r1 = r0 + __popc(e.x), r2 = r1 + __popc(e.y), r3 = r2 + __popc(e.z);
      reinterpret_cast<uint2*>(vox_wrank())[at] = make_uint2(r0 | (r1 << 16), r2 | (r3 << 16));
    }
  }
  return D;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Pass 2 over the ranks [S.r0, S.r1), C of them at a time: accumulate, then
// extract.  (A leaf read from 32-byte staging records was published by the
// mark pass: these passes read the 16- or 20-byte copy.)  The item's first
// staging record: thread 0 brings it in `stg`, or (CLUSTER) S.stage holds it
// once the cluster barrier that every thread has arrived at is complete; the
// first extraction, or the end if there is none, waits for that.
template <int MODE, bool CLUSTER>
__device__ __forceinline__ void vox_ranges(const BuildArgs& a, const VoxLevel& v, DevCounters* __restrict__ ctr, SumLayout lay,
                                           uint32_t C, unsigned long long stg) {
  VoxShared& S = vox_shared();
  constexpr bool WEIGHTED = MODE == LOD_WEIGHTED, PICKLIKE = MODE != LOD_FILTER && !WEIGHTED;
  const uint32_t tid = threadIdx.x;
  const bool leaf = S.I.leaf;
  const uint32_t total = leaf ? (uint32_t)S.I.n : S.cpre[S.nch];
  bool waited = !CLUSTER;
  for (uint32_t lo = S.r0, r1 = S.r1; lo < r1; lo += C) {
    const uint32_t span = r1 - lo < C ? r1 - lo : C;
    const int4* const src = leaf ? a.out + S.pbase : v.stage_in;
    const uint32_t* const pidx = PICKLIKE ? a.out_idx + S.pbase : nullptr;
    PickArgs P;
    if (PICKLIKE) {
      P.lo = lo;
      P.span = span;
      P.level = S.pick_level;
      P.idx_bound = S.idx_bound;
      P.stage_out = v.stage_out;
      P.stage_cap = v.stage_cap;
      P.error = &ctr->error;
      P.out_at = 0;
      if (!leaf) pick_inner<MODE>(P, src, total);
      else pick_leaf<MODE>(P, src, pidx, total);
    } else if (WEIGHTED) {
      acc_weighted(src, v.border_list, leaf, total, lo, span);
    } else if (leaf) {
      if (lay == kLeaf16) acc_leaf16(src, total, lo, span);
      else if (lay == kNarrow) acc_leaf_sums<false>(src, total, lo, span);
      else acc_leaf_sums<true>(src, total, lo, span);
    } else {
      if (lay == kNarrow) acc_inner_sums<false>(src, v.stage_in_sum, total, lo, span);
      else acc_inner_sums<true>(src, v.stage_in_sum, total, lo, span);
    }
    if (!CLUSTER && tid == 0) S.stage = stg;
    if (!waited) cluster_wait();
    waited = true;
    __syncthreads();  // every update of the pass is done
    const unsigned long long at = S.stage + lo;
    if (PICKLIKE) {
      P.out_at = at;
      extract_pick<MODE>(P);
      __syncthreads();
      if (S.settle) settle_pick<MODE>(P, src, pidx, leaf, total);
    } else if (WEIGHTED) {
      extract_weighted(v.stage_out, v.stage_cap, at, lo, span);
    } else if (lay == kLeaf16) {
      extract_sums<kLeaf16>(v.stage_out, v.stage_out_sum, v.stage_cap, at, lo, span);
    } else if (lay == kNarrow) {
      extract_sums<kNarrow>(v.stage_out, v.stage_out_sum, v.stage_cap, at, lo, span);
    } else {
      extract_sums<kWide>(v.stage_out, v.stage_out_sum, v.stage_cap, at, lo, span);
    }
    __syncthreads();
    if (MODE == LOD_FILTER && lay == kLeaf16 && r1 - lo > C) {  // more passes follow: they list their own wraps
      if (tid == 0) S.n_wraps = 0;
      __syncthreads();
    }
  }
  if (!waited) cluster_wait();
}

// Passes over the item's samples, the mark pass included (statistics).
__device__ __forceinline__ uint32_t vox_passes(uint32_t C) {
  const VoxShared& S = vox_shared();
  return 1u + (S.r1 - S.r0 + C - 1u) / C;
}

}  // namespace

// Voxelize one item (a child node c of an inner node p at level v.level):
// all of its ranks, or, for a queued unit (r_unit, p_unit), the ranks
// [D r / P, D (r + 1) / P) of its D occupied cells.  `first`: the item's
// first attempt, which reserves the item's staging block (D records) and,
// when its cells need several accumulate passes, may queue the ranges after
// the first for k_vox_units.  The CTA that holds range 0 also
// publishes what it reads (the leaf's points, the children's voxels).
// `next_item` (first attempts): where thread 0 leaves the item the CTA
// takes next, fetched while this one is marked.
template <int MODE>
__device__ __forceinline__ void vox_item(const BuildArgs& a, const VoxLevel& v, DevCounters* __restrict__ ctr, uint32_t it,
                                         uint32_t r_unit, uint32_t p_unit, bool first, uint32_t* next_item) {
  VoxShared& S = vox_shared();
  uint4* const bits4 = reinterpret_cast<uint4*>(vox_smem);
  const uint32_t tid = threadIdx.x;
  vox_header(a, v, it);
#pragma unroll
  for (uint32_t i = 0; i < kWords / 4u / kVoxThreads; ++i) bits4[tid + i * kVoxThreads] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  constexpr bool WEIGHTED = MODE == LOD_WEIGHTED, PICKLIKE = MODE != LOD_FILTER && !WEIGHTED;  // one sample kept per cell
  const bool leaf = S.I.leaf;
  const bool lead = r_unit == 0;  // the one CTA of the item that publishes
  const uint32_t total = leaf ? (uint32_t)S.I.n : S.cpre[S.nch];  // samples
  // the next item's counter value; its latency hides behind the mark pass
  uint32_t next_k = 0;
  if (next_item && tid == 0) next_k = atomicAdd(&ctr->item_head, 1u);

  if (WEIGHTED && tid < (uint32_t)__popc(S.pmask)) S.border[tid] = v.border[S.pfirst + tid];

  // ---- pass 1: mark the occupied cells
  if (!leaf) mark_inner<MODE == LOD_FILTER>(v.stage_in, 0u, total, lead ? v.dense : nullptr, v.dense_cap);
  else if (a.wide) mark_wide(a.wide + 2 * S.pbase, total, lead ? a.out + S.pbase : nullptr, lead ? a.out_idx + S.pbase : nullptr);
  else mark_leaf(a.out + S.pbase, total);
  __syncthreads();

  uint32_t next_it = next_k;
  if (next_item && tid == 0 && v.order && next_k < v.n_items) next_it = v.order[next_k];
  const uint32_t D = vox_rank_cells();
  // the narrowest sums that provably cannot overflow for the points of this cube
  const SumLayout lay = leaf && S.I.npts <= kLeafMaxSamples ? kLeaf16 : (S.I.npts <= kNarrowMaxSamples ? kNarrow : kWide);
  const uint32_t cap = PICKLIKE ? kCapPick : WEIGHTED ? kCapWeighted : (lay == kLeaf16 ? kCapLeaf : (lay == kNarrow ? kCapNarrow : kCapWide));
  const uint32_t C = (v.range_cells && v.range_cells < cap) ? v.range_cells : cap;  // ranks per pass
  // thread 0: the item's first staging record.  The reservation (or, for
  // a unit, the read of the first attempt's) is issued here and its value
  // first used before the first extraction, so its latency overlaps the
  // accumulate pass.
  unsigned long long stg = 0;
  if (tid == 0) {
    S.D = D;
    if (first) {
      stg = atomicAdd(v.stage_used, (unsigned long long)D);
      v.aux[S.I.g].occ = D;
      S.r0 = 0;
      S.r1 = D;
      const uint32_t P = (D + C - 1) / C;
      if (P > 1) atomicAdd(&ctr->vox_retries, 1ull);
      uint32_t q0 = 0;
      if (P > 1 && v.units && P >= v.queue_ranges && reserve_units(&ctr->units, v.unit_cap, P - 1, &q0)) {
        for (uint32_t r = 1; r < P; ++r) v.units[q0 + r - 1] = make_uint4(it, r, P, 0u);
        S.r1 = D / P;
      }
    } else {
      stg = v.aux[S.I.g].stage;  // reserved by the first attempt
      S.r0 = (uint32_t)((uint64_t)D * r_unit / p_unit);
      S.r1 = (uint32_t)((uint64_t)D * (r_unit + 1) / p_unit);
    }
    S.n_wraps = 0;
    S.settle = 0;
  }
  __syncthreads();

  vox_ranges<MODE, false>(a, v, ctr, lay, C, stg);
  if (tid == 0) {
    if (first) {
      v.aux[S.I.g].stage = stg;
      if (stg + D > v.stage_cap) atomicOr(&ctr->error, kErrStageCap);
    }
    if (next_item) *next_item = next_it;  // read after this item's last barrier
    const uint32_t passes = vox_passes(C);
    atomicAdd(&ctr->vox_passes, (unsigned long long)passes);
    atomicAdd(&ctr->vox_samples, (unsigned long long)passes * total);
    if (first) atomicMax(&ctr->vox_max_item, (unsigned long long)S.I.n);
  }
  __syncthreads();
}

// First attempt of every item, taken by persistent CTAs in the level's item
// order.  While an item is marked, its CTA already takes the next one.
template <int MODE>
__global__ void __launch_bounds__(kVoxThreads, kVoxCtasPerSm)
    k_vox(const __grid_constant__ BuildArgs a, const __grid_constant__ VoxLevel v, DevCounters* __restrict__ ctr) {
  VoxShared& S = vox_shared();
  vox_clear_dense<MODE>();
  if (threadIdx.x == 0) {
    const uint32_t k = atomicAdd(&ctr->item_head, 1u);
    S.next = (v.order && k < v.n_items) ? v.order[k] : k;
  }
  __syncthreads();
  for (;;) {
    const uint32_t it = S.next;  // every thread reads it before the item's first barrier
    if (it >= v.n_items) break;
    vox_item<MODE>(a, v, ctr, it, 0u, 1u, true, &S.next);
  }
}

// Rank ranges of items with many occupied cells, taken from the queue by
// persistent CTAs (the queue is complete when this starts).
template <int MODE>
__global__ void __launch_bounds__(kVoxThreads, kVoxCtasPerSm)
    k_vox_units(const __grid_constant__ BuildArgs a, const __grid_constant__ VoxLevel v, DevCounters* __restrict__ ctr) {
  VoxShared& S = vox_shared();
  const uint32_t n_units = min(ctr->units, v.unit_cap);
  if (blockIdx.x >= n_units) return;
  vox_clear_dense<MODE>();
  for (;;) {
    if (threadIdx.x == 0) S.next = atomicAdd(&ctr->unit_head, 1u);
    __syncthreads();
    const uint32_t u = S.next;
    __syncthreads();
    if (u >= n_units) break;
    const uint4 w = v.units[u];
    vox_item<MODE>(a, v, ctr, w.x, w.y, w.z, false, nullptr);
  }
}

namespace {

// Shared-memory address of byte `off` of vox_smem in CTA `cta` of the cluster.
__device__ __forceinline__ uint32_t far_addr(uint32_t off, uint32_t cta) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(vox_smem) + off), "r"(cta));
  return a;
}
__device__ __forceinline__ uint4 far_ld4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}

}  // namespace

// Levels with few items (the top of the tree, the deepest levels): a cluster
// of 2^lp CTAs takes an item.  Every CTA marks (and publishes) a share of the
// samples in a bitmap of its own; each merges a slice of all the bitmaps and
// collects the other slices, through distributed shared memory; then every
// CTA ranks the merged bitmap and takes a part of the ranks, reading all of
// the samples.
//
// Bound by the length of that chain for the largest item.  Measured against
// units that each marked the whole item before they took a part of its ranks
// (a launch to split the items and one for the units), and one CTA per item
// above a quarter of the SMs: 1M points (56 and 8 items) 83 -> 57 us, 10M indoor
// points first come (ten levels) 787 -> 602 us, 20M indoor points random (twelve)
// 1160 -> 991 us, the root's 8 items of 500M points 172 -> 101 us.  (Adding each
// CTA's share of the samples to the entries of the whole cluster by remote
// atomics instead is slower for most levels: 56 items of 1M points 36 -> 113 us,
// 8 items of 500M 172 -> 84.)
template <int MODE>
__global__ void __launch_bounds__(kVoxThreads, 1)
    k_vox_cluster(const __grid_constant__ BuildArgs a, const __grid_constant__ VoxLevel v, DevCounters* __restrict__ ctr, uint32_t lp) {
  VoxShared& S = vox_shared();
  constexpr bool WEIGHTED = MODE == LOD_WEIGHTED, PICKLIKE = MODE != LOD_FILTER && !WEIGHTED;
  const uint32_t tid = threadIdx.x, parts = 1u << lp, part = blockIdx.x & (parts - 1u), k = blockIdx.x >> lp;
  const uint32_t it = v.order ? v.order[k] : k;  // largest items first
  uint4* const bits4 = reinterpret_cast<uint4*>(vox_smem);
  vox_header(a, v, it);
#pragma unroll
  for (uint32_t i = 0; i < kWords / 4u / kVoxThreads; ++i) bits4[tid + i * kVoxThreads] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  const bool leaf = S.I.leaf;
  const uint32_t total = leaf ? (uint32_t)S.I.n : S.cpre[S.nch];
  const uint32_t first = (uint32_t)(((uint64_t)total * part) >> lp), end = (uint32_t)(((uint64_t)total * (part + 1u)) >> lp);
  if (WEIGHTED && tid < (uint32_t)__popc(S.pmask)) S.border[tid] = v.border[S.pfirst + tid];

  // ---- mark and publish the CTA's share
  if (!leaf) mark_inner<MODE == LOD_FILTER>(v.stage_in, first, end, v.dense, v.dense_cap);
  else if (a.wide) mark_wide(a.wide + 2 * (S.pbase + first), end - first, a.out + S.pbase + first, a.out_idx + S.pbase + first);
  else mark_leaf(a.out + S.pbase + first, end - first);
  cluster_arrive();
  vox_clear_dense<MODE>();
  cluster_wait();
  // ---- merge: slice `part` of every CTA's bitmap into the own one ...
  const uint32_t slice = (kWords / 4u) >> lp;  // in groups of four words
  for (uint32_t i = tid; i < slice; i += kVoxThreads) {
    const uint32_t at = part * slice + i;
    uint4 w = bits4[at];
    for (uint32_t q = 1; q < parts; ++q) {
      const uint4 x = far_ld4(far_addr(16u * at, (part + q) & (parts - 1u)));
      w.x |= x.x, w.y |= x.y, w.z |= x.z, w.w |= x.w;
    }
    bits4[at] = w;
  }
  cluster_arrive();
  cluster_wait();
  // ---- ... then the other slices from the CTAs that merged them (which
  // leave those alone from here on)
  for (uint32_t i = tid; i < kWords / 4u; i += kVoxThreads) {
    const uint32_t from = i / slice;
    if (from != part) bits4[i] = far_ld4(far_addr(16u * i, from));
  }
  __syncthreads();
  const uint32_t D = vox_rank_cells();
  const SumLayout lay = leaf && S.I.npts <= kLeafMaxSamples ? kLeaf16 : (S.I.npts <= kNarrowMaxSamples ? kNarrow : kWide);
  const uint32_t cap = PICKLIKE ? kCapPick : WEIGHTED ? kCapWeighted : (lay == kLeaf16 ? kCapLeaf : (lay == kNarrow ? kCapNarrow : kCapWide));
  const uint32_t C = (v.range_cells && v.range_cells < cap) ? v.range_cells : cap;  // ranks per pass
  if (tid == 0) {
    S.D = D;
    S.r0 = (uint32_t)(((uint64_t)D * part) >> lp);
    S.r1 = (uint32_t)(((uint64_t)D * (part + 1u)) >> lp);
    S.n_wraps = 0;
    S.settle = 0;
    if (part == 0) {
      // the item's staging block, told to the other CTAs
      const unsigned long long stg = atomicAdd(v.stage_used, (unsigned long long)D);
      v.aux[S.I.g].occ = D;
      v.aux[S.I.g].stage = stg;
      if (stg + D > v.stage_cap) atomicOr(&ctr->error, kErrStageCap);
      if (D > C << lp) atomicAdd(&ctr->vox_retries, 1ull);
      for (uint32_t q = 0; q < parts; ++q)
        asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(far_addr(kSharedOff + (uint32_t)offsetof(VoxShared, stage), q)), "l"(stg)
                     : "memory");
    }
  }
  // waited for before the first extraction: by then every CTA has collected
  // its slices (so any of them may leave) and knows the staging block
  cluster_arrive();
  __syncthreads();
  vox_ranges<MODE, true>(a, v, ctr, lay, C, 0ull);
  if (tid == 0) {
    const uint32_t passes = vox_passes(C);
    atomicAdd(&ctr->vox_passes, (unsigned long long)passes);
    atomicAdd(&ctr->vox_samples, (unsigned long long)(passes - 1u) * total + (end - first));
    if (part == 0) atomicMax(&ctr->vox_max_item, (unsigned long long)S.I.n);
  }
}

template <int MODE>
static void vox_attrs() {
  cudaFuncSetAttribute(k_vox<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  cudaFuncSetAttribute(k_vox_units<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  cudaFuncSetAttribute(k_vox_cluster<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

// One-time kernel attributes of the voxel pass (called before any launch,
// and before a stream capture of the voxel levels); returns the SM count.
int vox_init() {
  static int sms = [] {
    vox_attrs<LOD_FILTER>();
    vox_attrs<LOD_PICK>();
    vox_attrs<LOD_FIRST>();
    vox_attrs<LOD_RANDOM>();
    vox_attrs<LOD_WEIGHTED>();
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
  }();
  return sms;
}

// A level's items are shared by clusters of 2^share_log2 CTAs: levels of few
// items, by as many CTAs as the SMs hold at once (another wave of clusters
// costs more than it shortens: 56 items in clusters of 8 took 3 times as long as
// one CTA each).
static constexpr uint32_t share_log2(uint32_t n_items, uint32_t ctas) {
  return n_items <= ctas / 8u ? 3u : n_items <= ctas / 4u ? 2u : n_items <= ctas / 2u ? 1u : 0u;
}
static_assert(share_log2(19, 152) == 3 && share_log2(20, 152) == 2 && share_log2(38, 152) == 2 &&
              share_log2(39, 152) == 1 && share_log2(76, 152) == 1 && share_log2(77, 152) == 0, "one wave of clusters");
static_assert(share_log2(1u << 29, 152) == 0 && share_log2(1u << 30, 152) == 0 && share_log2(1u << 31, 152) == 0,
              "no wrap at levels of 2^29 items and more");

template <int MODE>
static cudaError_t launch_vox_mode(const BuildArgs& a, const VoxLevel& v, DevCounters* ctr, cudaStream_t st) {
  const uint32_t ctas = (uint32_t)(vox_init() * kVoxCtasPerSm);
  const uint32_t lp = share_log2(v.n_items, ctas);
  if (lp) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1u << lp;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(v.n_items << lp);
    cfg.blockDim = dim3(kVoxThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_vox_cluster<MODE>, a, v, ctr, lp);
    note_launch();
    return e;
  }
  k_vox<MODE><<<v.n_items < ctas ? v.n_items : ctas, kVoxThreads, kSmemBytes, st>>>(a, v, ctr);
  note_launch();
  if (v.units) k_vox_units<MODE><<<ctas, kVoxThreads, kSmemBytes, st>>>(a, v, ctr);
  if (v.units) note_launch();
  return cudaGetLastError();
}

cudaError_t launch_vox(const BuildArgs& a, const VoxLevel& v, DevCounters* ctr, cudaStream_t st) {
  if (!v.n_items) return cudaSuccess;
  switch (a.mode) {
    case LOD_PICK: return launch_vox_mode<LOD_PICK>(a, v, ctr, st);
    case LOD_FIRST: return launch_vox_mode<LOD_FIRST>(a, v, ctr, st);
    case LOD_RANDOM: return launch_vox_mode<LOD_RANDOM>(a, v, ctr, st);
    case LOD_WEIGHTED: return launch_vox_mode<LOD_WEIGHTED>(a, v, ctr, st);
    default: return launch_vox_mode<LOD_FILTER>(a, v, ctr, st);
  }
}

// Assign every item its place in the level's contiguous voxel block
// (exclusive scan of the occupied counts in node order), then give every
// parent the range of its children's items.
__global__ void __launch_bounds__(kBlock) k_level_scan(BuildArgs a, VoxLevel v, const uint32_t* __restrict__ parent_prefix,
                                                       uint32_t n_parents,
                                                       unsigned long long* __restrict__ tile_voxels,
                                                       DevCounters* __restrict__ ctr) {
  __shared__ unsigned long long warp_sum[32];
  __shared__ unsigned long long s_carry;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // this level's voxels follow those of the levels below in the voxel array
  const uint64_t level_base = v.vstate[0];
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  for (uint32_t chunk = 0; chunk < v.n_items; chunk += blockDim.x) {
    const uint32_t it = chunk + threadIdx.x;
    uint64_t g = 0;
    unsigned long long x = 0;
    if (it < v.n_items) {
      const uint32_t t = find_tile(v.item_prefix, a.n_tiles, it);
      g = a.tiles[t].node_base + v.lvl_start[(uint64_t)t * (kMaxLevels + 1) + v.level + 1] + (it - v.item_prefix[t]);
      x = v.aux[g].occ;
    }
    unsigned long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if ((int)lane >= o) incl += y;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t nw = blockDim.x >> 5;
      unsigned long long w = lane < nw ? warp_sum[lane] : 0ull;
      unsigned long long wi = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
        if ((int)lane >= o) wi += y;
      }
      if (lane < nw) warp_sum[lane] = wi - w;
    }
    __syncthreads();
    const unsigned long long excl = s_carry + warp_sum[warp] + incl - x;
    if (it < v.n_items) v.aux[g].dense = level_base + excl;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_carry = excl + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ctr->level_voxels = s_carry;
    if (level_base + s_carry > v.dense_cap) v.vstate[1] = 1ull;
  }
  __syncthreads();
  for (uint32_t ip = threadIdx.x; ip < n_parents; ip += blockDim.x) {
    const uint32_t t = find_tile(parent_prefix, a.n_tiles, ip);
    const TileDesc& td = a.tiles[t];
    const uint64_t pg = td.node_base + v.lvl_start[(uint64_t)t * (kMaxLevels + 1) + v.level] + (ip - parent_prefix[t]);
    lod_node_t& p = v.nodes[pg];
    if (p.flags & LOD_NODE_LEAF) continue;
    const uint64_t f = td.node_base + p.first_child;
    const uint64_t l = f + __popc(p.child_mask) - 1;
    const uint64_t off = v.aux[f].dense;
    const uint64_t cnt = v.aux[l].dense + v.aux[l].occ - off;
    p.voxel_offset = off;
    p.voxel_count = (uint32_t)cnt;
    atomicAdd(&tile_voxels[t], (unsigned long long)cnt);
  }
  __syncthreads();  // every thread has read vstate[0]
  if (threadIdx.x == 0) v.vstate[0] = level_base + s_carry;
  if (!v.next_order) return;
  // The order in which the next level up takes its items (the nodes of this
  // level): classes of equal bit length of the sample count, largest first,
  // so that the big items start early and every SM ends the level on small
  // ones.  Order within a class is immaterial (results do not depend on it).
  __shared__ uint32_t cls[33];
  if (threadIdx.x < 33) cls[threadIdx.x] = 0;
  __syncthreads();
  auto samples_class = [&](uint32_t ip) -> uint32_t {
    const uint32_t t = find_tile(parent_prefix, a.n_tiles, ip);
    const TileDesc& td = a.tiles[t];
    const lod_node_t& p = v.nodes[td.node_base + v.lvl_start[(uint64_t)t * (kMaxLevels + 1) + v.level] +
                                  (ip - parent_prefix[t])];
    const uint32_t n = (p.flags & LOD_NODE_LEAF) ? p.point_count : p.voxel_count;
    return 32u - (uint32_t)__clz(n);  // 0 for n = 0
  };
  for (uint32_t ip = threadIdx.x; ip < n_parents; ip += blockDim.x) atomicAdd(&cls[samples_class(ip)], 1u);
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int c = 32; c >= 0; --c) {
      const uint32_t k = cls[c];
      cls[c] = run;
      run += k;
    }
  }
  __syncthreads();
  for (uint32_t ip = threadIdx.x; ip < n_parents; ip += blockDim.x)
    v.next_order[atomicAdd(&cls[samples_class(ip)], 1u)] = ip;
}

cudaError_t launch_level_scan(const BuildArgs& a, const VoxLevel& v, const uint32_t* parent_prefix,
                              uint32_t n_parents, unsigned long long* tile_voxels, DevCounters* ctr,
                              cudaStream_t st) {
  k_level_scan<<<1, kBlock, 0, st>>>(a, v, parent_prefix, n_parents, tile_voxels, ctr);
  note_launch();
  return cudaGetLastError();
}

// Publish the staged voxels of the items of the topmost processed level
// (their parents, the roots, have no parent pass that would copy them).
// blockIdx.y takes a share of the item: a copy of 16-byte records, bound by
// memory latency when a single CTA makes it (8 items of 500M points: 47 ->
// 8 us with 32 shares each).
__global__ void __launch_bounds__(256) k_copy_items(BuildArgs a, VoxLevel v) {
  const uint32_t it = blockIdx.x;
  const uint32_t t = find_tile(v.item_prefix, a.n_tiles, it);
  const uint64_t g = a.tiles[t].node_base + v.lvl_start[(uint64_t)t * (kMaxLevels + 1) + v.level + 1] +
                     (it - v.item_prefix[t]);
  const NodeAux ca = v.aux[g];
  if (ca.dense + ca.occ > v.dense_cap) return;  // the build is redone with a larger array
  const bool filt = a.mode == LOD_FILTER;  // records may carry their sums packed, which are not published
  for (uint32_t i = blockIdx.y * blockDim.x + threadIdx.x; i < ca.occ; i += gridDim.y * blockDim.x) {
    int4 rec = v.stage_out[ca.stage + i];
    if (filt) rec.w = (int)kNone;
    v.dense[ca.dense + i] = rec;
  }
}

cudaError_t launch_copy_items(const BuildArgs& a, const VoxLevel& v, cudaStream_t st) {
  if (!v.n_items) return cudaSuccess;
  k_copy_items<<<dim3(v.n_items, v.n_items <= 64 ? 32u : 4u), 256, 0, st>>>(a, v);
  note_launch();
  return cudaGetLastError();
}

// The exact sums of those voxels, of which the staged records or the sums array
// behind them hold one each (out-of-core batches only, after the levels).
__global__ void __launch_bounds__(256) k_root_sums(BuildArgs a, VoxLevel v) {
  const uint32_t it = blockIdx.x;
  const uint32_t t = find_tile(v.item_prefix, a.n_tiles, it);
  const NodeAux ca = v.aux[a.tiles[t].node_base + v.lvl_start[(uint64_t)t * (kMaxLevels + 1) + v.level + 1] +
                           (it - v.item_prefix[t])];
  for (uint32_t i = threadIdx.x; i < ca.occ; i += blockDim.x) {
    const int4 rec = v.stage_out[ca.stage + i];
    v.root_sums[ca.dense - v.root_base + i] =
        (uint32_t)rec.w != kNone ? unpack_sums(rec) : v.stage_out_sum[ca.stage + i];
  }
}

cudaError_t launch_root_sums(const BuildArgs& a, const VoxLevel& v, cudaStream_t st) {
  if (!v.n_items) return cudaSuccess;
  k_root_sums<<<v.n_items, 256, 0, st>>>(a, v);
  note_launch();
  return cudaGetLastError();
}

// Publish the leaf points and indices of tiles whose root is a leaf (no
// voxel pass reads those points): blockIdx.y selects the tile.
__global__ void __launch_bounds__(256) k_unwide(BuildArgs a, const uint32_t* __restrict__ tiles) {
  const TileDesc& td = a.tiles[tiles[blockIdx.y]];
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < td.n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t p = td.pt_base + i;
    int4 q;
    uint32_t x;
    ld_wide(a.wide + 2 * p, q, x);
    a.out[p] = q;
    a.out_idx[p] = x;
  }
}

cudaError_t launch_unwide(const BuildArgs& a, const uint32_t* tiles, uint32_t n_tiles, uint32_t max_points,
                          cudaStream_t st) {
  if (!n_tiles) return cudaSuccess;
  const uint32_t gx = (uint32_t)umin64(((uint64_t)max_points + 255) / 256, 1024);
  for (uint32_t t0 = 0; t0 < n_tiles; t0 += 65535) {
    const uint32_t m = n_tiles - t0 < 65535 ? n_tiles - t0 : 65535;
    k_unwide<<<dim3(gx ? gx : 1, m), 256, 0, st>>>(a, tiles + t0);
    note_launch();
  }
  return cudaGetLastError();
}

// Full-precision variant (Section 7): the input point each voxel of a
// single-sample mode picked, gathered from the caller's input into an
// array parallel to the voxel array.
//
// One tile: its voxels are the whole array, taken flat, four random 16-byte
// reads of a thread in flight (bound by their latency and the 32-byte sectors
// around them).  Measured on 4.1M voxels of a 20M-point build against one CTA
// of 256 threads per node: 870 -> 41 us.
__global__ void __launch_bounds__(256) k_voxel_points(const TileDesc* __restrict__ tiles, uint64_t n_voxels,
                                                      const int4* __restrict__ dense, int4* __restrict__ out) {
  const TileDesc& td = tiles[0];
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n_voxels; i0 += 4u * step) {
    uint32_t pick[4];
    int4 p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) pick[k] = i0 + k * step < n_voxels ? (uint32_t)__ldg(&dense[i0 + k * step].w) : kNone;
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = pick[k] < td.n ? __ldg(td.in + pick[k]) : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i0 + k * step < n_voxels) out[i0 + k * step] = p[k];
  }
}

// Several tiles: the levels of all tiles alternate in the voxel array, so a
// voxel's tile follows from its node.  blockIdx.y selects the tile.
__global__ void __launch_bounds__(256) k_tile_voxel_points(const TileDesc* __restrict__ tiles,
                                                           const lod_node_t* __restrict__ nodes,
                                                           const uint32_t* __restrict__ n_nodes,
                                                           const int4* __restrict__ dense, int4* __restrict__ out) {
  const TileDesc& td = tiles[blockIdx.y];
  const uint32_t nn = n_nodes[blockIdx.y];
  for (uint32_t i = blockIdx.x; i < nn; i += gridDim.x) {
    const lod_node_t& nd = nodes[td.node_base + i];
    for (uint32_t j = threadIdx.x; j < nd.voxel_count; j += blockDim.x) {
      const uint32_t pick = (uint32_t)dense[nd.voxel_offset + j].w;
      out[nd.voxel_offset + j] = pick < td.n ? td.in[pick] : make_int4(0, 0, 0, 0);
    }
  }
}

cudaError_t launch_voxel_points(const TileDesc* tiles, uint32_t n_tiles, const lod_node_t* nodes,
                                const uint32_t* n_nodes, uint32_t max_nodes, uint64_t n_voxels, const int4* dense,
                                int4* out, cudaStream_t st) {
  if (!n_tiles || !max_nodes || !n_voxels) return cudaSuccess;
  if (n_tiles == 1) {
    const uint32_t gx = (uint32_t)umin64((n_voxels + 1023) / 1024, 8u * (uint32_t)vox_init());
    k_voxel_points<<<gx, 256, 0, st>>>(tiles, n_voxels, dense, out);
    note_launch();
    return cudaGetLastError();
  }
  const uint32_t gx = max_nodes < 4096 ? max_nodes : 4096;
  for (uint32_t t0 = 0; t0 < n_tiles; t0 += 65535) {
    const uint32_t m = n_tiles - t0 < 65535 ? n_tiles - t0 : 65535;
    k_tile_voxel_points<<<dim3(gx, m), 256, 0, st>>>(tiles + t0, nodes, n_nodes + t0, dense, out);
    note_launch();
  }
  return cudaGetLastError();
}

// Gather each node's voxels to a new offset (compact per-result copies).
__global__ void __launch_bounds__(256) k_gather_voxels(const lod_node_t* __restrict__ nodes,
                                                       const uint64_t* __restrict__ new_off,
                                                       const int4* __restrict__ src, int4* __restrict__ dst) {
  const lod_node_t nd = nodes[blockIdx.x];
  const int4* s = src + nd.voxel_offset;
  int4* d = dst + new_off[blockIdx.x];
  for (uint32_t i = threadIdx.x; i < nd.voxel_count; i += blockDim.x) d[i] = s[i];
}

cudaError_t launch_gather_voxels(const lod_node_t* nodes, uint32_t n_nodes, const uint64_t* new_off,
                                 const int4* src, int4* dst, cudaStream_t st) {
  if (!n_nodes) return cudaSuccess;
  k_gather_voxels<<<n_nodes, 256, 0, st>>>(nodes, new_off, src, dst);
  note_launch();
  return cudaGetLastError();
}

}  // namespace lodk
