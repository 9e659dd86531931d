// Neighbourhood-weighted average voxel sampling (Section 4.2.4 of the paper):
// the samples that reach across a parent's octants.
//
// An inner node's samples are its children's samples: the points of leaf
// children, and the voxels of inner children, each taken as one sample at
// the centre of its cell with its stored 8-bit colour.  A sample adds
// weight w = max(0, 1 - distance to the cell centre, in cells) times its
// colour to each cell of the 2x2x2 block around it (the cells whose centres
// are within one cell width along every axis), and marks the cell it lies
// in as occupied; only occupied cells become voxels, coloured by their
// weighted sum over their weight sum, rounded half up, alpha 255.  Counts
// are the cell's original points, as in the other modes.
//
// The unit of work is a (parent, child octant) item, as in the other modes
// (k_voxel.cu): the octant's occupied cells are those of the child's own
// samples, so their sums fit the item's shared-memory entries.  What the
// other octants add are the few samples whose block crosses a middle plane of
// the parent's grid (its second cell along an axis is cell 64).  This kernel
// lists them, one list per item, before the level's items run, and an item
// reads the lists of its up to seven siblings.
//
// It reads the level's samples once (and again, from L2, where a CTA found
// some to list).  Measured: 20M aerial points, all levels of one build, this
// and the voxel kernels against one dense 128^3 grid per CTA in global memory
// with 64-bit global atomics (one CTA per parent): 5.85 -> 1.44 ms.
#include "common.cuh"
#include "kernels.h"
#include "wgrid.cuh"

namespace lodk {

namespace {

constexpr int kBorderThreads = 512;

__device__ __forceinline__ bool crosses(const WBlock& b) { return b.j1[0] == 64 || b.j1[1] == 64 || b.j1[2] == 64; }

}  // namespace

// One CTA per item.  border[g] of the item's node g receives {first entry (64
// bits), entries, 1 for points and 0 for voxels}; an entry is the point
// itself, or a voxel's {cell | octant << 21, rgba, 0, 0}.
__global__ void __launch_bounds__(kBorderThreads) k_wborder(BuildArgs a, VoxLevel v, DevCounters* __restrict__ ctr) {
  __shared__ uint32_t wsum[kBorderThreads / 32];
  __shared__ unsigned long long s_base;
  const uint32_t it = blockIdx.x, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t lo = 0, hi = a.n_tiles;  // the item's tile: the largest t with item_prefix[t] <= it
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (v.item_prefix[mid] <= it) lo = mid;
    else hi = mid;
  }
  const TileDesc& td = a.tiles[lo];
  const uint64_t g = td.node_base + v.lvl_start[(uint64_t)lo * (kMaxLevels + 1) + v.level + 1] + (it - v.item_prefix[lo]);
  const lod_node_t c = v.nodes[g];
  const lod_node_t P = v.nodes[td.node_base + c.parent];
  const bool leaf = (c.flags & LOD_NODE_LEAF) != 0;
  const uint32_t k = (c.min[0] != P.min[0] ? 4u : 0u) | (c.min[1] != P.min[1] ? 2u : 0u) | (c.min[2] != P.min[2] ? 1u : 0u);
  const uint64_t pbase = td.pt_base + c.point_offset;
  const uint32_t wide = a.wide ? 2u : 1u;  // with kept indices the points still lie in the 32-byte records
  const int4* const pts = a.wide ? a.wide + 2 * pbase : a.out + pbase;
  const uint32_t nch = leaf ? 1u : (uint32_t)__popc(c.child_mask);
  uint32_t count = 0;
  uint64_t at = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (uint32_t r = 0; r < nch; ++r) {
      const NodeAux* ca = leaf ? nullptr : &v.aux[td.node_base + c.first_child + r];
      const int4* src = leaf ? pts : v.stage_in + ca->stage;
      const uint64_t n = leaf ? c.point_count : ca->occ;
      const uint32_t step = leaf ? wide : 1u;
      for (uint64_t i0 = threadIdx.x; i0 < n; i0 += 4u * kBorderThreads) {
        int4 q[4];  // four loads in flight
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t i = i0 + j * kBorderThreads;
          if (i < n) q[j] = __ldcg(src + step * i);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (i0 + j * kBorderThreads >= n) continue;
          const WBlock b = leaf ? w_point_block(q[j], P.min, P.log2_size) : w_voxel_block((uint32_t)q[j].x, k);
          if (!crosses(b)) continue;
          if (pass == 0) ++count;
          else if (at < v.border_cap) v.border_list[at++] = leaf ? q[j] : make_int4(q[j].x | (int)(k << 21), q[j].y, 0, 0);
        }
      }
    }
    if (pass == 1) break;
    // each thread's place in the item's list
    uint32_t incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if ((int)lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (uint32_t w = 0; w < kBorderThreads / 32; ++w) {
      if (w < warp) before += wsum[w];
      total += wsum[w];
    }
    if (threadIdx.x == 0) {
      s_base = total ? atomicAdd(&ctr->border_used, (unsigned long long)total) : 0ull;
      if (s_base + total > v.border_cap) atomicOr(&ctr->error, kErrStageCap);
      v.border[g] = make_uint4((uint32_t)s_base, (uint32_t)(s_base >> 32), total, leaf ? 1u : 0u);
    }
    __syncthreads();
    if (!total) return;
    at = s_base + before + incl - count;
  }
}

cudaError_t launch_wborder(const BuildArgs& a, const VoxLevel& v, DevCounters* ctr, cudaStream_t st) {
  if (!v.n_items) return cudaSuccess;
  k_wborder<<<v.n_items, kBorderThreads, 0, st>>>(a, v, ctr);
  note_launch();
  return cudaGetLastError();
}

}  // namespace lodk
