// Rendering of an LOD octree (Section 5 of the paper) into a headless
// framebuffer, as CUDA kernels instead of draw calls.
//
// Node selection: a node is drawn when it lies at least partly inside the
// view frustum and every ancestor is refined; a node is refined when it is
// drawn and its projected bounding box is larger than a pixel threshold
// (about 100 pixels in the paper, matching the 128^3 voxel grid).  The
// paper's layered structure replaces, not adds: a drawn inner node skips
// its voxels that lie in an octant whose child is drawn (the child draws
// finer samples there), and a drawn leaf draws all its points.
//
// Every drawn sample is projected with a row-major 4x4 matrix applied to
// its position relative to an integer origin (so that large int32
// coordinates keep their precision), and a pixel keeps the sample of
// smallest (depth, colour) through a 64-bit atomicMin on
// (float bits of depth) << 32 | rgba, depth = z/w * 1/2 + 1/2 in [0, 1]
// (non-negative floats order like their bits).
// All arithmetic is single precision with every operation rounded on its
// own (explicit _rn intrinsics, no fused multiply-add), so each pixel
// decision is reproducible bit for bit.
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace lodk {

namespace {

struct RClip {
  float x, y, z, w;
};

__device__ __forceinline__ RClip r_project(const lod_camera_t& c, float px, float py, float pz) {
  float r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float s = __fmul_rn(c.view_proj[4 * i + 0], px);
    s = __fadd_rn(s, __fmul_rn(c.view_proj[4 * i + 1], py));
    s = __fadd_rn(s, __fmul_rn(c.view_proj[4 * i + 2], pz));
    s = __fadd_rn(s, c.view_proj[4 * i + 3]);
    r[i] = s;
  }
  return {r[0], r[1], r[2], r[3]};
}

__device__ __forceinline__ float r_rel(int32_t v, int32_t o) { return __ll2float_rn((long long)v - (long long)o); }

// Frustum test and projected size (pixels) of the cube [min, min + 2^L)^3;
// a cube reaching behind the camera has infinite size.
__device__ void r_box(const lod_camera_t& c, const lod_node_t& nd, bool* inside, float* size) {
  const float edge = __int_as_float((int)(127u + nd.log2_size) << 23);  // 2^L, L <= 32
  float lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = r_rel(nd.min[a], c.origin[a]);
    hi[a] = __fadd_rn(lo[a], edge);
  }
  bool all[6] = {true, true, true, true, true, true};
  bool behind = false;
  float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const RClip q = r_project(c, (k & 4) ? hi[0] : lo[0], (k & 2) ? hi[1] : lo[1], (k & 1) ? hi[2] : lo[2]);
    all[0] = all[0] && (q.x < -q.w);
    all[1] = all[1] && (q.x > q.w);
    all[2] = all[2] && (q.y < -q.w);
    all[3] = all[3] && (q.y > q.w);
    all[4] = all[4] && (q.z < -q.w);
    all[5] = all[5] && (q.z > q.w);
    if (!(q.w > 0.0f)) {
      behind = true;
      continue;
    }
    const float sx = __fmul_rn(__fadd_rn(__fmul_rn(__fdiv_rn(q.x, q.w), 0.5f), 0.5f), (float)c.width);
    const float sy = __fmul_rn(__fadd_rn(__fmul_rn(__fdiv_rn(q.y, q.w), 0.5f), 0.5f), (float)c.height);
    if (k == 0 || sx < x0) x0 = sx;
    if (k == 0 || sx > x1) x1 = sx;
    if (k == 0 || sy < y0) y0 = sy;
    if (k == 0 || sy > y1) y1 = sy;
  }
  *inside = !(all[0] || all[1] || all[2] || all[3] || all[4] || all[5]);
  const float w = __fsub_rn(x1, x0), h = __fsub_rn(y1, y0);
  *size = behind ? INFINITY : (w > h ? w : h);
}

// Draws one sample; true if it reached a pixel.
__device__ __forceinline__ bool r_splat(const lod_camera_t& c, float px, float py, float pz, uint32_t rgba,
                                        unsigned long long* fb) {
  const RClip q = r_project(c, px, py, pz);
  // outside the clip volume: with w > 0 a quotient x / w, rounded to nearest,
  // lies above 1 exactly when x > w (x is then at least w's next float, and
  // ulp(w) / w > 2^-24), so most samples off the screen need no division
  if (!(q.w > 0.0f)) return false;
  if (q.x < -q.w || q.x > q.w || q.y < -q.w || q.y > q.w || q.z < -q.w || q.z > q.w) return false;
  const float nx = __fdiv_rn(q.x, q.w), ny = __fdiv_rn(q.y, q.w), nz = __fdiv_rn(q.z, q.w);
  uint32_t ix = (uint32_t)floorf(__fmul_rn(__fadd_rn(__fmul_rn(nx, 0.5f), 0.5f), (float)c.width));
  uint32_t iy = (uint32_t)floorf(__fmul_rn(__fadd_rn(__fmul_rn(ny, 0.5f), 0.5f), (float)c.height));
  ix = ix < c.width ? ix : c.width - 1;
  iy = iy < c.height ? iy : c.height - 1;
  const float depth = __fadd_rn(__fmul_rn(nz, 0.5f), 0.5f);
  const unsigned long long key = ((unsigned long long)__float_as_uint(depth) << 32) | rgba;
  // a pixel's key only ever falls, so whatever (possibly old) key is read
  // here, a sample that is not below it cannot win: most samples of a pixel
  // (tens on an overview) cost a cached read instead of an atomic
  unsigned long long* const at = fb + (uint64_t)iy * c.width + ix;
  if (key < *at) atomicMin(at, key);
  return true;
}

}  // namespace

// Samples of one entry of the draw list.
constexpr uint32_t kDrawChunk = 2048;

// One thread per node: drawn iff the node and every ancestor are in the
// frustum and every ancestor projects larger than the threshold.  A drawn
// node's samples go to the draw list in pieces, so that the drawing kernel's
// CTAs get equal work whatever the nodes' sizes.
__global__ void k_render_select(const lod_node_t* __restrict__ nodes, uint32_t n_nodes, lod_camera_t c,
                                uint8_t* __restrict__ visible, unsigned int* __restrict__ n_visible,
                                uint2* __restrict__ list, unsigned int* __restrict__ n_list) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  bool inside;
  float size;
  r_box(c, nodes[i], &inside, &size);
  bool vis = inside;
  for (uint32_t p = nodes[i].parent, depth = 0; vis && p != kNone && depth < 64; p = nodes[p].parent, ++depth) {
    r_box(c, nodes[p], &inside, &size);
    vis = inside && size > c.lod_pixels;
  }
  visible[i] = vis ? 1 : 0;
  if (!vis) return;
  atomicAdd(n_visible, 1u);
  const uint64_t n = (nodes[i].flags & LOD_NODE_LEAF) ? nodes[i].point_count : nodes[i].voxel_count;
  const uint32_t pieces = (uint32_t)((n + kDrawChunk - 1) / kDrawChunk);
  const uint32_t at = atomicAdd(n_list, pieces);
  for (uint32_t j = 0; j < pieces; ++j) list[at + j] = make_uint2(i, j);
}

// Persistent CTAs walk the draw list: leaves splat their points, inner nodes
// their voxels outside the octants of drawn children.  Bound by the random
// 8-byte reads of the framebuffer and by issue (a projection and three
// correctly rounded divisions a sample).  Measured on a full-HD overview of
// 50M indoor points (10-29M samples drawn), against one CTA per node at a
// time, an atomicMin for every sample and an atomic count: 0.75 -> 0.126 ms a frame.
__global__ void __launch_bounds__(256) k_render_draw(const lod_node_t* __restrict__ nodes, const int4* __restrict__ points,
                                                     const int4* __restrict__ voxels, lod_camera_t c,
                                                     const uint8_t* __restrict__ visible, const uint2* __restrict__ list,
                                                     const unsigned int* __restrict__ n_list,
                                                     unsigned long long* __restrict__ fb,
                                                     unsigned long long* __restrict__ drawn) {
  const uint32_t n = *n_list;
  uint32_t count = 0;
  for (uint32_t w = blockIdx.x; w < n; w += gridDim.x) {
    const uint2 job = list[w];
    const lod_node_t& nd = nodes[job.x];
    const uint64_t first = (uint64_t)job.y * kDrawChunk;
    const bool leaf = (nd.flags & LOD_NODE_LEAF) != 0;
    const uint64_t total = leaf ? nd.point_count : nd.voxel_count;
    const uint32_t m = (uint32_t)(total - first < kDrawChunk ? total - first : kDrawChunk);
    const int4* src = leaf ? points + nd.point_offset + first : voxels + nd.voxel_offset + first;
    uint32_t child_drawn = 0;  // bit k: the child in octant k is drawn and replaces the node's voxels there
    float lo[3] = {0.0f, 0.0f, 0.0f}, scale = 0.0f;
    if (!leaf) {
      for (uint32_t k = 0, ch = nd.first_child; k < 8; ++k)
        if (nd.child_mask & (1u << k)) child_drawn |= (uint32_t)visible[ch++] << k;
#pragma unroll
      for (int a = 0; a < 3; ++a) lo[a] = r_rel(nd.min[a], c.origin[a]);
      // cell centre (2 q + 1) 2^(L - 8): an exact power-of-two scaling
      scale = __int_as_float((int)(127 + (int)nd.log2_size - 8) << 23);
    }
    for (uint32_t j0 = threadIdx.x; j0 < m; j0 += 4u * 256u) {
      int4 q[4];  // four loads in flight
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j0 + 256u * u < m) q[u] = __ldcs(src + j0 + 256u * u);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (j0 + 256u * u >= m) break;
        float p[3];
        uint32_t rgba;
        if (leaf) {
          p[0] = r_rel(q[u].x, c.origin[0]);
          p[1] = r_rel(q[u].y, c.origin[1]);
          p[2] = r_rel(q[u].z, c.origin[2]);
          rgba = (uint32_t)q[u].w;
        } else {
          const uint32_t cell = (uint32_t)q[u].x;
          const uint32_t g[3] = {cell & 127u, (cell >> 7) & 127u, cell >> 14};
          if (child_drawn & (1u << (((g[0] >> 6) << 2) | ((g[1] >> 6) << 1) | (g[2] >> 6)))) continue;
#pragma unroll
          for (int a = 0; a < 3; ++a) p[a] = __fadd_rn(lo[a], __fmul_rn((float)(2u * g[a] + 1u), scale));
          rgba = (uint32_t)q[u].y;
        }
        count += r_splat(c, p[0], p[1], p[2], rgba, fb) ? 1u : 0u;
      }
    }
  }
  if (!drawn) return;
  count = __reduce_add_sync(0xFFFFFFFFu, count);
  if ((threadIdx.x & 31u) == 0 && count) atomicAdd(drawn, (unsigned long long)count);
}

uint64_t render_list_entries(uint32_t n_nodes, uint64_t n_points, uint64_t n_voxels) {
  return n_nodes + (n_points + n_voxels) / kDrawChunk;
}

cudaError_t launch_render(const lod_node_t* nodes, uint32_t n_nodes, const int4* points, const int4* voxels,
                          const lod_camera_t& cam, uint8_t* visible, unsigned int* n_visible, uint2* list,
                          unsigned int* n_list, unsigned long long* fb, unsigned long long* drawn, int sms, cudaStream_t st) {
  if (!n_nodes) return cudaSuccess;
  k_render_select<<<(n_nodes + 127) / 128, 128, 0, st>>>(nodes, n_nodes, cam, visible, n_visible, list, n_list);
  note_launch();
  k_render_draw<<<8 * sms, 256, 0, st>>>(nodes, points, voxels, cam, visible, list, n_list, fb, drawn);
  note_launch();
  return cudaGetLastError();
}

}  // namespace lodk
