// Active-primitive compaction and linear BVH build.
//
// Compaction ("hair data reorganisation", Section 6 "Real-time performance"):
// a cluster at the strand level contributes every segment of its member
// strands, a cluster at level L contributes every segment of its level-L
// thick hairs.  Per-cluster counts are scanned and each cluster's block writes
// its global primitive ids.
//
// LBVH (Karras 2012, "Maximizing parallelism in the construction of BVHs,
// octrees, and k-d trees"): 21-bit Morton codes (7 bits per axis) of the
// primitive box centroids in the strand boxes' bounds, stable single-sweep
// radix sort of (code, position in the active list), one thread per internal
// node finds its key range and split from the longest common prefix (ties
// between equal codes broken by index).  Bounds go bottom-up in two kernels:
// k_gather_refit gathers the leaf boxes in Morton order and finishes the nodes
// whose leaf range lies inside its thread block's leaves (nearly all of them)
// in barrier-separated rounds in shared memory; k_climb finishes the few nodes
// that span blocks by atomic minima of the planes from each climb start, and
// k_span_records packs those nodes.
//
// Node layouts, children's boxes stored in the parent; a child index >= 0 is
// an internal node, < 0 is primitive ~index:
//  * On a grid (2 x uint4 = 32 bytes, one sector): per child the x, y and z
//    intervals and the child index.  An interval is lo | hi << 16 on the BVH's
//    grid (Bvh::frame: 65,520 steps over the bounds of every strand and
//    thick-hair box), rounded outward and widened by one step more, which
//    covers the half step that the traversal's decoding can be off.  FP32
//    boxes take two sectors: a far larger part of the traversal's loads missed
//    L1 (the 4K frame of 500k strands: 25% of the sectors).
//  * In FP32 (4 x float4 = 64 bytes), for scenes that the grid does not
//    resolve (scene_grid): (lo0.x, hi0.x, lo0.y, hi0.y), (lo1.x, hi1.x, lo1.y,
//    hi1.y), (lo0.z, hi0.z, lo1.z, hi1.z), (child0, child1, -, -).
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace hr {
namespace {

// Active primitives per cluster, and the thick-hair total in counts[C + 1]
// (zeroed by the caller) for the statistics.
__global__ void k_cluster_counts(const uint8_t* __restrict__ lod, const uint32_t* __restrict__ cl_first,
                                 uint32_t C, uint32_t L, uint32_t S, uint32_t* counts) {
  const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const uint32_t l = min((uint32_t)lod[c], L);
  const uint32_t m = cl_first[c + 1] - cl_first[c];
  // a cluster of m < 4^l strands has m non-empty level-l thick hairs
  const uint32_t eths = min(1u << (2 * l), m);
  counts[c] = (l == L) ? m * S : eths * S;
  if (l < L) atomicAdd(counts + C + 1, eths * S);
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

constexpr size_t kFrameWords = 7;

// What a build or refit takes from the scene as a whole (Bvh::frame), and the
// leaves' bounds and the climb's counts cleared for k_gather_refit:
//  * The grid of the node boxes, from the bounds of the strands' and the thick
//    hairs' boxes: low corner (two steps below the bounds; its fourth word says
//    whether the nodes are in FP32), step, 1 / step.
//  * The centroid codes' low corner and 1 / extent.
// The whole block calls it, R boxes of strand segments a thread (count in all).
// The grid resolves a scene whose boxes are many steps long; one far vertex or
// parts of very different scale make it so coarse that neighbouring boxes
// become the same, and so does the codes' cell.  So where more than one of these
// segments in kCoarsePart is not kFineSteps steps long in any axis, or the bounds
// are not finite, the nodes are in FP32, and the codes spread over the bulk of the
// segments instead of the bounds: from the 25th least minimum of the lanes' 32
// groups to their 25th greatest maximum (three groups in four may hold far ones)
// and half as much on each side.
// BVH and image, us a frame of 100k strands, one vertex put ever farther away,
// on the grid / in FP32 by the steps of the median segment: a close view at 202
// steps 3,692 / 3,821, at 113 3,844 / 3,820, at 60 4,080 / 3,814, at 16 5,577 /
// 3,812, at 1 136,091 / 3,817; a far view at 113 1,535 / 1,629, at 60 1,628 /
// 1,626, at 16 1,709 / 1,631, at 1 4,979 / 1,623.
constexpr float kFineSteps = 64.f;
constexpr uint32_t kCoarsePart = 8;
template <int R>
__device__ __forceinline__ void scene_grid(const uint32_t* __restrict__ bounds, const float4 (&l)[R],
                                           const float4 (&h)[R], bool has, uint32_t count,
                                           float4* frame, unsigned* counts) {
  __shared__ uint32_t s_coarse, s_lo[3][32], s_hi[3][32];
  const uint32_t lane = threadIdx.x & 31;
  if (threadIdx.x == 0) s_coarse = 0u;
  __syncthreads();
  float lo[3], hi[3], st[3], clo[3], cinv[3];
  for (int i = 0; i < 3; ++i) {
    lo[i] = clo[i] = from_ordered(bounds[i]);
    hi[i] = from_ordered(bounds[3 + i]);
    cinv[i] = hi[i] > lo[i] ? 1.f / (hi[i] - lo[i]) : 0.f;
    const uint32_t el = bounds[kEthBounds + i], eh = bounds[kEthBounds + 3 + i];
    if (el <= eh) {  // there are thick hairs
      lo[i] = fminf(lo[i], from_ordered(el));
      hi[i] = fmaxf(hi[i], from_ordered(eh));
    }
    st[i] = fmaxf((hi[i] - lo[i]) * (1.0f / 65520.0f), 1e-30f);
    lo[i] = fmaf(-2.0f, st[i], lo[i]);
  }
  uint32_t coarse = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool fine = h[r].x - l[r].x >= kFineSteps * st[0] || h[r].y - l[r].y >= kFineSteps * st[1] ||
                      h[r].z - l[r].z >= kFineSteps * st[2];
    coarse += __popc(__ballot_sync(0xffffffffu, has && !fine));
  }
  if (lane == 0 && coarse) atomicAdd(&s_coarse, coarse);
  __syncthreads();
  const bool finite = fabsf(lo[0] + lo[1] + lo[2]) + st[0] + st[1] + st[2] < __int_as_float(0x7f800000);
  const bool wide = s_coarse * kCoarsePart > count || !finite;
  if (wide) {
    if (threadIdx.x < 32)
      for (int i = 0; i < 3; ++i) s_lo[i][lane] = 0xffffffffu, s_hi[i][lane] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float c[3] = {0.5f * (l[r].x + h[r].x), 0.5f * (l[r].y + h[r].y), 0.5f * (l[r].z + h[r].z)};
      for (int i = 0; has && i < 3; ++i) {
        atomicMin(&s_lo[i][lane], low_bits(c[i]));
        atomicMax(&s_hi[i][lane], high_bits(c[i]));
      }
    }
    __syncthreads();
    const uint32_t groups = min(32u, count), rank = groups * 3 / 4;
    for (int i = 0; i < 3; ++i) {
      uint32_t a = 0, b = 0;
      for (uint32_t g = 0; g < groups; ++g) {
        uint32_t ra = 0, rb = 0;
        for (uint32_t q = 0; q < groups; ++q) {
          ra += s_lo[i][q] < s_lo[i][g] || (s_lo[i][q] == s_lo[i][g] && q < g);
          rb += s_hi[i][q] > s_hi[i][g] || (s_hi[i][q] == s_hi[i][g] && q < g);
        }
        if (ra == rank) a = g;
        if (rb == rank) b = g;
      }
      const float l0 = from_ordered(s_lo[i][a]), h0 = from_ordered(s_hi[i][b]), e = h0 - l0;
      const bool some = e > 0.f && e < 1e38f;
      clo[i] = some ? fmaf(-0.5f, e, l0) : 0.f;
      cinv[i] = some ? 0.5f / e : 0.f;
    }
  }
  if (threadIdx.x) return;
  frame[0] = make_float4(lo[0], lo[1], lo[2], wide ? 1.f : 0.f);
  frame[1] = make_float4(st[0], st[1], st[2], 0.f);
  frame[2] = make_float4(1.0f / st[0], 1.0f / st[1], 1.0f / st[2], 0.f);
  uint32_t* leaf_bounds = reinterpret_cast<uint32_t*>(frame + 3);
  for (int i = 0; i < 6; ++i) leaf_bounds[i] = i < 3 ? 0xffffffffu : 0u;
  frame[5] = make_float4(clo[0], clo[1], clo[2], 0.f);
  frame[6] = make_float4(cinv[0], cinv[1], cinv[2], 0.f);
  if (counts) counts[0] = counts[1] = 0u;
}

// The same from 1,024 of the n strand segments, spread evenly and not in step
// with the strands, by a block of 256.
constexpr uint32_t kGridBlock = 256;
__device__ __forceinline__ void sample_grid(const uint32_t* __restrict__ bounds,
                                            const float4* __restrict__ box, uint32_t n, float4* frame,
                                            unsigned* counts) {
  float4 l[4], h[4];
#pragma unroll
  for (uint32_t r = 0; r < 4; ++r) {
    const size_t at = __umulhi((r * kGridBlock + threadIdx.x) * 2654435769u, n);  // golden-ratio steps
    l[r] = box[2 * at], h[r] = box[2 * at + 1];
  }
  scene_grid<4>(bounds, l, h, true, 1024, frame, counts);
}

__global__ void __launch_bounds__(kGridBlock)
    k_scene_grid(const uint32_t* __restrict__ bounds, const float4* __restrict__ box, uint32_t n,
                 float4* frame, unsigned* counts) {
  sample_grid(bounds, box, n, frame, counts);
}

__global__ void __launch_bounds__(256, 8) k_cluster_fill(const uint8_t* __restrict__ lod, const uint32_t* __restrict__ cl_first,
                               const uint32_t* __restrict__ order, const uint32_t* __restrict__ offs,
                               const uint32_t* __restrict__ eth_off, uint32_t C, uint32_t L,
                               uint32_t N, uint32_t S, uint32_t* ids,
                               const uint32_t* __restrict__ bounds, const float4* __restrict__ box,
                               float4* frame, unsigned* counts) {
  if (blockIdx.x == 0) {
    sample_grid(bounds, box, N * S, frame, counts);
    return;
  }
  const uint32_t c = blockIdx.x - 1;
  const uint32_t l = min((uint32_t)lod[c], L);
  const uint32_t base = offs[c];
  if (l == L) {
    const uint32_t r0 = cl_first[c], m = cl_first[c + 1] - r0;
    for (uint32_t j = threadIdx.x; j < m * S; j += blockDim.x) {
      const uint32_t s = order[r0 + j / S];
      ids[base + j] = s * S + j % S;
    }
  } else {
    const uint32_t sub = 1u << (2 * l);
    const uint32_t e0 = eth_off[l] + c * sub;
    const uint32_t m = cl_first[c + 1] - cl_first[c];
    if (m >= sub) {
      for (uint32_t j = threadIdx.x; j < sub * S; j += blockDim.x)
        ids[base + j] = N * S + (e0 + j / S) * S + j % S;
    } else {
      // fewer strands than buckets: member i alone fills bucket floor(i 4^l / m)
      for (uint32_t j = threadIdx.x; j < m * S; j += blockDim.x) {
        const uint32_t b = (uint32_t)(((uint64_t)(j / S) * sub) / m);
        ids[base + j] = N * S + (e0 + b) * S + j % S;
      }
    }
  }
}

__global__ void __launch_bounds__(256, 8) k_iota(uint32_t* ids, uint32_t n, const uint32_t* __restrict__ bounds,
                       const float4* __restrict__ box, float4* frame, unsigned* counts) {
  if (blockIdx.x == 0) {
    sample_grid(bounds, box, n, frame, counts);
    return;
  }
  const uint32_t i = (blockIdx.x - 1) * blockDim.x + threadIdx.x;
  if (i < n) ids[i] = i;
}

// Primitive centroid codes keep the top 7 bits of each axis (21 bits, three
// radix passes).  Primitives in one cell keep the order of the active list
// (clusters in root Morton order, each strand's segments in order along the
// strand), and Karras' index tie-break splits them by that order.  At the
// full-head workload this took the BVH build plus frame from 1.51 to 1.42 ms
// against 10 bits per axis; 8 bits gave 1.47, 6 bits 1.48 and 5 bits 1.91
// (the cells then hold too many primitives).
constexpr int kMortonBits = 21;

__device__ __forceinline__ uint32_t prim_code(const float4 l, const float4 h, const float4* frame) {
  const float4 lo = frame[5], inv_ext = frame[6];
  const float cx = (0.5f * (l.x + h.x) - lo.x) * inv_ext.x;
  const float cy = (0.5f * (l.y + h.y) - lo.y) * inv_ext.y;
  const float cz = (0.5f * (l.z + h.z) - lo.z) * inv_ext.z;
  const uint32_t qx = (uint32_t)min(1023.f, fmaxf(0.f, cx * 1024.f));
  const uint32_t qy = (uint32_t)min(1023.f, fmaxf(0.f, cy * 1024.f));
  const uint32_t qz = (uint32_t)min(1023.f, fmaxf(0.f, cz * 1024.f));
  return ((spread10(qx) << 2) | (spread10(qy) << 1) | spread10(qz)) >> (30 - kMortonBits);
}

__global__ void k_prim_morton(const float4* __restrict__ box, const uint32_t* __restrict__ ids,
                              uint32_t n, const float4* __restrict__ frame, uint32_t* keys) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint32_t id = ids[i];
  keys[i] = prim_code(box[2 * (size_t)id], box[2 * (size_t)id + 1], frame);
}
// Length of the common prefix of (key, index) at i and j; -1 outside [0, n).
__device__ __forceinline__ int delta(const uint32_t* __restrict__ keys, int n, uint32_t ki, int i,
                                     int j) {
  if ((unsigned)j >= (unsigned)n) return -1;
  const uint32_t x = ki ^ keys[j];
  return x ? __clz(x) : 32 + __clz((uint32_t)i ^ (uint32_t)j);
}

// Children and leaf range of internal node i; also writes their parent links.
__device__ __forceinline__ int4 karras_node(const uint32_t* __restrict__ keys, int n, int i,
                                            int* parent_int, int* parent_leaf) {
  const uint32_t ki = keys[i];
  const int d = (delta(keys, n, ki, i, i + 1) - delta(keys, n, ki, i, i - 1)) >= 0 ? 1 : -1;
  const int dmin = delta(keys, n, ki, i, i - d);
  int lmax = 2;
  while (delta(keys, n, ki, i, i + lmax * d) > dmin) lmax <<= 1;
  int l = 0;
  for (int t = lmax >> 1; t >= 1; t >>= 1)
    if (delta(keys, n, ki, i, i + (l + t) * d) > dmin) l += t;
  const int j = i + l * d;
  const int dnode = delta(keys, n, ki, i, j);
  int s = 0;
  for (int k = 1;; ++k) {  // t = ceil(l / 2^k)
    const int t = (l + (1 << k) - 1) >> k;
    if (delta(keys, n, ki, i, i + (s + t) * d) > dnode) s += t;
    if (t == 1) break;
  }
  const int gamma = i + s * d + min(d, 0);
  const int lo = min(i, j), hi = max(i, j);
  int c0, c1;
  if (lo == gamma) {
    c0 = ~gamma;
    parent_leaf[gamma] = 2 * i;
  } else {
    c0 = gamma;
    parent_int[gamma] = 2 * i;
  }
  if (hi == gamma + 1) {
    c1 = ~(gamma + 1);
    parent_leaf[gamma + 1] = 2 * i + 1;
  } else {
    c1 = gamma + 1;
    parent_int[gamma + 1] = 2 * i + 1;
  }
  return make_int4(c0, c1, lo, hi);
}

__global__ void k_karras(const uint32_t* __restrict__ keys, int n, int4* child,
                         int* parent_int, int* parent_leaf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n - 1) child[i] = karras_node(keys, n, i, parent_int, parent_leaf);
}

// The global primitive id of every leaf (Morton order).
__global__ void k_gather(const uint32_t* __restrict__ sorted_ids, uint32_t n, uint32_t* leaf_id) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) leaf_id[i] = sorted_ids[i];
}

// Boxes of the two node layouts.  Both have: the box of a leaf, the union,
// the six words whose minima are the union's (k_climb), a node's two children's
// boxes out of its record, and the record.
//
// On the grid: per axis lo | (65535 - hi) << 16, so that the union of two
// boxes is the smaller of each half.
struct QBox {
  uint32_t x, y, z;
};
constexpr uint32_t kFlipHi = 0xffff0000u;  // 65535 - hi <-> hi
__device__ __forceinline__ uint32_t q_axis(float l, float h, float lo, float inv_step) {
  if (!(l <= h)) return 0xffffffffu;  // not a number (its record is never hit): empty, adds nothing
  const float a = floorf((l - lo) * inv_step) - 1.f, b = ceilf((h - lo) * inv_step) + 1.f;
  const uint32_t qa = (uint32_t)fminf(fmaxf(a, 0.f), 65535.f);
  const uint32_t qb = (uint32_t)fminf(fmaxf(b, 0.f), 65535.f);
  return qa | ((65535u - qb) << 16);
}
__device__ __forceinline__ void leaf_box(QBox& b, const float4 l, const float4 h, const float4* grid) {
  const float4 lo = grid[0], is = grid[2];
  b = QBox{q_axis(l.x, h.x, lo.x, is.x), q_axis(l.y, h.y, lo.y, is.y), q_axis(l.z, h.z, lo.z, is.z)};
}
__device__ __forceinline__ QBox box_union(const QBox a, const QBox b) {
  return QBox{__vminu2(a.x, b.x), __vminu2(a.y, b.y), __vminu2(a.z, b.z)};
}
__device__ __forceinline__ void box_words(const QBox b, uint32_t w[6]) {
  w[0] = b.x & 0xffffu, w[1] = b.x >> 16, w[2] = b.y & 0xffffu, w[3] = b.y >> 16;
  w[4] = b.z & 0xffffu, w[5] = b.z >> 16;
}
__device__ __forceinline__ void words_box(QBox& b, const uint32_t* w) {
  b = QBox{w[0] | w[1] << 16, w[2] | w[3] << 16, w[4] | w[5] << 16};
}
__device__ __forceinline__ void child_boxes(QBox& a, QBox& b, const uint4* nodes, int node) {
  const uint4 c0 = nodes[2 * (size_t)node], c1 = nodes[2 * (size_t)node + 1];
  a = QBox{c0.x ^ kFlipHi, c0.y ^ kFlipHi, c0.z ^ kFlipHi};
  b = QBox{c1.x ^ kFlipHi, c1.y ^ kFlipHi, c1.z ^ kFlipHi};
}

// In FP32.  fminf and fmaxf leave a NaN out of a union; a box that is not a
// number in an axis does not bound its record there.
struct FBox {
  float lx, ly, lz, hx, hy, hz;
};
__device__ __forceinline__ void leaf_box(FBox& b, const float4 l, const float4 h, const float4*) {
  b = FBox{l.x, l.y, l.z, h.x, h.y, h.z};
}
__device__ __forceinline__ FBox box_union(const FBox a, const FBox b) {
  return FBox{fminf(a.lx, b.lx), fminf(a.ly, b.ly), fminf(a.lz, b.lz),
              fmaxf(a.hx, b.hx), fmaxf(a.hy, b.hy), fmaxf(a.hz, b.hz)};
}
__device__ __forceinline__ void box_words(const FBox b, uint32_t w[6]) {
  w[0] = low_bits(b.lx), w[2] = low_bits(b.ly), w[4] = low_bits(b.lz);
  w[1] = ~high_bits(b.hx), w[3] = ~high_bits(b.hy), w[5] = ~high_bits(b.hz);
}
__device__ __forceinline__ void words_box(FBox& b, const uint32_t* w) {
  b = FBox{from_ordered(w[0]), from_ordered(w[2]), from_ordered(w[4]),
           from_ordered(~w[1]), from_ordered(~w[3]), from_ordered(~w[5])};
}
__device__ __forceinline__ void child_boxes(FBox& a, FBox& b, const uint4* nodes, int node) {
  const float4* r = reinterpret_cast<const float4*>(nodes) + 4 * (size_t)node;
  const float4 n0 = r[0], n1 = r[1], n2 = r[2];
  a = FBox{n0.x, n0.z, n2.x, n0.y, n0.w, n2.y};
  b = FBox{n1.x, n1.z, n2.z, n1.y, n1.w, n2.w};
}

// The record of a node from its children's boxes and indices.  The records are
// stored with an L2 evict-last policy: the frame kernel that follows the build
// reads them (with 64-byte records the full-head frame took 0.60 instead of
// 0.63 ms).
template <int N>
__device__ __forceinline__ void store_record(uint4* o, const uint4 (&v)[N]) {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
#pragma unroll
  for (int q = 0; q < N; ++q)
    asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;"
                 :: "l"(o + q), "r"(v[q].x), "r"(v[q].y), "r"(v[q].z), "r"(v[q].w), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void store_node(uint4* nodes, int node, const QBox c0, int i0, const QBox c1,
                                           int i1) {
  const uint4 v[2] = {make_uint4(c0.x ^ kFlipHi, c0.y ^ kFlipHi, c0.z ^ kFlipHi, (uint32_t)i0),
                      make_uint4(c1.x ^ kFlipHi, c1.y ^ kFlipHi, c1.z ^ kFlipHi, (uint32_t)i1)};
  store_record(nodes + 2 * (size_t)node, v);
}
__device__ __forceinline__ void store_node(uint4* nodes, int node, const FBox a, int i0, const FBox b,
                                           int i1) {
  auto u = [](float f) { return __float_as_uint(f); };
  const uint4 v[4] = {make_uint4(u(a.lx), u(a.hx), u(a.ly), u(a.hy)),
                      make_uint4(u(b.lx), u(b.hx), u(b.ly), u(b.hy)),
                      make_uint4(u(a.lz), u(a.hz), u(b.lz), u(b.hz)),
                      make_uint4((uint32_t)i0, (uint32_t)i1, 0u, 0u)};
  store_record(nodes + 4 * (size_t)node, v);
}

// What a node that spans blocks keeps in its record until k_span_records: its
// slot in the first word, and its children's indices in their places.
template <typename Box>
constexpr size_t kNodeWords = sizeof(Box) == sizeof(QBox) ? 2 : 4;
template <typename Box>
__device__ __forceinline__ void span_note(uint4* nodes, int node, unsigned slot, int i0, int i1) {
  uint4* o = nodes + kNodeWords<Box> * (size_t)node;
  if (kNodeWords<Box> == 2) {
    o[0] = make_uint4(slot, 0u, 0u, (uint32_t)i0);
    o[1] = make_uint4(0u, 0u, 0u, (uint32_t)i1);
  } else {
    o[0] = make_uint4(slot, 0u, 0u, 0u);
    o[3] = make_uint4((uint32_t)i0, (uint32_t)i1, 0u, 0u);
  }
}
template <typename Box>
__device__ __forceinline__ int2 span_children(const uint4* nodes, int node) {
  const uint4* o = nodes + kNodeWords<Box> * (size_t)node;
  return kNodeWords<Box> == 2 ? make_int2((int)o[0].w, (int)o[1].w) : make_int2((int)o[3].x, (int)o[3].y);
}

// Warp-aggregated append of one child (node index, or ~leaf) per lane that
// has one to the list of climb starts; every lane of the warp calls it.
__device__ __forceinline__ void append_start(bool has, int v, unsigned* count, int* list) {
  const unsigned m = __ballot_sync(0xffffffffu, has);
  if (!m) return;
  const int lane = threadIdx.x & 31, lead = __ffs(m) - 1;
  unsigned base = 0;
  if (lane == lead) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, lead);
  if (has) list[base + __popc(m & ((1u << lane) - 1u))] = v;
}

// The block's bounds (shared memory, ordered float bits) widened by the boxes of
// the threads with one.  Whole warps call it.
__device__ __forceinline__ void widen_bounds(const float4 bl, const float4 bh, bool has, uint32_t* bound) {
  const uint32_t lo[3] = {low_bits(bl.x + 0.f), low_bits(bl.y + 0.f), low_bits(bl.z + 0.f)};
  const uint32_t hi[3] = {high_bits(bh.x + 0.f), high_bits(bh.y + 0.f), high_bits(bh.z + 0.f)};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const uint32_t l = __reduce_min_sync(0xffffffffu, has ? lo[i] : 0xffffffffu);
    const uint32_t h = __reduce_max_sync(0xffffffffu, has ? hi[i] : 0u);
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&bound[i], l);
      atomicMax(&bound[3 + i], h);
    }
  }
}

// Records of the nodes whose leaves lie in the block's (thread j's node is
// `node`, with children ch, if `local`), one level of readiness per round.
// The whole block calls it, its leaves' ids and cleared flags in shared
// memory; leaf(i) is the box of the block's leaf i.
template <typename Box, typename Leaf>
__device__ __forceinline__ void local_records(bool local, const int4 ch, int node, int b0, int j,
                                              const uint32_t* s_id, const Leaf leaf, Box* s_nbox,
                                              unsigned char* s_done, uint4* nodes) {
  bool pending = local;
  for (;;) {
    bool ready = false;
    if (pending)
      ready = (ch.x < 0 || s_done[ch.x - b0]) && (ch.y < 0 || s_done[ch.y - b0]);
    if (ready) {
      const Box c0 = ch.x < 0 ? leaf(~ch.x - b0) : s_nbox[ch.x - b0];
      const Box c1 = ch.y < 0 ? leaf(~ch.y - b0) : s_nbox[ch.y - b0];
      // a leaf child is named by its primitive id (the leaf lies in this block)
      store_node(nodes, node, c0, ch.x < 0 ? ~(int)s_id[~ch.x - b0] : ch.x, c1,
                 ch.y < 0 ? ~(int)s_id[~ch.y - b0] : ch.y);
      s_nbox[j] = box_union(c0, c1);
    }
    const int any = __syncthreads_or(ready);  // this round's reads of s_done are over
    if (ready) {
      s_done[j] = 1;
      pending = false;
    }
    if (!any) break;
    __syncthreads();  // this round's flags are visible
  }
}

// The same in FP32, the leaves' boxes read from memory.
__device__ __forceinline__ void wide_records(bool local, const int4 ch, int node, int b0, int j,
                                          const uint32_t* s_id, const float4* box, FBox* s_nbox,
                                          unsigned char* s_done, uint4* nodes) {
  auto leaf = [&](int i) {
    FBox b;
    leaf_box(b, box[2 * (size_t)s_id[i]], box[2 * (size_t)s_id[i] + 1], nullptr);
    return b;
  };
  local_records(local, ch, node, b0, j, s_id, leaf, s_nbox, s_done, nodes);
}

// Leaf boxes and bottom-up bounds in one kernel.  Thread j of block b owns
// leaf b0 + j and internal node b0 + j (b0 = b * B).  A node record names a
// leaf child by ~(its global primitive id), so the frame kernel reads the
// primitive's records where they are (no copy into leaf order).
//  1. Gather: each thread reads its leaf's box (and id) into shared memory, on
//     the grid: three words, united by three 16-bit pair minima.  (FP32 boxes
//     take that room for the nodes and are read from memory again.)
//  2. Local subtrees: node i's leaf range starts or ends at leaf i, so a node
//     whose range lies inside the block's leaves ("local") is owned by a
//     thread of the block and so are its children.  These are finished in
//     rounds separated by barriers: a node whose children are done takes
//     their boxes from shared memory, writes its record and its union.  The
//     rounds number the local subtrees' height; no fences, no atomics.
//  3. The few nodes that span blocks are left to k_climb: their owners give
//     them a slot of twelve words (their children's coordinates, all taken as
//     minima), noted in the record, and the owner of each local node (or
//     leaf) whose parent spans blocks lists it as a climb start, so that no
//     block stays resident behind a climb.
template <int B>
__global__ void __launch_bounds__(B, 8) k_gather_refit(
    const int4* __restrict__ child, const int* __restrict__ parent_int,
    const int* __restrict__ parent_leaf, const float4* __restrict__ box,
    float4* frame, const uint32_t* sorted_ids, int n, uint4* nodes,
    uint32_t* leaf_id, unsigned* counts, int* starts, int* span_node, uint32_t* span) {
  __shared__ int4 s_child[B];
  __shared__ uint32_t s_id[B];  // global primitive id of each of the block's leaves
  __shared__ union {
    struct {
      QBox lbox[B], nbox[B];  // leaf boxes, unions of the block's local nodes
    } q;
    FBox nbox[B];
  } s_box;
  __shared__ unsigned char s_done[B];
  __shared__ uint32_t s_bound[6];
  const int b0 = blockIdx.x * B;
  const int j = threadIdx.x;
  const int leaf = b0 + j, node = b0 + j;
  const bool has_node = node <= n - 2;
  const bool wide = __ldg(&frame[0].w) != 0.f;
  int4 ch = make_int4(0, 0, -1, -1);
  if (has_node) ch = __ldg(child + node);
  s_child[j] = ch;
  s_done[j] = 0;
  const bool node_local = has_node && ch.z >= b0 && ch.w < b0 + B;
  // 1. gather
  int lparent = -1;
  float4 bl = make_float4(0.f, 0.f, 0.f, 0.f), bh = bl;
  if (leaf < n) {
    const uint32_t id = sorted_ids[leaf];
    lparent = parent_leaf[leaf] >> 1;
    leaf_id[leaf] = id;
    s_id[j] = id;
    bl = box[2 * (size_t)id];
    bh = box[2 * (size_t)id + 1];
    if (!wide) leaf_box(s_box.q.lbox[j], bl, bh, frame);
  }
  if (j < 6) s_bound[j] = j < 3 ? 0xffffffffu : 0u;
  __syncthreads();
  // the leaves' exact bounds (the camera rays are re-based at their entry into
  // them): the block's, and of those the few that reach further than any so
  // far (one read a block: a read a warp queued up at the one line, 0.17 ms
  // for 4.6M leaves)
  widen_bounds(bl, bh, leaf < n, s_bound);
  __syncthreads();
  if (j < 6) {
    uint32_t* g = reinterpret_cast<uint32_t*>(frame + 3) + j;
    const uint32_t v = s_bound[j], far = __ldcg(g);
    if (j < 3) {
      if (v < far) atomicMin(g, v);
    } else if (v > far) {
      atomicMax(g, v);
    }
  }
  // 2. local subtrees
  if (!wide)
    local_records(node_local, ch, node, b0, j, s_id, [&](int i) { return s_box.q.lbox[i]; }, s_box.q.nbox,
                  s_done, nodes);
  else
    wide_records(node_local, ch, node, b0, j, s_id, box, s_box.nbox, s_done, nodes);
  // 3. nodes that span blocks: empty child boxes, widened by k_climb
  const bool spans = has_node && !node_local;
  const unsigned m = __ballot_sync(0xffffffffu, spans);
  if (m) {
    const int lane = j & 31, lead = __ffs(m) - 1;
    unsigned base = 0;
    if (lane == lead) base = atomicAdd(counts + 1, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, lead);
    if (spans) {
      const unsigned slot = base + __popc(m & ((1u << lane) - 1u));
      span_node[slot] = node;
      for (int q = 0; q < 12; ++q) span[12 * (size_t)slot + q] = 0xffffffffu;
      const int c0 = ch.x < 0 ? ~(int)sorted_ids[~ch.x] : ch.x;
      const int c1 = ch.y < 0 ? ~(int)sorted_ids[~ch.y] : ch.y;
      if (!wide) span_note<QBox>(nodes, node, slot, c0, c1);
      else span_note<FBox>(nodes, node, slot, c0, c1);
    }
  }
  bool start_leaf = false, start_node = false;
  if (leaf < n && lparent >= 0)
    start_leaf = !(lparent >= b0 && lparent < b0 + B && s_child[lparent - b0].z >= b0 &&
                   s_child[lparent - b0].w < b0 + B);
  if (node_local && node != 0) {
    const int p = __ldg(parent_int + node) >> 1;
    start_node = !(p >= b0 && p < b0 + B && s_child[p - b0].z >= b0 && s_child[p - b0].w < b0 + B);
  }
  append_start(start_leaf, ~leaf, counts, starts);
  append_start(start_node, node, counts, starts);
}

// Bounds of the nodes that span blocks.  Each climb start (a leaf or local
// node whose parent spans blocks; its record is complete) lowers, with integer
// atomics, its own words in its parent's slot, then its parent's in the
// grandparent's, and so on to the root.  Each of the six coordinates stops at
// the first ancestor that it does not change: that one already holds a value
// at least as wide from another start below it, which carries it on up.  No
// ordering between starts is needed.
template <typename Box>
__device__ __forceinline__ void climb(const unsigned* __restrict__ counts, const int* __restrict__ starts,
                                      const int* __restrict__ parent_int,
                                      const int* __restrict__ parent_leaf, const float4* __restrict__ box,
                                      const float4* __restrict__ frame,
                                      const uint32_t* __restrict__ leaf_id,
                                      const uint4* __restrict__ nodes, uint32_t* span) {
  constexpr size_t W = kNodeWords<Box>;
  const unsigned m = *counts;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const int cur = __ldg(starts + i);
    Box u;
    int p;  // 2 * node + side; negative above the root
    if (cur < 0) {
      const size_t id = __ldg(leaf_id + ~cur);
      leaf_box(u, __ldg(box + 2 * id), __ldg(box + 2 * id + 1), frame);
      p = __ldg(parent_leaf + ~cur);
    } else {
      Box c0, c1;
      child_boxes(c0, c1, nodes, cur);
      u = box_union(c0, c1);
      p = __ldg(parent_int + cur);
    }
    uint32_t b[6];
    box_words(u, b);
    unsigned live = 0x3fu;
    // A start is a chain of levels, its time their latency: the links of the
    // level above are read while this level's atomics are out, and a node's
    // side comes with its link (a thumbnail of 3,001 strands 261 -> 248 us a call)
    uint32_t slot = __ldg(&nodes[W * (size_t)(p >> 1)].x);
    while (p >= 0) {
      uint32_t* r = span + 12 * (size_t)slot + 6 * (p & 1);
      uint32_t old[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) old[q] = (live >> q) & 1u ? atomicMin(r + q, b[q]) : 0u;
      p = p >> 1 ? __ldg(parent_int + (p >> 1)) : -1;
      if (p >= 0) slot = __ldg(&nodes[W * (size_t)(p >> 1)].x);
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (old[q] <= b[q]) live &= ~(1u << q);
      if (!live) break;
    }
  }
}
__global__ void k_climb(const unsigned* __restrict__ counts, const int* __restrict__ starts,
                        const int* __restrict__ parent_int, const int* __restrict__ parent_leaf,
                        const float4* __restrict__ box, const float4* __restrict__ frame,
                        const uint32_t* __restrict__ leaf_id, const uint4* __restrict__ nodes,
                        uint32_t* span) {
  if (__ldg(&frame[0].w) == 0.f)
    climb<QBox>(counts, starts, parent_int, parent_leaf, box, frame, leaf_id, nodes, span);
  else
    climb<FBox>(counts, starts, parent_int, parent_leaf, box, frame, leaf_id, nodes, span);
}

// The records of the nodes that span blocks, from their slots.
template <typename Box>
__device__ __forceinline__ void span_records(unsigned m, const int* __restrict__ span_node,
                                             const uint32_t* __restrict__ span, uint4* nodes) {
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const int node = span_node[i];
    const int2 ch = span_children<Box>(nodes, node);
    Box c0, c1;
    words_box(c0, span + 12 * (size_t)i);
    words_box(c1, span + 12 * (size_t)i + 6);
    store_node(nodes, node, c0, ch.x, c1, ch.y);
  }
}
__global__ void k_span_records(const unsigned* __restrict__ counts, const int* __restrict__ span_node,
                               const uint32_t* __restrict__ span, const float4* __restrict__ frame,
                               uint4* nodes) {
  if (__ldg(&frame[0].w) == 0.f)
    span_records<QBox>(counts[1], span_node, span, nodes);
  else
    span_records<FBox>(counts[1], span_node, span, nodes);
}

// A whole BVH of 2 to 1,024 leaves in one block, a leaf and a node per thread:
// codes, their stable sort (lanes with equal digits by votes, digits counted
// per warp, pairs exchanged through shared memory), Karras' nodes, the records
// and bounds.  `ids` null: every primitive in order.  The nine kernels it
// takes the place of (79 us for 1,024 leaves, launched one after the other)
// are latency and no work.
constexpr int kSmallLeaves = 1024, kSmallWarps = kSmallLeaves / 32;
struct SmallBvh {
  union {
    uint32_t whist[kSmallWarps][256];  // during the sort
    struct {
      QBox lbox[kSmallLeaves], nbox[kSmallLeaves];
    } box;
    FBox nbox[kSmallLeaves];
  };
  uint32_t key[kSmallLeaves], id[kSmallLeaves];
  unsigned char done[kSmallLeaves];
  uint32_t sum[8];
  float4 frame[kFrameWords];
};
__global__ void __launch_bounds__(kSmallLeaves)
    k_small_bvh(const float4* __restrict__ box, const uint32_t* __restrict__ ids, int n,
                const uint32_t* __restrict__ bounds, float4* frame, int4* child, int* parent_int,
                int* parent_leaf, uint32_t* leaf_id, uint4* nodes) {
  __shared__ SmallBvh sm;
  const int j = threadIdx.x, lane = j & 31, w = j >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const bool valid = j < n;
  uint32_t id = valid ? (ids ? ids[j] : (uint32_t)j) : 0u, key = 0u;
  {
    const float4 l[1] = {box[2 * (size_t)id]}, h[1] = {box[2 * (size_t)id + 1]};
    scene_grid<1>(bounds, l, h, valid, (uint32_t)n, sm.frame, nullptr);
    __syncthreads();
    if (valid) key = prim_code(l[0], h[0], sm.frame);
  }
  for (int shift = 0; shift < kMortonBits; shift += 8) {
    for (int i = j; i < kSmallWarps * 256; i += kSmallLeaves) (&sm.whist[0][0])[i] = 0;
    __syncthreads();
    const uint32_t d = (key >> shift) & 0xffu;
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
    if (!valid) peers = ~peers;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool bit = (d >> b) & 1u;
      const uint32_t vote = __ballot_sync(0xffffffffu, bit);
      peers &= bit ? vote : ~vote;
    }
    const uint32_t in = __popc(peers & lt);
    if (valid && in == 0) sm.whist[w][d] = __popc(peers);
    __syncthreads();
    uint32_t c = 0, incl = 0;
    if (j < 256) {
#pragma unroll 8
      for (int q = 0; q < kSmallWarps; ++q) {
        const uint32_t t = sm.whist[q][j];
        sm.whist[q][j] = c;
        c += t;
      }
      incl = c;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) sm.sum[w] = incl;
    }
    __syncthreads();
    if (j < 256) {
      uint32_t start = incl - c;
      for (int q = 0; q < w; ++q) start += sm.sum[q];
      for (int q = 0; q < kSmallWarps; ++q) sm.whist[q][j] += start;
    }
    __syncthreads();
    if (valid) {
      const uint32_t q = sm.whist[w][d] + in;
      sm.key[q] = key;
      sm.id[q] = id;
    }
    __syncthreads();
    if (valid) {
      key = sm.key[j];
      id = sm.id[j];
    }
  }
  // leaves: boxes on the grid and exact bounds (the whist words are free)
  __syncthreads();
  const bool wide = sm.frame[0].w != 0.f;
  float4 bl = make_float4(0.f, 0.f, 0.f, 0.f), bh = bl;
  if (valid) {
    bl = box[2 * (size_t)id];
    bh = box[2 * (size_t)id + 1];
    if (!wide) leaf_box(sm.box.lbox[j], bl, bh, sm.frame);
    leaf_id[j] = id;
  }
  sm.done[j] = 0;
  widen_bounds(bl, bh, valid, reinterpret_cast<uint32_t*>(sm.frame + 3));
  const bool has_node = j < n - 1;
  int4 ch = make_int4(0, 0, -1, -1);
  if (has_node) child[j] = ch = karras_node(sm.key, n, j, parent_int, parent_leaf);
  __syncthreads();
  if (j < (int)kFrameWords) frame[j] = sm.frame[j];
  if (!wide)
    local_records(has_node, ch, j, 0, j, sm.id, [&](int i) { return sm.box.lbox[i]; }, sm.box.nbox, sm.done,
                  nodes);
  else
    wide_records(has_node, ch, j, 0, j, sm.id, box, sm.nbox, sm.done, nodes);
}

__global__ void k_bytes_differ(const uint8_t* __restrict__ x, const uint8_t* __restrict__ y,
                               uint32_t n, uint32_t* diff) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && x[i] != y[i]) *diff = 1u;
}

// Nodes that span blocks of 256 leaves, at most: each holds both leaves at some
// boundary of two blocks, so it lies on the path from the root to their split,
// along which the common prefix grows from one node to the next: by a bit of
// the codes or, between equal codes, of the index.  (A slot for six leaves at
// 5M leaves, where one for each would be 52 bytes a leaf.)
size_t max_span_nodes(size_t n) {
  size_t bits = kMortonBits;
  while ((1ull << (bits - kMortonBits)) < n) ++bits;
  return std::min(n - 1, ((n + 255) / 256 - 1) * bits);
}

// Every node's record over the topology in bv and the primitives `ids` in leaf
// order, after scene_grid on the same stream.
hr_status gather_refit(hr_ctx* ctx, hr_asset* a, Bvh& bv, const uint32_t* ids, cudaStream_t st) {
  const uint32_t n = bv.n;
  unsigned* counts = nullptr;  // climb starts, nodes that span blocks
  int *starts = nullptr, *span_node = nullptr;
  uint32_t* span = nullptr;
  HR_TRY(scratch(ctx, 39, 16, (void**)&counts));
  const size_t slots = max_span_nodes(n);
  HR_TRY(scratch(ctx, 46, slots * 13 * 4, (void**)&span));
  HR_TRY(scratch(ctx, 48, (size_t)n * 2 * 4, (void**)&starts));  // one per leaf and per node at most
  span_node = reinterpret_cast<int*>(span + 12 * slots);
  k_gather_refit<256><<<(n + 255) / 256, 256, 0, st>>>(bv.child, bv.par_int, bv.par_leaf,
                                                       a->prim_box, bv.frame, ids, (int)n, bv.nodes,
                                                       bv.leaf_id, counts, starts, span_node, span);
  HR_LAUNCHED(ctx);
  if (n <= 256) return HR_OK;  // one block: every node is local
  static int climb_grid = 0;
  if (!climb_grid) {
    int dev = 0, sms = 1, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_climb, 256, 0) != cudaSuccess || per < 1) {
      cudaGetLastError();
      per = 1;
    }
    climb_grid = sms * per;
  }
  const unsigned grid = (unsigned)std::min<size_t>((size_t)climb_grid, ((size_t)n * 2 + 255) / 256);
  k_climb<<<grid, 256, 0, st>>>(counts, starts, bv.par_int, bv.par_leaf, a->prim_box,
                                bv.frame, bv.leaf_id, bv.nodes, span);
  HR_LAUNCHED(ctx);
  k_span_records<<<grid, 256, 0, st>>>(counts, span_node, span, bv.frame, bv.nodes);
  HR_LAUNCHED(ctx);
  return HR_OK;
}

}  // namespace

void free_bvh(hr_ctx* ctx, Bvh& bv) {
  if (bv.cap) {
    dfree(ctx, bv.nodes, (size_t)std::max(bv.cap, 2u) * 4 * sizeof(uint4));
    dfree(ctx, bv.frame, kFrameWords * sizeof(float4));
    dfree(ctx, bv.leaf_id, (size_t)bv.cap * 4);
    dfree(ctx, bv.child, (size_t)bv.cap * sizeof(int4));
    dfree(ctx, bv.par_int, (size_t)bv.cap * 4);
    dfree(ctx, bv.par_leaf, (size_t)bv.cap * 4);
  }
  if (bv.lod_built) dfree(ctx, bv.lod_built, bv.lod_cap);
  bv = Bvh();
}

hr_status build_bvh(hr_ctx* ctx, hr_asset* a, const uint8_t* lod_dev, Bvh& bv, cudaStream_t st) {
  const uint32_t N = a->N, S = a->S;
  bv.valid = 0;
  // 1. active primitives
  uint32_t n = 0, n_eth = 0;
  const bool strands = a->C == 0 || a->n_levels == 0 || lod_dev == nullptr;
  uint32_t* cnt = nullptr;
  if (strands) {
    n = N * S;
  } else {
    const uint32_t C = a->C;
    HR_TRY(scratch(ctx, 31, (size_t)(C + 2) * 4, (void**)&cnt));
    HR_CUDA(ctx, cudaMemsetAsync(cnt + C, 0, 8, st));
    k_cluster_counts<<<(C + 255) / 256, 256, 0, st>>>(lod_dev, a->cl_first, C, a->n_levels, S, cnt);
    HR_LAUNCHED(ctx);
    HR_TRY(scan_u32(ctx, cnt, C + 1, st));
    uint32_t tot[2] = {0, 0};  // active primitives, of which thick-hair segments
    HR_CUDA(ctx, cudaMemcpyAsync(tot, cnt + C, 8, cudaMemcpyDeviceToHost, st));
    HR_CUDA(ctx, cudaStreamSynchronize(st));
    n = tot[0];
    n_eth = tot[1];
  }
  // 2. storage (grow only)
  if (n > bv.cap) {
    if (bv.cap) {
      HR_CUDA(ctx, cudaStreamSynchronize(st));
      free_bvh(ctx, bv);
    }
    HR_TRY(dalloc(ctx, (void**)&bv.nodes, (size_t)std::max(n, 2u) * 4 * sizeof(uint4), "BVH nodes"));
    HR_TRY(dalloc(ctx, (void**)&bv.frame, kFrameWords * sizeof(float4), "BVH grid"));
    HR_TRY(dalloc(ctx, (void**)&bv.leaf_id, (size_t)n * 4, "BVH leaf ids"));
    HR_TRY(dalloc(ctx, (void**)&bv.child, (size_t)n * sizeof(int4), "BVH children"));
    HR_TRY(dalloc(ctx, (void**)&bv.par_int, (size_t)n * 4, "BVH parents"));
    HR_TRY(dalloc(ctx, (void**)&bv.par_leaf, (size_t)n * 4, "BVH leaf parents"));
    bv.cap = n;
  }
  // (after the grow: free_bvh resets every field)
  bv.n = n;
  bv.n_eth = n_eth;
  // their ids, and the scene's grid in a block of its own
  uint32_t* ids = nullptr;
  unsigned* counts = nullptr;
  const bool small = n >= 2 && n <= (uint32_t)kSmallLeaves;
  HR_TRY(scratch(ctx, 39, 16, (void**)&counts));
  if (strands) {
    if (!small) {
      HR_TRY(scratch(ctx, 30, (size_t)n * 4, (void**)&ids));
      k_iota<<<(n + 255) / 256 + 1, 256, 0, st>>>(ids, n, a->d_bounds, a->prim_box, bv.frame, counts);
      HR_LAUNCHED(ctx);
    }
  } else if (n) {
    uint32_t* eoff = nullptr;
    HR_TRY(scratch(ctx, 32, 16 * 4, (void**)&eoff));
    HR_CUDA(ctx, cudaMemcpyAsync(eoff, a->eth_offset, 16 * 4, cudaMemcpyHostToDevice, st));
    HR_TRY(scratch(ctx, 30, (size_t)n * 4, (void**)&ids));
    k_cluster_fill<<<a->C + 1, 256, 0, st>>>(lod_dev, a->cl_first, a->order, cnt, eoff, a->C, a->n_levels,
                                             N, S, ids, a->d_bounds, a->prim_box, bv.frame, counts);
    HR_LAUNCHED(ctx);
  }
  // what the topology is built for (checked by refit_bvh); the hierarchy as it is now
  HR_CUDA(ctx, cudaMemsetAsync(a->d_bounds + kHierChanged, 0, 4, st));
  bv.topo = 0;
  bv.built_C = a->C;
  bv.built_E = a->E;
  bv.built_total = a->n_prims_total;
  bv.built_with_lod = lod_dev != nullptr;
  if (lod_dev) {
    if (bv.lod_cap < a->C) {
      if (bv.lod_built) dfree(ctx, bv.lod_built, bv.lod_cap);
      bv.lod_built = nullptr;
      bv.lod_cap = 0;
      HR_TRY(dalloc(ctx, (void**)&bv.lod_built, a->C, "BVH LoD"));
      bv.lod_cap = a->C;
    }
    HR_CUDA(ctx, cudaMemcpyAsync(bv.lod_built, lod_dev, a->C, cudaMemcpyDeviceToDevice, st));
  }
  if (n == 0) {
    bv.valid = 1;
    bv.topo = 1;
    return HR_OK;
  }
  if (small) {  // all in one block
    k_small_bvh<<<1, kSmallLeaves, 0, st>>>(a->prim_box, ids, (int)n, a->d_bounds, bv.frame, bv.child,
                                            bv.par_int, bv.par_leaf, bv.leaf_id, bv.nodes);
    HR_LAUNCHED(ctx);
    bv.valid = 1;
    bv.topo = 1;
    return HR_OK;
  }
  // 3. Morton codes and sort
  uint32_t *keys, *k2, *v2;
  HR_TRY(scratch(ctx, 33, (size_t)n * 4, (void**)&keys));
  HR_TRY(scratch(ctx, 34, (size_t)n * 4, (void**)&k2));
  HR_TRY(scratch(ctx, 35, (size_t)n * 4, (void**)&v2));
  k_prim_morton<<<(n + 255) / 256, 256, 0, st>>>(a->prim_box, ids, n, bv.frame, keys);
  HR_LAUNCHED(ctx);
  HR_TRY(radix_sort_pairs(ctx, keys, ids, k2, v2, n, kMortonBits, st, kLookbackPolls, &keys, &ids));
  if (n == 1) {
    k_gather<<<1, 32, 0, st>>>(ids, n, bv.leaf_id);
    HR_LAUNCHED(ctx);
    bv.valid = 1;
    bv.topo = 1;
    return HR_OK;
  }
  // 4. hierarchy, then leaf records and bounds in one bottom-up pass
  k_karras<<<(n - 1 + 255) / 256, 256, 0, st>>>(keys, (int)n, bv.child, bv.par_int, bv.par_leaf);
  HR_LAUNCHED(ctx);
  HR_TRY(gather_refit(ctx, a, bv, ids, st));
  bv.valid = 1;
  bv.topo = 1;
  return HR_OK;
}

hr_status refit_bvh(hr_ctx* ctx, hr_asset* a, const uint8_t* lod_dev, Bvh& bv, cudaStream_t st) {
  if (!bv.topo || bv.built_C != a->C || bv.built_E != a->E || bv.built_total != a->n_prims_total ||
      bv.built_with_lod != (lod_dev != nullptr))
    return set_error(ctx, HR_ESTATE, "refit: the BVH was built for another hierarchy");
  {
    // one read-back: the LoD selection against the build's, and whether a
    // hierarchy build changed the strand order since
    uint32_t* diff = nullptr;
    HR_TRY(scratch(ctx, 36, 8, (void**)&diff));
    HR_CUDA(ctx, cudaMemsetAsync(diff, 0, 4, st));
    if (lod_dev) {
      k_bytes_differ<<<(a->C + 255) / 256, 256, 0, st>>>(lod_dev, bv.lod_built, a->C, diff);
      HR_LAUNCHED(ctx);
    }
    HR_CUDA(ctx, cudaMemcpyAsync(diff + 1, a->d_bounds + kHierChanged, 4, cudaMemcpyDeviceToDevice, st));
    uint32_t h[2] = {0, 0};
    HR_CUDA(ctx, cudaMemcpyAsync(h, diff, 8, cudaMemcpyDeviceToHost, st));
    HR_CUDA(ctx, cudaStreamSynchronize(st));
    if (h[0]) return set_error(ctx, HR_ESTATE, "refit: the LoD selection changed since the build");
    if (h[1]) return set_error(ctx, HR_ESTATE, "refit: the strand order changed since the build");
  }
  bv.valid = 0;
  const uint32_t n = bv.n;
  // a single leaf has no node; its records are the primitive's own
  if (n > 1) {
    unsigned* counts = nullptr;
    HR_TRY(scratch(ctx, 39, 16, (void**)&counts));
    k_scene_grid<<<1, 256, 0, st>>>(a->d_bounds, a->prim_box, a->N * a->S, bv.frame, counts);
    HR_LAUNCHED(ctx);
    HR_TRY(gather_refit(ctx, a, bv, bv.leaf_id, st));
  }
  bv.valid = 1;
  return HR_OK;
}

}  // namespace hr
