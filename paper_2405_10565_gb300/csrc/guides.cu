// Guide hairs, the guide-driven hierarchy and linear skinning (Section 5.1
// steps 1, 2 and 4; Section 5.2 "Runtime").
//
//  * Guides: k-means over the strands with D(i, j) = sum_k |p^{i,k} -
//    p^{j,k}|^2 over corresponding vertices, each cluster's guide its medoid
//    (the member with the smallest sum of distances to the others).
//  * Hierarchy: every strand's three nearest guides; strands sharing the same
//    three form one cluster of the coarsest level, listed in (Morton code of
//    the root, id) order; finer levels, fits and records as for the Morton
//    hierarchy.
//  * Skinning: every strand vertex and every thick-hair cross-section centre
//    and corner (c +- a e1, c +- b e2) gets weights in the triangular prism
//    of its cluster's three guides' corresponding points, p = g0 + w1 (g1 -
//    g0) + w2 (g2 - g0) + h n (n the unit normal of the triangle; a
//    degenerate triangle keeps the offset p - g0).  A new pose of the guides
//    moves the strands and the thick hairs without a new clustering or fit.
//
// D, the centroid sums and the medoid sums are FP32 without contraction, in
// vertex order and, over members, in ascending strand id: the decisions they
// make (cluster ids, medoids, nearest guides) are reproducible and compare bit
// for bit with a plain FP32 evaluation in that order.  The prisms are FP64 and
// their points' weights double-word FP32 (once per hierarchy), the skinning FP32
// (every frame).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "dword.cuh"

namespace hr {
namespace {

constexpr uint32_t kMaxGuides = 1024;  // three guide indices of 10 bits in one key

// One vertex's term of D: ((dx dx + dy dy) + dz dz), each operation rounded.
__device__ __forceinline__ float point_d(const float4 a, const float4 b) {
  const float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y), dz = __fsub_rn(a.z, b.z);
  return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

__device__ __forceinline__ float strand_d(const float4* __restrict__ A, const float4* __restrict__ B,
                                          uint32_t S1) {
  float d = 0.f;
#pragma unroll 4
  for (uint32_t k = 0; k < S1; ++k) d = __fadd_rn(d, point_d(__ldg(A + k), __ldg(B + k)));
  return d;
}

__global__ void k_seed(const float4* __restrict__ verts, uint32_t S1, const uint32_t* __restrict__ order,
                       uint32_t N, uint32_t G, float4* cent) {
  const uint32_t g = blockIdx.x;
  const uint32_t s = order[(uint32_t)(((uint64_t)(2 * g + 1) * N) / (2ull * G))];
  for (uint32_t k = threadIdx.x; k < S1; k += blockDim.x) {
    const float4 p = verts[(size_t)s * S1 + k];
    cent[(size_t)g * S1 + k] = make_float4(p.x, p.y, p.z, 0.f);
  }
}

// A tile of 32 strands that are neighbours on the scalp (consecutive Morton
// ranks), one per lane, searched by the block's four warps against a set of
// polylines (centroids or guides): warp w takes rows 4w .. 4w + 3 of every 16.
// Every term of D is non-negative and FP32 rounding is monotone, so a partial
// sum never falls: a group of four rows is left as soon as every lane's
// partial sums are above the lane's bound, which changes no result.  The
// lanes being neighbours, they leave together.  With the tile's vertices in
// shared memory (k-major, 33 words a row so that filling and reading are free
// of bank conflicts) a strand is read from memory once per search.  Bound:
// FP32 issue; without the bound and the tile (one thread per strand over all
// rows, its own scattered loads for each eight rows) the assignment of 100k
// strands x 65 vertices to 256 centroids took 1.83 ms.
constexpr uint32_t kTileWarps = 4;
constexpr uint32_t kTileMaxVerts = 256;  // 99 KB of shared memory; longer strands are read in place
__device__ __forceinline__ size_t tile_word(uint32_t k, uint32_t c, uint32_t lane) {
  return (size_t)(k * 3 + c) * 33 + lane;
}
inline size_t tile_bytes(uint32_t S1) { return (size_t)S1 * 3 * 33 * sizeof(float); }

__device__ __forceinline__ void tile_fill(float* sp, const float4* __restrict__ verts, uint32_t S1,
                                          const uint32_t* __restrict__ order, uint32_t r0,
                                          uint32_t n) {
  for (uint32_t i = threadIdx.x; i < n * S1; i += blockDim.x) {
    const uint32_t row = i / S1, k = i - row * S1;
    const float4 p = __ldg(verts + (size_t)__ldg(order + r0 + row) * S1 + k);
    sp[tile_word(k, 0, row)] = p.x;
    sp[tile_word(k, 1, row)] = p.y;
    sp[tile_word(k, 2, row)] = p.z;
  }
}

// D of the lane's strand (tile, or its row P) to four rows at once, left early
// once no lane of the warp has a partial sum at or below its bound (then
// returns false).  Whole warps call it.
template <bool TILE>
__device__ __forceinline__ bool four_d(const float* sp, const float4* __restrict__ P,
                                       const float4* const row[4], uint32_t S1, float bound,
                                       float d[4]) {
  const uint32_t lane = threadIdx.x & 31;
  d[0] = d[1] = d[2] = d[3] = 0.f;
  for (uint32_t k0 = 0; k0 < S1; k0 += 8) {
    const uint32_t k1 = min(k0 + 8, S1);
#pragma unroll 4
    for (uint32_t k = k0; k < k1; ++k) {
      float4 p;
      if (TILE)
        p = make_float4(sp[tile_word(k, 0, lane)], sp[tile_word(k, 1, lane)],
                        sp[tile_word(k, 2, lane)], 0.f);
      else
        p = __ldg(P + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = __fadd_rn(d[j], point_d(p, __ldg(row[j] + k)));
    }
    const bool alive = d[0] <= bound || d[1] <= bound || d[2] <= bound || d[3] <= bound;
    if (!__any_sync(0xffffffffu, alive)) return false;
  }
  return true;
}

template <bool TILE>
__device__ __forceinline__ float one_d(const float* sp, const float4* __restrict__ P,
                                       const float4* __restrict__ row, uint32_t S1) {
  const uint32_t lane = threadIdx.x & 31;
  float d = 0.f;
#pragma unroll 4
  for (uint32_t k = 0; k < S1; ++k) {
    const float4 p = TILE ? make_float4(sp[tile_word(k, 0, lane)], sp[tile_word(k, 1, lane)],
                                        sp[tile_word(k, 2, lane)], 0.f)
                          : __ldg(P + k);
    d = __fadd_rn(d, point_d(p, __ldg(row + k)));
  }
  return d;
}

// Nearest centroid of every strand (ties: the lower cluster; cluster 0 when
// no D is finite).  The first bound is D to a likely centroid: the strand's
// previous cluster, or before the first assignment the seed of its Morton rank.
template <bool TILE>
__global__ void __launch_bounds__(32 * kTileWarps)
    k_assign(const float4* __restrict__ verts, uint32_t N, uint32_t S1,
             const float4* __restrict__ cent, uint32_t G, const uint32_t* __restrict__ order,
             bool have_prev, uint32_t* assign) {
  extern __shared__ float sp[];
  __shared__ float s_d[kTileWarps][32];
  __shared__ uint32_t s_g[kTileWarps][32];
  const uint32_t r0 = blockIdx.x * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t n = min(32u, N - r0);
  if (TILE) tile_fill(sp, verts, S1, order, r0, n);
  const uint32_t id = order[min(r0 + lane, N - 1)];
  const float4* P = verts + (size_t)id * S1;
  uint32_t bg = 0;
  float best = -1.f;  // lanes past the last strand: never alive
  __syncthreads();
  if (lane < n) {
    const uint32_t g = have_prev ? assign[id] : (uint32_t)(((uint64_t)(r0 + lane) * G) / N);
    best = one_d<TILE>(sp, P, cent + (size_t)g * S1, S1);
    if (best < __int_as_float(0x7f800000)) {
      bg = g;
    } else {  // infinite or not a number: no bound
      best = __int_as_float(0x7f800000);
    }
  }
  for (uint32_t g0 = 4 * w; g0 < G; g0 += 4 * kTileWarps) {
    const float4* row[4];
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) row[j] = cent + (size_t)min(g0 + j, G - 1) * S1;
    float d[4];
    if (!four_d<TILE>(sp, P, row, S1, best, d)) continue;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
      if (g0 + j < G && (d[j] < best || (d[j] == best && g0 + j < bg))) {
        best = d[j];
        bg = g0 + j;
      }
  }
  s_d[w][lane] = best;
  s_g[w][lane] = bg;
  __syncthreads();
  if (w == 0 && lane < n) {
    for (uint32_t q = 1; q < kTileWarps; ++q)
      if (s_d[q][lane] < best || (s_d[q][lane] == best && s_g[q][lane] < bg)) {
        best = s_d[q][lane];
        bg = s_g[q][lane];
      }
    assign[id] = bg;
  }
}

__global__ void k_iota_copy(const uint32_t* __restrict__ src, uint32_t n, uint32_t* keys,
                            uint32_t* vals) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = src[i];
  vals[i] = i;
}

// First rank of every key 0 .. G in the sorted keys.
__global__ void k_key_starts(const uint32_t* __restrict__ key, uint32_t n, uint32_t G,
                             uint32_t* start) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g > G) return;
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(key + mid) < g) lo = mid + 1; else hi = mid;
  }
  start[g] = lo;
}

// Centroid of every cluster: the members' vertices summed in ascending strand
// id (FP32), divided by the count; an empty cluster keeps its centroid.  One
// thread per coordinate: the sum is a chain, so its latency is hidden by 16
// members' loads in flight (84 us for 100k strands in 256 clusters, the longest
// cluster's chain; one load at a time took 235) and the coordinates of a cluster are
// spread over several blocks.
constexpr uint32_t kUpdateBlock = 64;
__global__ void __launch_bounds__(kUpdateBlock)
    k_update(const float4* __restrict__ verts, uint32_t S1, const uint32_t* __restrict__ start,
             const uint32_t* __restrict__ ids, float4* cent) {
  const uint32_t g = blockIdx.x;
  const uint32_t r0 = start[g], r1 = start[g + 1];
  const uint32_t j = blockIdx.y * kUpdateBlock + threadIdx.x;
  if (r1 == r0 || j >= S1 * 3) return;
  const uint32_t k = j / 3, c = j % 3;
  const float* V = reinterpret_cast<const float*>(verts) + (size_t)k * 4 + c;
  const size_t stride = (size_t)S1 * 4;
  float acc = 0.f;
  uint32_t r = r0;
  for (; r + 16 <= r1; r += 16) {
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __ldg(V + stride * __ldg(ids + r + q));
#pragma unroll
    for (int q = 0; q < 16; ++q) acc = __fadd_rn(acc, v[q]);
  }
  for (; r < r1; ++r) acc = __fadd_rn(acc, __ldg(V + stride * __ldg(ids + r)));
  reinterpret_cast<float*>(cent + (size_t)g * S1)[k * 4 + c] = __fdiv_rn(acc, (float)(r1 - r0));
}

// ---------------------------------------------------------------- medoids
//
// Medoid of every cluster: the member i whose FP32 sum s_i of D to the members
// (in ascending id) is least; ties to the lower strand id; -1 for an empty
// cluster.  In exact arithmetic s_i = m T_i + W with T_i the squared distance
// of i to the cluster's mean and W = sum_q T_q, and every term of s_i is
// non-negative, so the FP32 sum is within a relative gamma_(m + S1 + 5) of it.
// Only members whose lower bound does not exceed the least upper bound can be
// the medoid; the FP32 sums are formed for these alone (a few per cluster,
// where all m^2 pairs took 16.9 ms for 100k strands in 256 clusters; 0.2 now).  Where
// the bounds are not finite every member stays a candidate.

struct MedoidWork {
  double* csum;      // [G][S1 * 3] sums of the members' coordinates, then (hi, lo) of their means
  double* W;         // [G] sum of T
  unsigned long long* best;  // [G] (bits of the least FP32 sum, strand id)
  uint32_t* tmin;    // [G] bits of the least T
  uint32_t* vmax;    // [G] bits of the largest squared norm of a member's coordinates
  uint32_t* n_cand;  // [1]
  float* T;          // [N] by rank
  uint32_t* cand;    // [N] ranks
};

__global__ void k_medoid_init(MedoidWork mw, uint32_t G, uint64_t n_sum) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_sum) mw.csum[i] = 0.0;
  if (i < G) {
    mw.W[i] = 0.0;
    mw.best[i] = 0x7f800000ffffffffull;  // (infinity, no strand)
    mw.tmin[i] = 0xffffffffu;
    mw.vmax[i] = 0u;
  }
  if (i == 0) *mw.n_cand = 0u;
}

// Sums of the members' coordinates: a block takes 64 ranks, a thread one
// coordinate, in double-word FP32, added to the cluster's FP64 sum where the
// cluster changes.  The order of these additions varies by run; the bounds
// below leave room for it.
constexpr uint32_t kSumRanks = 64;
__global__ void __launch_bounds__(256)
    k_member_sums(const float4* __restrict__ verts, uint32_t N, uint32_t S1,
                  const uint32_t* __restrict__ key, const uint32_t* __restrict__ ids, double* csum) {
  __shared__ uint32_t s_key[kSumRanks], s_id[kSumRanks];
  const uint32_t r0 = blockIdx.x * kSumRanks, n = min(kSumRanks, N - r0);
  if (threadIdx.x < n) {
    s_key[threadIdx.x] = key[r0 + threadIdx.x];
    s_id[threadIdx.x] = ids[r0 + threadIdx.x];
  }
  __syncthreads();
  const float* V = reinterpret_cast<const float*>(verts);
  for (uint32_t j = threadIdx.x; j < S1 * 3; j += blockDim.x) {
    const size_t off = (size_t)(j / 3) * 4 + j % 3;
    float hi = 0.f, lo = 0.f;
#pragma unroll 8
    for (uint32_t i = 0; i < n; ++i) {
      float e;
      hi = two_sum(hi, __ldg(V + (size_t)s_id[i] * S1 * 4 + off), e);
      lo = __fadd_rn(lo, e);
      if (i + 1 == n || s_key[i + 1] != s_key[i]) {
        atomicAdd(csum + (size_t)s_key[i] * S1 * 3 + j, (double)hi + (double)lo);
        hi = lo = 0.f;
      }
    }
  }
}

// Means of the non-empty clusters as double-word FP32 pairs, in place.
__global__ void k_means(double* csum, const uint32_t* __restrict__ start, uint32_t G, uint32_t S1) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (uint64_t)G * S1 * 3) return;
  const uint32_t g = (uint32_t)(i / (S1 * 3));
  const uint32_t m = start[g + 1] - start[g];
  const double c = csum[i] / (double)max(m, 1u);
  const float hi = (float)c;
  reinterpret_cast<float2*>(csum)[i] = make_float2(hi, (float)(c - (double)hi));
}

// T of every member: one warp per rank.
__global__ void __launch_bounds__(256)
    k_member_spread(const float4* __restrict__ verts, uint32_t N, uint32_t S1,
                    const uint32_t* __restrict__ key, const uint32_t* __restrict__ ids,
                    MedoidWork mw) {
  const uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= N) return;
  const uint32_t g = key[r];
  const float* V = reinterpret_cast<const float*>(verts + (size_t)ids[r] * S1);
  const float2* M = reinterpret_cast<const float2*>(mw.csum) + (size_t)g * S1 * 3;
  float acc = 0.f, nrm = 0.f;
  for (uint32_t j = lane; j < S1 * 3; j += 32) {
    const float2 c = __ldg(M + j);
    const float v = __ldg(V + (size_t)(j / 3) * 4 + j % 3);
    const float d = __fsub_rn(__fsub_rn(v, c.x), c.y);
    acc = fmaf(d, d, acc);
    nrm = fmaf(v, v, nrm);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, o);
    nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
  }
  if (lane == 0) {
    mw.T[r] = acc;
    atomicAdd(mw.W + g, (double)acc);
    atomicMin(mw.tmin + g, __float_as_uint(acc));
    atomicMax(mw.vmax + g, __float_as_uint(nrm));
  }
}

// Members that can be the medoid.  u = 2^-24; T and W are within (S1 3 / 32 +
// 16) u of exact (the lanes' chains, their tree, the mean's two words), the
// FP32 sums within (m + S1 + 8) u, each with a tenth on top; squares that
// underflow add at most m S1 3 2^-147.  Where the least sum may overflow (the
// medoid is then the lowest id) every member stays a candidate.  A mean off by delta moves s_i by at
// most 2 m |delta| sqrt(T); the sums of 64 ranks are within 2^-36 of their
// terms' magnitudes (Sum2), so |delta| is below 2^-35 of the largest norm.
__global__ void k_medoid_candidates(const uint32_t* __restrict__ key, uint32_t N, uint32_t S1,
                                    const uint32_t* __restrict__ start, MedoidWork mw) {
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  const uint32_t g = key[r];
  const double m = (double)(start[g + 1] - start[g]), u = 5.9604644775390625e-08;
  const double tau = 1.1 * ((double)S1 * 3.0 / 32.0 + 16.0) * u, eps = 1.1 * (m + S1 + 8.0) * u;
  const double W = mw.W[g], tmin = (double)__uint_as_float(mw.tmin[g]), t = (double)mw.T[r];
  const double move = 2.0 * m * (sqrt(t) + sqrt(tmin)) * 2.9103830456733704e-11 *
                      sqrt((double)__uint_as_float(mw.vmax[g]));
  const double lower = (m * t + W) * (1.0 - tau) * (1.0 - eps);
  const double upper = (m * tmin + W) * (1.0 + tau) * (1.0 + eps) + move +
                       m * S1 * 3.0 * 5.605193857299268e-45;
  if (lower > upper && upper < 3.4028234e38 && eps < 0.5) return;  // NaN compares false: stays
  mw.cand[atomicAdd(mw.n_cand, 1u)] = r;
}

// The FP32 sums of the candidates, one block each: 256 members' D at a time,
// added in order by one thread, which stops once the sum (it never falls) is
// above the cluster's least.
__global__ void __launch_bounds__(256)
    k_medoid_sums(const float4* __restrict__ verts, uint32_t S1, const uint32_t* __restrict__ key,
                  const uint32_t* __restrict__ start, const uint32_t* __restrict__ ids,
                  MedoidWork mw) {
  __shared__ float s_d[256];
  __shared__ int s_over;
  const uint32_t n = *mw.n_cand;
  for (uint32_t c = blockIdx.x; c < n; c += gridDim.x) {
    const uint32_t r = mw.cand[c], g = key[r], id = ids[r];
    const uint32_t q0 = start[g], q1 = start[g + 1];
    const float4* P = verts + (size_t)id * S1;
    float s = 0.f;
    if (threadIdx.x == 0) s_over = 0;
    for (uint32_t q = q0; q < q1; q += 256) {
      const uint32_t cnt = min(256u, q1 - q);
      if (threadIdx.x < cnt)
        s_d[threadIdx.x] = strand_d(P, verts + (size_t)ids[q + threadIdx.x] * S1, S1);
      __syncthreads();
      if (threadIdx.x == 0) {
#pragma unroll 8
        for (uint32_t i = 0; i < cnt; ++i) s = __fadd_rn(s, s_d[i]);
        const float least = __uint_as_float((uint32_t)(__ldcg(mw.best + g) >> 32));
        if (s > least) s_over = 1;
      }
      __syncthreads();
      if (s_over) break;
    }
    if (threadIdx.x == 0 && !s_over && s == s)
      atomicMin(mw.best + g, ((unsigned long long)__float_as_uint(s) << 32) | id);
    __syncthreads();  // s_over and s_d are free again
  }
}

__global__ void k_medoid_write(const unsigned long long* __restrict__ best,
                               const uint32_t* __restrict__ start, uint32_t G, int32_t* guides) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < G) guides[g] = start[g + 1] > start[g] ? (int32_t)(uint32_t)best[g] : -1;
}

// ---------------------------------------------------------------- nearest guides

// The three guides nearest to every guide, itself among them (any three
// guides give a valid bound below, near ones a tight one).
__global__ void __launch_bounds__(128)
    k_guide_neighbours(const float4* __restrict__ verts, uint32_t S1,
                       const int32_t* __restrict__ guides, uint32_t G, uint32_t* nb) {
  __shared__ float s_d[kMaxGuides];
  const uint32_t g = blockIdx.x;
  const float inf = __int_as_float(0x7f800000);
  const int32_t s = guides[g];
  for (uint32_t j = threadIdx.x; j < G; j += blockDim.x) {
    const int32_t t = guides[j];
    float d = inf;
    if (s >= 0 && t >= 0) {
      d = strand_d(verts + (size_t)s * S1, verts + (size_t)t * S1, S1);
      if (!(d < 1e38f)) d = 1e38f;  // a guide all the same
    }
    s_d[j] = d;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  for (int q = 0; q < 3; ++q) {
    float bd = inf;
    uint32_t bj = 0xffffffffu;
    for (uint32_t j = threadIdx.x; j < G; j += 32)
      if (s_d[j] < bd) {
        bd = s_d[j];
        bj = j;
      }
    for (int o = 16; o; o >>= 1) {
      const float od = __shfl_xor_sync(0xffffffffu, bd, o);
      const uint32_t oj = __shfl_xor_sync(0xffffffffu, bj, o);
      if (od < bd || (od == bd && oj < bj)) {
        bd = od;
        bj = oj;
      }
    }
    if (threadIdx.x == 0) {
      nb[3 * g + q] = bj;
      if (bj != 0xffffffffu) s_d[bj] = inf;
    }
    __syncwarp();
  }
}

// The three nearest of a set, ordered by (D, index); empty places are
// (infinity, 0).
struct Near3 {
  float d0, d1, d2;
  uint32_t g0, g1, g2;
};
__device__ __forceinline__ void near3_insert(Near3& b, float d, uint32_t g) {
  if (!(d < __int_as_float(0x7f800000))) return;
  if (!(d < b.d2 || (d == b.d2 && g < b.g2))) return;
  if (d < b.d1 || (d == b.d1 && g < b.g1)) {
    b.d2 = b.d1;
    b.g2 = b.g1;
    if (d < b.d0 || (d == b.d0 && g < b.g0)) {
      b.d1 = b.d0;
      b.g1 = b.g0;
      b.d0 = d;
      b.g0 = g;
    } else {
      b.d1 = d;
      b.g1 = g;
    }
  } else {
    b.d2 = d;
    b.g2 = g;
  }
}

// The three nearest guides of every strand (ties: the lower guide), as a key
// of three ascending 10-bit guide indices, for the strands in Morton order.
// The first bound is the largest D to the guide of the strand's cluster and
// that guide's neighbours: the third nearest is no farther.
template <bool TILE>
__global__ void __launch_bounds__(32 * kTileWarps)
    k_nearest3(const float4* __restrict__ verts, uint32_t N, uint32_t S1,
               const int32_t* __restrict__ guides, uint32_t G, const uint32_t* __restrict__ nb,
               const uint32_t* __restrict__ assign, const uint32_t* __restrict__ order,
               uint32_t* key) {
  extern __shared__ float sp[];
  __shared__ float s_d[kTileWarps][3][32];
  __shared__ uint32_t s_g[kTileWarps][3][32];
  const uint32_t r0 = blockIdx.x * 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t n = min(32u, N - r0);
  if (TILE) tile_fill(sp, verts, S1, order, r0, n);
  const uint32_t id = order[min(r0 + lane, N - 1)];
  const float4* P = verts + (size_t)id * S1;
  const float inf = __int_as_float(0x7f800000);
  float bound = -1.f;
  __syncthreads();
  if (lane < n) {
    bound = 0.f;
    const uint32_t* q = nb + 3 * (size_t)assign[id];
    for (int j = 0; j < 3; ++j) {
      float d = inf;
      if (q[j] < G) d = one_d<TILE>(sp, P, verts + (size_t)guides[q[j]] * S1, S1);
      bound = d < inf ? fmaxf(bound, d) : inf;
    }
  }
  Near3 b{inf, inf, inf, 0u, 0u, 0u};
  for (uint32_t g0 = 4 * w; g0 < G; g0 += 4 * kTileWarps) {
    const float4* row[4];
    bool live[4];
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      const int32_t s = g0 + j < G ? __ldg(guides + g0 + j) : -1;
      live[j] = s >= 0;
      row[j] = verts + (size_t)max(s, 0) * S1;
    }
    float d[4];
    if (!four_d<TILE>(sp, P, row, S1, fminf(bound, b.d2), d)) continue;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j)
      if (live[j]) near3_insert(b, d[j], g0 + j);
  }
  s_d[w][0][lane] = b.d0; s_d[w][1][lane] = b.d1; s_d[w][2][lane] = b.d2;
  s_g[w][0][lane] = b.g0; s_g[w][1][lane] = b.g1; s_g[w][2][lane] = b.g2;
  __syncthreads();
  if (w != 0 || lane >= n) return;
  for (uint32_t q = 1; q < kTileWarps; ++q)
    for (int j = 0; j < 3; ++j) near3_insert(b, s_d[q][j][lane], s_g[q][j][lane]);
  // ascending guide indices
  uint32_t x = b.g0, y = b.g1, z = b.g2, t;
  if (x > y) t = x, x = y, y = t;
  if (y > z) t = y, y = z, z = t;
  if (x > y) t = x, x = y, y = t;
  key[r0 + lane] = (x << 20) | (y << 10) | z;
}

// Cluster starts from the ranks where the sorted key changes (excl = the
// exclusive scan of those flags); the number of clusters into *C.
__global__ void k_starts(const uint32_t* __restrict__ key, const uint32_t* __restrict__ excl,
                         uint32_t N, uint32_t* cl_first, uint32_t* cl_tri, uint32_t* C) {
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  const bool head = r == 0 || key[r] != key[r - 1];
  if (head) {
    cl_first[excl[r]] = r;
    cl_tri[excl[r]] = key[r];
  }
  if (r == N - 1) {
    const uint32_t n = excl[r] + (head ? 1u : 0u);
    cl_first[n] = N;
    *C = n;
  }
}

__global__ void k_head_flags(const uint32_t* __restrict__ key, uint32_t N, uint32_t* flags) {
  const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < N) flags[r] = (r == 0 || key[r] != key[r - 1]) ? 1u : 0u;
}

// ---------------------------------------------------------------- prism weights

struct D3 {
  double x, y, z;
};
__device__ __forceinline__ D3 d3(const float4 p) { return D3{p.x, p.y, p.z}; }
__device__ __forceinline__ D3 dsub(D3 a, D3 b) { return D3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double ddot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 dcross(D3 a, D3 b) {
  return D3{a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// The prism of one (cluster, vertex): with q = p - g0 the weights are linear,
// w1 = q . (e2 x n) / |e1 x e2|, w2 = q . (n x e1) / |e1 x e2|, h = q . n, or
// the offset q itself, flag 1, for a degenerate triangle (|e1 x e2| <=
// 1e-6 |e1| |e2|).  The three vectors are FP64 results kept as double-word
// FP32 pairs (2^-48).
struct Prism {
  float3 g0;
  df a1[3], a2[3], n[3];
  bool flat;
};

__device__ __forceinline__ df df_from(double x) {
  const float hi = (float)x;
  return df{hi, (float)(x - (double)hi)};
}

__device__ __forceinline__ Prism make_prism(const float4 p0, const float4 p1, const float4 p2) {
  Prism pr;
  pr.g0 = make_float3(p0.x, p0.y, p0.z);
  const D3 g0 = d3(p0), e1 = dsub(d3(p1), g0), e2 = dsub(d3(p2), g0);
  const D3 n = dcross(e1, e2);
  const double nn = sqrt(ddot(n, n));
  const double scale = sqrt(ddot(e1, e1)) * sqrt(ddot(e2, e2));
  pr.flat = !(nn > 1e-6 * scale);
  const double in = 1.0 / nn;
  const D3 nh{n.x * in, n.y * in, n.z * in};
  const D3 u = dcross(e2, nh), v = dcross(nh, e1);
  pr.a1[0] = df_from(u.x * in); pr.a1[1] = df_from(u.y * in); pr.a1[2] = df_from(u.z * in);
  pr.a2[0] = df_from(v.x * in); pr.a2[1] = df_from(v.y * in); pr.a2[2] = df_from(v.z * in);
  pr.n[0] = df_from(nh.x); pr.n[1] = df_from(nh.y); pr.n[2] = df_from(nh.z);
  return pr;
}

__device__ __forceinline__ float df_dot3(const df q[3], const df a[3]) {
  return df_float(df_add(df_add(df_mul(q[0], a[0]), df_mul(q[1], a[1])), df_mul(q[2], a[2])));
}

// (w1, w2, h, 0) of the point g0 + q, or (q, 1) for a degenerate triangle.
__device__ __forceinline__ float4 prism_weights(const Prism& pr, const df q[3]) {
  if (pr.flat) return make_float4(df_float(q[0]), df_float(q[1]), df_float(q[2]), 1.f);
  return make_float4(df_dot3(q, pr.a1), df_dot3(q, pr.a2), df_dot3(q, pr.n), 0.f);
}

// x - y as an exact pair.
__device__ __forceinline__ df df_diff(float x, float y) {
  float e;
  const float s = two_sum(x, -y, e);
  return df{s, e};
}

__device__ __forceinline__ uint32_t eth_cluster(uint32_t e, const uint32_t* off, uint32_t L) {
  uint32_t k = 0;
  while (k + 1 < L && e >= off[k + 1]) ++k;
  return (e - off[k]) >> (2 * k);
}

struct Offs {
  uint32_t n_levels;
  uint32_t off[16];
};

// Skinning weights of one cluster: every member strand's vertices and every
// thick-hair cross-section's centre and four corners (c +- a e1, c +- b e2).
// A thread keeps one vertex index k, forms the prism of the cluster's three
// guides there once in FP64 (1 / 64 of the FP32 rate) and takes every point at
// k through it in double-word FP32.  Of 2.03M weights of six heads 4,223 are not
// the float nearest to the exact value (80-bit evaluation), against 4,401 with
// FP64 throughout, and the largest relative error is the same (5.95e-8, half an
// ulp).  Neighbouring threads read and write
// neighbouring vertices.  255 us for 100k strands x 65 and 22k thick hairs;
// FP64 prisms per point took 1.51 and 0.81 ms.  A cluster's points are shared
// out to gridDim.y blocks: few guides make few and large clusters (a build of
// 100k strands with 3, 8 and 32 guides 134, 24.5 and 7.1 ms with a block a
// cluster, 97, 20.2 and 6.2 shared out; 2.88 both ways with 256).
constexpr uint32_t kWeightBlock = 256;
constexpr uint32_t kWeightMembers = 64;   // strands a block takes, on average
constexpr uint32_t kWeightBlocks = 1216;  // eight an SM
__global__ void __launch_bounds__(kWeightBlock)
    k_prism_weights(const float4* __restrict__ verts, uint32_t S1,
                    const uint32_t* __restrict__ order, const uint32_t* __restrict__ cl_first,
                    const uint32_t* __restrict__ cl_tri, const int32_t* __restrict__ guides,
                    const float4* __restrict__ xsec, Offs lv, float4* w_strand, float4* w_eth) {
  const uint32_t c = blockIdx.x;
  const uint32_t lanes = max(1u, kWeightBlock / S1);  // points taken side by side
  const uint32_t step = lanes * gridDim.y;
  uint32_t ga, gb, gc;
  tri_of(cl_tri[c], ga, gb, gc);
  const size_t r0 = (size_t)guides[ga] * S1, r1 = (size_t)guides[gb] * S1,
               r2 = (size_t)guides[gc] * S1;
  const uint32_t m0 = cl_first[c], m1 = cl_first[c + 1];
  for (uint32_t t = threadIdx.x; t < lanes * S1; t += kWeightBlock) {
    const uint32_t k = t % S1, side = t / S1 + lanes * blockIdx.y;
    if (m0 + side >= m1 && (lv.n_levels == 0 || side >> (2 * (lv.n_levels - 1)))) continue;  // none left
    const Prism pr = make_prism(__ldg(verts + r0 + k), __ldg(verts + r1 + k), __ldg(verts + r2 + k));
    const float3 g0 = pr.g0;
    for (uint32_t m = m0 + side; m < m1; m += step) {
      const size_t idx = (size_t)__ldg(order + m) * S1 + k;
      const float4 p = __ldg(verts + idx);
      const df q[3] = {df_diff(p.x, g0.x), df_diff(p.y, g0.y), df_diff(p.z, g0.z)};
      w_strand[idx] = prism_weights(pr, q);
    }
    for (uint32_t l = 0; l < lv.n_levels; ++l) {
      const uint32_t sub = 1u << (2 * l), e0 = lv.off[l] + c * sub;
      for (uint32_t j = side; j < sub; j += step) {
        const size_t idx = (size_t)(e0 + j) * S1 + k;
        const float4 x = xsec[idx * 3], y = xsec[idx * 3 + 1], z = xsec[idx * 3 + 2];
        float4* o = w_eth + idx * 5;
        if (!(x.w > 0.f)) {  // empty thick hair
          for (int i = 0; i < 5; ++i) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          continue;
        }
        const df q[3] = {df_diff(x.x, g0.x), df_diff(x.y, g0.y), df_diff(x.z, g0.z)};
        o[0] = prism_weights(pr, q);
        const float ax[2] = {x.w, y.w}, dir[2][3] = {{y.x, y.y, y.z}, {z.x, z.y, z.z}};
        for (int i = 0; i < 2; ++i)
          for (int s = 0; s < 2; ++s) {
            const float a = s ? -ax[i] : ax[i];
            df p[3];
            for (int d = 0; d < 3; ++d) {
              float pe;
              const float ph = two_prod(a, dir[i][d], pe);
              p[d] = df_add(q[d], df{ph, pe});
            }
            o[1 + 2 * i + s] = prism_weights(pr, p);
          }
      }
    }
  }
}

// ---------------------------------------------------------------- skinning (FP32)

// New strand vertices from the guides' new vertices gv [G][S1] (radius kept).
__global__ void k_skin_strands(const float4* __restrict__ gv, uint32_t N, uint32_t S1,
                               const uint32_t* __restrict__ cluster_of,
                               const uint32_t* __restrict__ cl_tri,
                               const float4* __restrict__ w, float4* verts) {
  const uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (uint64_t)N * S1) return;
  const uint32_t i = (uint32_t)(idx / S1), k = (uint32_t)(idx % S1);
  uint32_t ga, gb, gc;
  tri_of(cl_tri[cluster_of[i]], ga, gb, gc);
  const float3 p = skin(w[idx], __ldg(gv + (size_t)ga * S1 + k), __ldg(gv + (size_t)gb * S1 + k),
                        __ldg(gv + (size_t)gc * S1 + k));
  verts[idx] = make_float4(p.x, p.y, p.z, verts[idx].w);
}

// New thick-hair cross-sections from the skinned centre and corners: a and
// e1 from the corners c +- a e1, b and e2 from c +- b e2.
__global__ void k_skin_eth(const float4* __restrict__ gv, uint32_t S1, uint32_t E, Offs lv,
                           const uint32_t* __restrict__ cl_tri, const float4* __restrict__ w,
                           float4* xsec) {
  const uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (uint64_t)E * S1) return;
  if (!(xsec[idx * 3].w > 0.f)) return;  // empty thick hair
  const uint32_t e = (uint32_t)(idx / S1), k = (uint32_t)(idx % S1);
  uint32_t ga, gb, gc;
  tri_of(cl_tri[eth_cluster(e, lv.off, lv.n_levels)], ga, gb, gc);
  const float4 g0 = __ldg(gv + (size_t)ga * S1 + k), g1 = __ldg(gv + (size_t)gb * S1 + k),
               g2 = __ldg(gv + (size_t)gc * S1 + k);
  float3 p[5];
  for (int j = 0; j < 5; ++j) p[j] = skin(w[idx * 5 + j], g0, g1, g2);
  const float3 u = make_float3(p[1].x - p[2].x, p[1].y - p[2].y, p[1].z - p[2].z);
  const float3 v = make_float3(p[3].x - p[4].x, p[3].y - p[4].y, p[3].z - p[4].z);
  const float lu = sqrtf(u.x * u.x + u.y * u.y + u.z * u.z);
  const float lv_ = sqrtf(v.x * v.x + v.y * v.y + v.z * v.z);
  const float iu = lu > 0.f ? 1.f / lu : 0.f, iv = lv_ > 0.f ? 1.f / lv_ : 0.f;
  xsec[idx * 3] = make_float4(p[0].x, p[0].y, p[0].z, 0.5f * lu);
  xsec[idx * 3 + 1] = make_float4(u.x * iu, u.y * iu, u.z * iu, 0.5f * lv_);
  xsec[idx * 3 + 2] = make_float4(v.x * iv, v.y * iv, v.z * iv, 0.f);
}

// Assignments and nearest guides of 32-strand tiles, with the tile in shared
// memory where it fits.
template <typename K>
hr_status allow_tile(hr_ctx* ctx, K kernel) {
  HR_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)tile_bytes(kTileMaxVerts)));
  return HR_OK;
}

unsigned blocks_for(uint64_t n, unsigned b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

namespace {

// The skinning state of a guided hierarchy (not the guides themselves).
void drop_weights(hr_ctx* ctx, hr_asset* a) {
  const size_t S1 = a->S + 1;
  if (a->cl_tri) dfree(ctx, a->cl_tri, (size_t)a->guided_C * 4), a->cl_tri = nullptr;
  if (a->w_strand) dfree(ctx, a->w_strand, (size_t)a->N * S1 * sizeof(float4)), a->w_strand = nullptr;
  if (a->w_eth) dfree(ctx, a->w_eth, (size_t)a->guided_E * S1 * 5 * sizeof(float4)), a->w_eth = nullptr;
  a->guided_C = a->guided_E = 0;
}

hr_status guided_build(hr_ctx* ctx, hr_asset* a, uint32_t G, uint32_t iters, uint32_t max_levels) {
  cudaStream_t st = ctx_stream(ctx);
  const uint32_t N = a->N, S1 = a->S + 1;
  // scratch: Morton order and codes, keys / values and their temporaries,
  // the assignment, counts and starts, centroids, the medoids' sums
  uint32_t *order, *codes, *kk, *vv, *k2, *v2, *assign, *start, *dC, *nb;
  float4* cent;
  HR_TRY(scratch(ctx, 52, (size_t)N * 4, (void**)&order));
  HR_TRY(scratch(ctx, 53, (size_t)N * 4, (void**)&codes));
  HR_TRY(scratch(ctx, 54, (size_t)N * 4, (void**)&kk));
  HR_TRY(scratch(ctx, 55, (size_t)N * 4, (void**)&vv));
  HR_TRY(scratch(ctx, 56, (size_t)N * 4, (void**)&k2));
  HR_TRY(scratch(ctx, 57, (size_t)N * 4, (void**)&v2));
  HR_TRY(scratch(ctx, 58, (size_t)N * 4, (void**)&assign));
  HR_TRY(scratch(ctx, 59, ((size_t)std::max(G, N) + 2) * 4, (void**)&start));
  HR_TRY(scratch(ctx, 60, (size_t)G * S1 * sizeof(float4) + 16, (void**)&cent));
  HR_TRY(scratch(ctx, 61, 16, (void**)&dC));
  HR_TRY(scratch(ctx, 15, (size_t)G * 3 * 4, (void**)&nb));
  const uint64_t n_sum = (uint64_t)G * S1 * 3;
  MedoidWork mw{};
  HR_TRY(scratch(ctx, 16, (n_sum + 2 * (size_t)G) * 8 + ((size_t)2 * G + 4 + 2 * (size_t)N) * 4,
                 (void**)&mw.csum));
  mw.W = mw.csum + n_sum;
  mw.best = reinterpret_cast<unsigned long long*>(mw.W + G);
  mw.tmin = reinterpret_cast<uint32_t*>(mw.best + G);
  mw.vmax = mw.tmin + G;
  mw.n_cand = mw.vmax + G;
  mw.T = reinterpret_cast<float*>(mw.n_cand + 4);
  mw.cand = reinterpret_cast<uint32_t*>(mw.T + N);
  int32_t* guides = a->guides;
  HR_TRY(root_morton_order(ctx, a, codes, order, st));
  int bits = 1;
  while ((1u << bits) < G) ++bits;
  const bool tile = S1 <= kTileMaxVerts;
  const size_t smem = tile ? tile_bytes(S1) : 0;
  const unsigned tiles = blocks_for(N, 32);
  if (tile) {
    HR_TRY(allow_tile(ctx, k_assign<true>));
    HR_TRY(allow_tile(ctx, k_nearest3<true>));
  }
  bool have_prev = false;
  auto assign_all = [&]() -> hr_status {
    (tile ? k_assign<true> : k_assign<false>)<<<tiles, 32 * kTileWarps, smem, st>>>(
        a->verts, N, S1, cent, G, order, have_prev, assign);
    HR_LAUNCHED(ctx);
    have_prev = true;
    return HR_OK;
  };
  // the members of every cluster in ascending strand id (key, id), and the starts
  uint32_t *mkey = nullptr, *mid = nullptr;
  auto members = [&]() -> hr_status {
    k_iota_copy<<<blocks_for(N, 256), 256, 0, st>>>(assign, N, kk, vv);
    HR_LAUNCHED(ctx);
    HR_TRY(radix_sort_pairs(ctx, kk, vv, k2, v2, N, bits, st, kLookbackPolls, &mkey, &mid));
    k_key_starts<<<blocks_for(G + 1, 128), 128, 0, st>>>(mkey, N, G, start);
    HR_LAUNCHED(ctx);
    return HR_OK;
  };
  k_seed<<<G, 64, 0, st>>>(a->verts, S1, order, N, G, cent);
  HR_LAUNCHED(ctx);
  for (uint32_t it = 0; it < iters; ++it) {
    HR_TRY(assign_all());
    HR_TRY(members());
    k_update<<<dim3(G, blocks_for(S1 * 3, kUpdateBlock)), kUpdateBlock, 0, st>>>(a->verts, S1, start,
                                                                                 mid, cent);
    HR_LAUNCHED(ctx);
  }
  HR_TRY(assign_all());
  HR_TRY(members());
  // medoids
  k_medoid_init<<<blocks_for(std::max<uint64_t>(n_sum, G), 256), 256, 0, st>>>(mw, G, n_sum);
  HR_LAUNCHED(ctx);
  k_member_sums<<<blocks_for(N, kSumRanks), 256, 0, st>>>(a->verts, N, S1, mkey, mid, mw.csum);
  HR_LAUNCHED(ctx);
  k_means<<<blocks_for(n_sum, 256), 256, 0, st>>>(mw.csum, start, G, S1);
  HR_LAUNCHED(ctx);
  k_member_spread<<<blocks_for(N, 8), 256, 0, st>>>(a->verts, N, S1, mkey, mid, mw);
  HR_LAUNCHED(ctx);
  k_medoid_candidates<<<blocks_for(N, 256), 256, 0, st>>>(mkey, N, S1, start, mw);
  HR_LAUNCHED(ctx);
  k_medoid_sums<<<std::min(N, 1216u), 256, 0, st>>>(a->verts, S1, mkey, start, mid, mw);
  HR_LAUNCHED(ctx);
  k_medoid_write<<<blocks_for(G, 128), 128, 0, st>>>(mw.best, start, G, guides);
  HR_LAUNCHED(ctx);
  // at least three guides
  std::vector<int32_t> gh(G);
  HR_CUDA(ctx, cudaMemcpyAsync(gh.data(), guides, (size_t)G * 4, cudaMemcpyDeviceToHost, st));
  HR_CUDA(ctx, cudaStreamSynchronize(st));
  uint32_t n_valid = 0;
  for (int32_t g : gh) n_valid += g >= 0;
  if (n_valid < 3) return set_error(ctx, HR_EINVAL, "fewer than three non-empty guide clusters");
  // three nearest guides of every strand (Morton order), then the strands by
  // (key, Morton code, id): a stable sort of the keys of the Morton order
  k_guide_neighbours<<<G, 128, 0, st>>>(a->verts, S1, guides, G, nb);
  HR_LAUNCHED(ctx);
  (tile ? k_nearest3<true> : k_nearest3<false>)<<<tiles, 32 * kTileWarps, smem, st>>>(
      a->verts, N, S1, guides, G, nb, assign, order, kk);
  HR_LAUNCHED(ctx);
  HR_CUDA(ctx, cudaMemcpyAsync(vv, order, (size_t)N * 4, cudaMemcpyDeviceToDevice, st));
  HR_TRY(radix_sort_pairs(ctx, kk, vv, k2, v2, N, 30, st));
  // cluster starts where the key changes
  k_head_flags<<<blocks_for(N, 256), 256, 0, st>>>(kk, N, assign);
  HR_LAUNCHED(ctx);
  HR_TRY(scan_u32(ctx, assign, N, st));
  uint32_t* cl_tri_tmp = k2;  // [C <= N]
  k_starts<<<blocks_for(N, 256), 256, 0, st>>>(kk, assign, N, start, cl_tri_tmp, dC);
  HR_LAUNCHED(ctx);
  uint32_t C = 0;
  HR_CUDA(ctx, cudaMemcpyAsync(&C, dC, 4, cudaMemcpyDeviceToHost, st));
  HR_CUDA(ctx, cudaStreamSynchronize(st));
  HR_TRY(build_hierarchy_from(ctx, a, C, max_levels, vv, start));
  // the hierarchy's arrays are set: the guide state for skinning, in the
  // arrays of an earlier build where their sizes stay
  if (a->guided_C != C || a->guided_E != a->E) drop_weights(ctx, a);
  if (!a->cl_tri) HR_TRY(dalloc(ctx, (void**)&a->cl_tri, (size_t)C * 4, "cluster guides"));
  a->guided_C = C;
  HR_CUDA(ctx, cudaMemcpyAsync(a->cl_tri, cl_tri_tmp, (size_t)C * 4, cudaMemcpyDeviceToDevice, st));
  if (!a->w_strand)
    HR_TRY(dalloc(ctx, (void**)&a->w_strand, (size_t)N * S1 * sizeof(float4), "strand weights"));
  if (a->E && !a->w_eth) {
    HR_TRY(dalloc(ctx, (void**)&a->w_eth, (size_t)a->E * S1 * 5 * sizeof(float4), "thick-hair weights"));
    a->guided_E = a->E;
  }
  Offs lv{};
  lv.n_levels = a->n_levels;
  for (uint32_t k = 0; k <= a->n_levels && k < 16; ++k) lv.off[k] = a->eth_offset[k];
  const uint32_t parts = std::min(
      65535u, std::max(blocks_for(N / C, kWeightMembers), blocks_for(kWeightBlocks, C)));
  k_prism_weights<<<dim3(C, parts), kWeightBlock, 0, st>>>(a->verts, S1, a->order, a->cl_first,
                                                           a->cl_tri, guides, a->xsec, lv,
                                                           a->w_strand, a->w_eth);
  HR_LAUNCHED(ctx);
  return HR_OK;
}

}  // namespace

void drop_guides(hr_ctx* ctx, hr_asset* a) {
  drop_weights(ctx, a);
  if (a->guides) dfree(ctx, a->guides, (size_t)a->G * 4);
  a->guides = nullptr;
  a->G = 0;
}

hr_status build_guided_hierarchy(hr_ctx* ctx, hr_asset* a, uint32_t G, uint32_t iters,
                                 uint32_t max_levels) {
  const uint32_t N = a->N;
  if (G < 3 || G > kMaxGuides || G > N)
    return set_error(ctx, HR_EINVAL, "n_guides must be in 3..min(1024, n_strands)");
  if (a->G != G) {
    drop_guides(ctx, a);
    HR_TRY(dalloc(ctx, (void**)&a->guides, (size_t)G * 4, "guides"));
    a->G = G;
  }
  const hr_status s = guided_build(ctx, a, G, iters, max_levels);
  if (s != HR_OK) drop_weights(ctx, a);  // no skinning with an unfinished hierarchy
  return s;
}

hr_status skin_asset(hr_ctx* ctx, hr_asset* a, const float4* gv_dev) {
  cudaStream_t st = ctx_stream(ctx);
  const uint32_t N = a->N, S1 = a->S + 1;
  if (S1 <= kUpdateMaxVerts) {
    HR_TRY(skin_strands(ctx, a, gv_dev));
  } else {  // strands too long for a block's shared memory
    k_skin_strands<<<blocks_for((uint64_t)N * S1, 256), 256, 0, st>>>(gv_dev, N, S1, a->cluster_of,
                                                                     a->cl_tri, a->w_strand, a->verts);
    HR_LAUNCHED(ctx);
    HR_TRY(refresh_strand_prims(ctx, a));
    HR_TRY(clear_eth_bounds(ctx, a));
  }
  if (a->E) {
    Offs lv{};
    lv.n_levels = a->n_levels;
    for (uint32_t k = 0; k <= a->n_levels && k < 16; ++k) lv.off[k] = a->eth_offset[k];
    k_skin_eth<<<blocks_for((uint64_t)a->E * S1, 256), 256, 0, st>>>(gv_dev, S1, a->E, lv, a->cl_tri,
                                                                    a->w_eth, a->xsec);
    HR_LAUNCHED(ctx);
    HR_TRY(moved_eth_records(ctx, a));
  }
  a->bvh.valid = 0;
  return HR_OK;
}

}  // namespace hr
