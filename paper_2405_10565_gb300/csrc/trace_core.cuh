// Device code of the hot path: camera rays, BVH traversal, ray versus
// elliptic-cylinder tests, k-buffer, scattering models and compositing.
//
//  * Camera: sample sid = pixel * spp + s; sub-pixel position from SplitMix64
//    outputs 2 sid and 2 sid + 1 of the frame seed (top 24 bits each).
//  * Traversal: stack-based over the binary LBVH whose nodes hold both
//    children's boxes (one node fetch tests two boxes); nearer child
//    first.  The search interval shrinks to the K-th nearest hit and to the
//    nearest opaque (strand) hit: nothing behind an opaque hit can contribute.
//  * Intersection: the record maps the ray into the cylinder's unit frame;
//    the quadratic is solved about the point of closest approach and the root
//    kept is the nearest one with w in [0, 1] (open cylinder).
//  * Shading: f_single (Eq. 1) for strands, f_ours (Eq. 5-13) for thick
//    hairs, per light; forward/backward single-fibre albedos from the
//    longitudinal-integral table.
//  * Compositing: front to back over the k-buffer sorted by (t, id).
#pragma once

#include "common.cuh"
#include "dword.cuh"

namespace hr {
namespace tr {

#define kInf __int_as_float(0x7f800000)
constexpr int kStack = 64;
// Blocks an SM of the tracing kernels (72 registers; the node visits and leaf
// tests do not spill, the shading does a little).  With 5, 6, 7 and 8: the far
// view of the full head 1.31, 1.31, 1.31, 1.45 ms a call, its close view 4.05,
// 3.85, 3.65, 3.60, the 4K frame of straight hair 10.5, 10.0, 9.6, 9.6, the
// curled clusters 1.47, 1.44, 1.40, 1.43 (the last blocks cost L1: shared
// memory, stacks and more rays' records).
constexpr int kTraceBlocks = 7;

__device__ __forceinline__ uint64_t splitmix_out(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float3 a, float s) { return f3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float clampf(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }

__device__ __forceinline__ float3 hit_point(const float3 o, const float3 d, float t) { return o + d * t; }

// ------------------------------------------------------------------ geometry

// ------------------------------------------------------------------ precision
//
// The hit decisions are taken in FP32 wherever FP32 rounding cannot change
// them, and precisely otherwise.
//  * Every camera ray is built in double-word FP32 (the oracle's FP64
//    construction to about 2^-44) and re-based at its entry into the scene's
//    bounding box: the FP32 ray (o', d) starts next to the hair, and depths
//    are kept relative to that origin.  FP32 rounding then
//    moves a hit by ~2^-24 of the scene's size instead of ~2^-24 of the
//    camera distance.
//  * intersect32 bounds the rounding of its affine rows and of the roots.  A
//    test within that bound of the cylinder's outline or of an end of the
//    segment, a hit whose depth bound could reorder it against another hit or
//    the search cut, or whose bound is wide, is decided by refine: the
//    double-word ray re-based near the hit relative to the segment's start
//    point, and the quadratic solved about that point.  Kept FP32 hits whose
//    order against a precise one their bounds leave open are refined too.
// Far cameras and thin fibres (4K views of 1e-3 strands ten units away)
// otherwise turn up FP32 rounding errors of a few 1e-7 in position, enough
// to swap two strands at nearly equal depth or drop a hit at the very edge of
// a fibre.

constexpr int kMiss = 0, kHit = 1, kBorder = 2;
constexpr float kEps32 = 5.9604645e-8f;   // FP32 unit roundoff, 2^-24
constexpr float kBoundK = 6.f;            // rounding steps per affine row, with margin
// Relative depth (of the absolute depth) that widens the box cull, and above
// which an FP32 depth bound sends the hit to refine.
constexpr float kTieRel = 1.52587890625e-05f;  // 2^-16

struct RayKey {  // what rebuilds the ray precisely: the sample id and the re-basing offset
  uint64_t sid;
  float s_off;  // o' = o + s_off v, v the unnormalised direction (|v| >= 1)
};

// Ray against the open elliptic cylinder of one record, in FP32, with a
// bound on the rounding of each decision.  kMiss when the ray misses by more
// than the bound; kBorder when the rounding could change the outcome; else
// kHit with the nearest root t in (0, tmax] (axial coordinate in [0, 1]),
// and its error bound terr.
// r0, r1: the record's rows u and v; M = |o.x| + |o.y| + |o.z| of the ray.
__device__ __forceinline__ int intersect32(const FrameArgs& fa, const uint32_t id, const float4 r0,
                                           const float4 r1, const float3 o, const float3 d,
                                           const float M, const float tmax, float& t_hit, float& terr) {
  const float u0 = fmaf(r0.x, o.x, fmaf(r0.y, o.y, fmaf(r0.z, o.z, r0.w)));
  const float v0 = fmaf(r1.x, o.x, fmaf(r1.y, o.y, fmaf(r1.z, o.z, r1.w)));
  const float du = fmaf(r0.x, d.x, fmaf(r0.y, d.y, r0.z * d.z));
  const float dv = fmaf(r1.x, d.x, fmaf(r1.y, d.y, r1.z * d.z));
  const float A = fmaf(du, du, dv * dv);
  if (!(A > 0.f)) return kMiss;
  const float inv = 1.0f / A;
  const float tc = -fmaf(u0, du, v0 * dv) * inv;
  const float uc = fmaf(tc, du, u0), vc = fmaf(tc, dv, v0);
  const float h2 = fmaf(uc, uc, vc * vc);
  // rounding bound of (uc, vc): the rows' intermediate terms reach |r| (|o| + |tc|)
  const float mag = M + fabsf(tc);
  const float eu = kBoundK * kEps32 *
                   fmaf(fabsf(r0.x) + fabsf(r0.y) + fabsf(r0.z), mag, fabsf(r0.w));
  const float ev = kBoundK * kEps32 *
                   fmaf(fabsf(r1.x) + fabsf(r1.y) + fabsf(r1.z), mag, fabsf(r1.w));
  const float e = eu + ev;
  const float dh = e * (2.f + e);
  if (h2 > 1.f + dh) return kMiss;
  bool border = h2 >= 1.f - dh;  // near the outline
  const float g = fmaxf(1.f - h2, 0.f);
  const float half = sqrtf(g * inv);
  const float tm = tc - half, tp = tc + half;
  // depth bound: the (u, v) error over |(du, dv)|, the root's slope (near
  // the outline at most sqrt(dh / A)), and the rounding of t itself
  const float magt = mag + half;
  const float eroot = border ? sqrtf(dh * inv) : dh * half * (0.5f / g);
  terr = fmaf(e, sqrtf(inv), fmaf(4.f * kEps32, magt, eroot));
  if (tp + terr <= 0.f || tm - terr > tmax) return kMiss;
  const float4 r2 = __ldg(fa.prim_wa + 2 * (size_t)id);
  const float w0 = fmaf(r2.x, o.x, fmaf(r2.y, o.y, fmaf(r2.z, o.z, r2.w)));
  const float dw = fmaf(r2.x, d.x, fmaf(r2.y, d.y, r2.z * d.z));
  // axial coordinate of each root, and its error bound (the row's rounding
  // and the root's depth error times the axial rate)
  const float ew = fmaf(kBoundK * kEps32,
                        fmaf(fabsf(r2.x) + fabsf(r2.y) + fabsf(r2.z), magt, fabsf(r2.w)),
                        fabsf(dw) * terr);
  const float wm = fmaf(tm, dw, w0), wp = fmaf(tp, dw, w0);
  // each root: certainly in range, possibly in range, or certainly not
  const bool m_in = tm > terr && wm >= ew && wm <= 1.f - ew;
  const bool m_may = tm > -terr && wm >= -ew && wm <= 1.f + ew;
  const bool p_in = tp > terr && wp >= ew && wp <= 1.f - ew;
  const bool p_may = tp > -terr && wp >= -ew && wp <= 1.f + ew;
  float t;
  if (m_in) {
    t = tm;
  } else if (m_may) {
    t = fmaxf(tm, 0.f);
    border = true;
  } else if (p_in) {
    t = tp;
  } else if (p_may) {
    t = fmaxf(tp, 0.f);
    border = true;
  } else {
    return kMiss;
  }
  if (t - terr > tmax) return kMiss;
  t_hit = t;
  return border ? kBorder : kHit;
}

// Camera ray of a sample in double-word FP32, the oracle's construction to
// about 2^-44: sub-pixel offset from the top 24 bits of SplitMix64 outputs
// 2 sid and 2 sid + 1, image-plane offset ((x + jx) - W / 2,
// H / 2 - (y + jy)) / pix (exact pairs times the double-word 1 / pix);
// perspective
// rays leave the eye along v = (fwd + sx right) + sy up, orthographic ones
// leave (eye + sx right) + sy up along fwd.  v is left unnormalised: the
// ray's point at parameter s is o + s v.
struct PreciseRay {
  df o[3], v[3];
};
static __device__ void camera_ray_dw(const LaunchCam& c, uint64_t seed, uint32_t spp, uint64_t sid,
                                     PreciseRay& r) {
  const float jx = (float)(uint32_t)(splitmix_out(seed, 2 * sid) >> 40) * (1.0f / 16777216.0f);
  const float jy = (float)(uint32_t)(splitmix_out(seed, 2 * sid + 1) >> 40) * (1.0f / 16777216.0f);
  uint32_t px, py;
  if (sid < (1ull << 32)) {
    const uint32_t pixel = (uint32_t)sid / spp;
    px = pixel % (uint32_t)c.W;
    py = pixel / (uint32_t)c.W;
  } else {
    const uint64_t pixel = sid / spp;
    px = (uint32_t)(pixel % (uint64_t)c.W);
    py = (uint32_t)(pixel / (uint64_t)c.W);
  }
  const float x = (float)px, y = (float)py;
  float ex, ey;
  const float ax = two_sum(__fsub_rn(x, 0.5f * (float)c.W), jx, ex);
  const float ay = two_sum(__fsub_rn(0.5f * (float)c.H, y), -jy, ey);
  const df ipix{c.ipix_hi, c.ipix_lo};
  const df sx = df_mul(df{ax, ex}, ipix), sy = df_mul(df{ay, ey}, ipix);
  const float E[3] = {c.eye.x, c.eye.y, c.eye.z}, R[3] = {c.right.x, c.right.y, c.right.z};
  const float U[3] = {c.up.x, c.up.y, c.up.z}, F[3] = {c.fwd.x, c.fwd.y, c.fwd.z};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const df w = df_add(df_add(df_mul(sx, R[i]), c.kind == 1 ? F[i] : E[i]), df_mul(sy, U[i]));
    if (c.kind == 1) {
      r.o[i] = df{E[i], 0.f};
      r.v[i] = w;
    } else {
      r.o[i] = w;
      r.v[i] = df{F[i], 0.f};
    }
  }
}

// |v|^2 of a double-word vector and its square root in double-word (one
// Newton correction from the exact FMA residual).
__device__ __forceinline__ df df_norm2(const df v[3]) {
  return df_add(df_add(df_mul(v[0], v[0]), df_mul(v[1], v[1])), df_mul(v[2], v[2]));
}
__device__ __forceinline__ df df_sqrt(df a) {
  const float r = __fsqrt_rn(a.hi);
  return df_fast(r, __fdiv_rn(__fadd_rn(fmaf(-r, r, a.hi), a.lo), 2.f * r));
}

// Exact bounds of the BVH's leaves.
__device__ __forceinline__ void root_box(const FrameArgs& fa, float3& lo, float3& hi) {
  const uint32_t* b = reinterpret_cast<const uint32_t*>(fa.frame + 3);
  lo = f3(from_ordered(__ldg(b)), from_ordered(__ldg(b + 1)), from_ordered(__ldg(b + 2)));
  hi = f3(from_ordered(__ldg(b + 3)), from_ordered(__ldg(b + 4)), from_ordered(__ldg(b + 5)));
}

// The FP32 ray of a sample: the direction normalised in FP32 (correctly
// rounded steps, so |d| = 1 within a few ulps), and the origin moved to a
// little before the ray's entry into the scene's bounding box (the root
// node's two boxes), o' = o + s_off v, formed in double-word before rounding.
// Hits are at depth t' past o' along d; no primitive lies before the entry,
// so t' > 0 for every hit.
__device__ __forceinline__ void primary_ray(const FrameArgs& fa, uint64_t sid, float3& o,
                                            float3& d, RayKey& rk) {
  PreciseRay ry;
  camera_ray_dw(fa.cam, fa.seed, fa.spp, sid, ry);
  const float vx = ry.v[0].hi, vy = ry.v[1].hi, vz = ry.v[2].hi;
  const float il = __frcp_rn(__fsqrt_rn(fmaf(vx, vx, fmaf(vy, vy, __fmul_rn(vz, vz)))));
  d = f3(__fmul_rn(vx, il), __fmul_rn(vy, il), __fmul_rn(vz, il));
  float s_off = 0.f;
  if (fa.n_prims >= 2) {
    float3 blo, bhi;
    root_box(fa, blo, bhi);
    const float3 oo = f3(ry.o[0].hi, ry.o[1].hi, ry.o[2].hi);
    const float3 inv = f3(1.0f / (fabsf(d.x) > 1e-12f ? d.x : copysignf(1e-12f, d.x)),
                          1.0f / (fabsf(d.y) > 1e-12f ? d.y : copysignf(1e-12f, d.y)),
                          1.0f / (fabsf(d.z) > 1e-12f ? d.z : copysignf(1e-12f, d.z)));
    const float lx = (blo.x - oo.x) * inv.x, hx = (bhi.x - oo.x) * inv.x;
    const float ly = (blo.y - oo.y) * inv.y, hy = (bhi.y - oo.y) * inv.y;
    const float lz = (blo.z - oo.z) * inv.z, hz = (bhi.z - oo.z) * inv.z;
    const float t0 = fmaxf(fmaxf(fminf(lx, hx), fminf(ly, hy)), fminf(lz, hz));
    const float t1 = fminf(fminf(fmaxf(lx, hx), fmaxf(ly, hy)), fmaxf(lz, hz));
    // 2^-10 before the FP32 entry: far more than the slab test's rounding
    if (t0 > 0.f && t0 <= t1) s_off = t0 * (1.f - 9.765625e-4f) * il;
  }
  rk = RayKey{sid, s_off};
  o = f3(df_float(df_add(ry.o[0], df_mul(ry.v[0], s_off))),
         df_float(df_add(ry.o[1], df_mul(ry.v[1], s_off))),
         df_float(df_add(ry.o[2], df_mul(ry.v[2], s_off))));
}

// The precise decision of one test, for hits the FP32 test cannot order or
// classify.  The ray is built in double-word FP32 and re-based at its point
// s0 v (s0 from the FP32 depth estimate) relative to the segment's start
// point c0 (a strand vertex or a thick-hair cross-section centre): that point
// lies within about a segment length of c0, so rounding it to FP32 costs
// ~2^-24 of a segment length instead of ~2^-24 of the camera distance.  The
// cylinder (the record's FP32 linear rows, through c0) is then solved about
// it in FP32: the nearest root of o + s v with s > 0 and axial coordinate in
// [0, 1].  t_est and the result are depths past the re-based origin
// o' = o + s_off v; the result is a normalised pair t' = t_hi + t_lo.  About 300 FP32 operations, against ~200 FP64 operations (1/64 of
// the FP32 rate on this GPU) for the same test in FP64.
static __device__ __noinline__ bool refine(const FrameArgs& fa, const RayKey& rk, uint32_t id,
                                           float t_est, float& t_hi, float& t_lo) {
  PreciseRay ry;
  camera_ray_dw(fa.cam, fa.seed, fa.spp, rk.sid, ry);
  const float4 r0 = __ldg(fa.prim_uv + 2 * (size_t)id), r1 = __ldg(fa.prim_uv + 2 * (size_t)id + 1),
               r2 = __ldg(fa.prim_wa + 2 * (size_t)id);
  const uint32_t S = fa.S, NS = fa.N * fa.S;
  float4 c0;
  if (id < NS)
    c0 = __ldg(fa.verts + (size_t)(id / S) * (S + 1) + id % S);
  else
    c0 = __ldg(fa.xsec + ((size_t)((id - NS) / S) * (S + 1) + (id - NS) % S) * 3);
  const float vx = ry.v[0].hi, vy = ry.v[1].hi, vz = ry.v[2].hi;
  const df L = df_sqrt(df_norm2(ry.v));  // depth along the unit direction = s |v|
  // re-base at o + (s_off + s0) v, s0 the FP32 depth estimate past o' in units of v
  const float s0 = t_est / L.hi;
  float sb;
  const float sa = two_sum(rk.s_off, s0, sb);
  const df sp0{sa, sb};
  const float C0[3] = {c0.x, c0.y, c0.z};
  float p[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) p[i] = df_float(df_add(df_add(ry.o[i], -C0[i]), df_mul(ry.v[i], sp0)));
  const float u0 = fmaf(r0.x, p[0], fmaf(r0.y, p[1], __fmul_rn(r0.z, p[2])));
  const float v0 = fmaf(r1.x, p[0], fmaf(r1.y, p[1], __fmul_rn(r1.z, p[2])));
  const float w0 = fmaf(r2.x, p[0], fmaf(r2.y, p[1], __fmul_rn(r2.z, p[2])));
  const float du = fmaf(r0.x, vx, fmaf(r0.y, vy, __fmul_rn(r0.z, vz)));
  const float dv = fmaf(r1.x, vx, fmaf(r1.y, vy, __fmul_rn(r1.z, vz)));
  const float dw = fmaf(r2.x, vx, fmaf(r2.y, vy, __fmul_rn(r2.z, vz)));
  const float A = fmaf(du, du, __fmul_rn(dv, dv));
  if (!(A > 0.f)) return false;
  const float inv = 1.0f / A;
  const float sc = __fmul_rn(-fmaf(u0, du, __fmul_rn(v0, dv)), inv);
  const float uc = fmaf(sc, du, u0), vc = fmaf(sc, dv, v0);
  const float h2 = fmaf(uc, uc, __fmul_rn(vc, vc));
  if (h2 > 1.f) return false;
  const float half = sqrtf(__fmul_rn(__fsub_rn(1.f, h2), inv));
  const float sm = __fsub_rn(sc, half), sp = __fadd_rn(sc, half);
  const float wm = fmaf(sm, dw, w0), wp = fmaf(sp, dw, w0);
  float s;
  // in front of the eye: s_off + s0 + s > 0 (s_off is 0 unless the eye is
  // outside the scene box, and then every root is far in front of it)
  if (__fadd_rn(sa, sm) > 0.f && wm >= 0.f && wm <= 1.f)
    s = sm;
  else if (__fadd_rn(sa, sp) > 0.f && wp >= 0.f && wp <= 1.f)
    s = sp;
  else
    return false;
  float e;
  const float th = two_sum(s0, s, e);
  const df t = df_mul(df_fast(th, e), L);
  t_hi = t.hi;
  t_lo = t.lo;
  return true;
}

// The K nearest hits: depth and entry word.  The entry word holds the
// global primitive id (which also addresses the primitive's records; a thick
// hair's chord is recomputed from them when it is shaded) and two flags:
// kExact when the depth was decided precisely and kOpaque for a strand hit.
// The depth is t + tr, with tr = 0 until it is decided precisely; entries order
// by (depth, id).  Shading takes t.  So that t does not depend on the order of the
// tests (frames repeat bit for bit whichever kernel finishes a ray), it is the
// precise depth only where the hit needs one for its own sake, whatever else the
// ray hits; where only the order against another hit did, t stays the FP32
// depth and tr takes the rest.  (A light path starts at t + tr: it can cross a
// hair or miss it by less than FP32's rounding, and frames with shadow rays put
// no ray aside.)
constexpr uint32_t kIdMask = 0x3fffffffu, kOpaque = 0x40000000u, kExact = 0x80000000u;
constexpr uint32_t kNoEntry = kIdMask;  // an empty slot (t = inf)
// The ray and its hits live in shared memory, a column per thread (no bank
// conflicts), or one per warp where the warp works on one ray: the node visits
// need only the slab constants in registers, and the shading loops over the
// entries instead of being unrolled over them.  With them in registers the
// frame kernel needed 128 registers (16 warps an SM) and K copies of the
// shading code.
template <int KMAX, int COLS>
struct RayMem {
  float o[3][COLS], d[3][COLS];  // the FP32 ray
  float M[COLS];                 // |o.x| + |o.y| + |o.z|
  float s_off[COLS];             // RayKey
  uint32_t sid[2][COLS];
  float t[KMAX][COLS], tr[KMAX][COLS];
  uint32_t id[KMAX][COLS];
};

// The k-buffer's depth.  kmax_for gives depths 1 and 2 kernels of their own, so
// there it is known and the loops over the entries unroll (129 strands with
// shadow rays at K = 2: 78.5 -> 69 us a call; a 968 x 666 head at K = 2: 568 ->
// 555).
template <int KMAX>
__device__ __forceinline__ uint32_t kbuf_depth(const FrameArgs& fa) {
  return KMAX <= 2 ? (uint32_t)KMAX : fa.k;
}

template <int KMAX, int COLS>
__device__ __forceinline__ void ray_store(RayMem<KMAX, COLS>& rm, uint32_t c, const float3 o,
                                          const float3 d, const RayKey& rk) {
  rm.o[0][c] = o.x; rm.o[1][c] = o.y; rm.o[2][c] = o.z;
  rm.d[0][c] = d.x; rm.d[1][c] = d.y; rm.d[2][c] = d.z;
  rm.M[c] = fabsf(o.x) + fabsf(o.y) + fabsf(o.z);
  rm.s_off[c] = rk.s_off;
  rm.sid[0][c] = (uint32_t)rk.sid;
  rm.sid[1][c] = (uint32_t)(rk.sid >> 32);
}
template <int KMAX, int COLS>
__device__ __forceinline__ float3 ray_o(const RayMem<KMAX, COLS>& rm, uint32_t c) {
  return f3(rm.o[0][c], rm.o[1][c], rm.o[2][c]);
}
template <int KMAX, int COLS>
__device__ __forceinline__ float3 ray_d(const RayMem<KMAX, COLS>& rm, uint32_t c) {
  return f3(rm.d[0][c], rm.d[1][c], rm.d[2][c]);
}

__device__ __forceinline__ bool key_less(float t, float tr, uint32_t id, float t2, float tr2,
                                         uint32_t id2) {
  // t - t2 is exact where tr can matter; both infinite: not less
  const float d = __fsub_rn(t, t2), e = __fsub_rn(tr2, tr);
  return d < e || (d == e && (id & kIdMask) < (id2 & kIdMask));
}

// The entry (t, tr, id) into the sorted places 0 .. j, the last one's old
// entry falling off.
template <int KMAX, int COLS>
__device__ __forceinline__ void kbuf_place(RayMem<KMAX, COLS>& rm, uint32_t c, int j, float t, float tr,
                                           uint32_t id) {
  for (; j > 0 && key_less(t, tr, id, rm.t[j - 1][c], rm.tr[j - 1][c], rm.id[j - 1][c]); --j) {
    rm.t[j][c] = rm.t[j - 1][c];
    rm.tr[j][c] = rm.tr[j - 1][c];
    rm.id[j][c] = rm.id[j - 1][c];
  }
  rm.t[j][c] = t;
  rm.tr[j][c] = tr;
  rm.id[j][c] = id;
}

// The search cut: the depth of the k-th entry, or of the first opaque entry
// when it comes earlier (nothing behind an opaque hit is composited).
template <int KMAX, int COLS>
__device__ __forceinline__ float kbuf_cut(const RayMem<KMAX, COLS>& rm, uint32_t c, const uint32_t k) {
  uint32_t j = 0;
  while (j + 1 < k && !(rm.id[j][c] & kOpaque)) ++j;
  return rm.t[j][c];
}

struct Counts {
  uint32_t nodes, tests, sshade, eshade, hits, rays, precise_tests, precise_entries;
  uint32_t steps;  // node visits plus primitive tests, counted by the frame kernel (tile schedule)
};

// Test primitive `id` (a leaf names its global primitive id) and keep it in
// the k-buffer when it is among the K nearest before the nearest opaque
// (strand) hit.  An FP32 hit is kept as it is when its depth bound terr is
// narrow, it is not near the outline or an end, and neither the cut nor any
// entry lies within terr + errmax of it, errmax being the widest bound of the
// entries whose t is an FP32 depth: these are then pairwise further apart
// than the sum of their bounds, so their FP32 order is their true order.
// Otherwise the hit is decided precisely, and so is every FP32 entry within
// errmax of its precise depth (the only entries whose order against it the
// FP32 depths leave open).
template <int KMAX, int COLS, bool COUNT>
__device__ __forceinline__ void keep_hit(const FrameArgs& fa, RayMem<KMAX, COLS>& rm, uint32_t c,
                                         uint32_t id, int r, float th, float terr, float& tcut,
                                         float& errmax, Counts& cn) {
  const uint32_t k = kbuf_depth<KMAX>(fa);
  const float slack = terr + errmax;
  const float s_off = rm.s_off[c];
  const bool own = r == kBorder || terr > kTieRel * (s_off + th);  // whatever else the ray hits
  bool need = own || th >= tcut - slack;
  for (uint32_t j = 0; j < k; ++j) need |= fabsf(th - rm.t[j][c]) <= slack;
  uint32_t word = id | (id < fa.N * fa.S ? kOpaque : 0u);  // strand ids come first
  float tr = 0.f;
  if (need) {
    const RayKey rk{rm.sid[0][c] | (uint64_t)rm.sid[1][c] << 32, s_off};
    if (COUNT) ++cn.precise_tests;
    float h, l;
    if (!refine(fa, rk, id, th, h, l)) {
      if (own) return;
      h = th, l = 0.f;  // not expected inside the FP32 bounds
    }
    const float depth = h;
    if (own)
      th = h, tr = l;
    else
      tr = __fadd_rn(__fsub_rn(h, th), l);
    word |= kExact;
    bool moved = false;
#pragma unroll 1
    for (uint32_t j = 0; j < k; ++j) {
      const float t = rm.t[j][c];
      if (t < kInf && !(rm.id[j][c] & kExact) && fabsf(depth - t) <= errmax) {
        if (COUNT) ++cn.precise_entries;
        if (refine(fa, rk, rm.id[j][c] & kIdMask, t, h, l)) rm.tr[j][c] = __fadd_rn(__fsub_rn(h, t), l);
        rm.id[j][c] |= kExact;
        moved = true;
      }
    }
    if (moved) {  // refined depths moved by at most errmax: restore the order
#pragma unroll 1
      for (uint32_t i = 1; i < k; ++i) kbuf_place(rm, c, (int)i, rm.t[i][c], rm.tr[i][c], rm.id[i][c]);
    }
  }
  if (!own) errmax = fmaxf(errmax, terr);
  if (key_less(th, tr, word, rm.t[k - 1][c], rm.tr[k - 1][c], rm.id[k - 1][c]))
    kbuf_place(rm, c, (int)k - 1, th, tr, word);
  tcut = kbuf_cut(rm, c, k);
}

template <int KMAX, int COLS, bool COUNT>
__device__ __forceinline__ void leaf_test(const FrameArgs& fa, RayMem<KMAX, COLS>& rm, uint32_t id,
                                          float& tcut, float& errmax, Counts& cn) {
  const uint32_t c = threadIdx.x;
  float th, terr;
  if (COUNT) ++cn.tests;
  const float4 r0 = __ldg(fa.prim_uv + 2 * (size_t)id), r1 = __ldg(fa.prim_uv + 2 * (size_t)id + 1);
  const int r = intersect32(fa, id, r0, r1, ray_o(rm, c), ray_d(rm, c), rm.M[c], tcut + errmax, th, terr);
  if (r != kMiss) keep_hit<KMAX, COLS, COUNT>(fa, rm, c, id, r, th, terr, tcut, errmax, cn);
}

// A ray against the node boxes (bvh.cu).  The plane at grid coordinate q is met at
// depth (lo + q step - o) / d.  A byte permutation of the box word with 2^23's
// bits gives 2^23 + q as a float, and picks the near or the far plane by the
// ray's direction at no further cost, so a plane takes one permutation and one
// FMA with scale = step / d and offset = (lo - o) / d - 2^23 scale.  The
// offset's rounding is at most half a step of depth, which the boxes' extra
// step covers.  A zero direction component would turn the products into
// inf - inf, so its sign is kept and its magnitude floored.  For boxes in FP32
// scale is 1 / d and offset -o / d.
struct Slabs {
  float3 scale, off;
  uint32_t nx, ny, nz;  // permutation that picks the near plane (xor kFar: the far one)
  bool wide;            // the boxes are in FP32
};
constexpr uint32_t kNearLo = 0x7610u, kFar = 0x0022u, kTwo23 = 0x4b000000u;
__device__ __forceinline__ void slab_axis(float o, float d, float lo, float step, bool wide, float& scale,
                                          float& off, uint32_t& sel) {
  const float inv = 1.0f / (fabsf(d) > 1e-12f ? d : copysignf(1e-12f, d));
  scale = wide ? inv : step * inv;
  off = wide ? -(o * inv) : fmaf(-8388608.f, scale, (lo - o) * inv);
  sel = inv < 0.f ? kNearLo ^ kFar : kNearLo;
}
__device__ __forceinline__ Slabs ray_slabs(const FrameArgs& fa, const float3 o, const float3 d) {
  const float4 lo = __ldg(fa.frame), st = __ldg(fa.frame + 1);
  Slabs s;
  s.wide = lo.w != 0.f;
  slab_axis(o.x, d.x, lo.x, st.x, s.wide, s.scale.x, s.off.x, s.nx);
  slab_axis(o.y, d.y, lo.y, st.y, s.wide, s.scale.y, s.off.y, s.ny);
  slab_axis(o.z, d.z, lo.z, st.z, s.wide, s.scale.z, s.off.z, s.nz);
  return s;
}
__device__ __forceinline__ float slab_t(uint32_t w, uint32_t sel, float scale, float off) {
  return fmaf(__uint_as_float(__byte_perm(w, kTwo23, sel)), scale, off);
}
// Entry depth (not below 0) of a child's box; false when the ray leaves it
// before or enters it after tmax.
__device__ __forceinline__ bool slab_test(const Slabs& s, const uint4 c, float tmax, float& t_in) {
  t_in = fmaxf(fmaxf(slab_t(c.x, s.nx, s.scale.x, s.off.x), slab_t(c.y, s.ny, s.scale.y, s.off.y)),
               fmaxf(slab_t(c.z, s.nz, s.scale.z, s.off.z), 0.f));
  const float t_out = fminf(fminf(slab_t(c.x, s.nx ^ kFar, s.scale.x, s.off.x),
                                  slab_t(c.y, s.ny ^ kFar, s.scale.y, s.off.y)),
                            fminf(slab_t(c.z, s.nz ^ kFar, s.scale.z, s.off.z), tmax));
  return t_in <= t_out;
}

// The same for a box in FP32: (lo.x, hi.x, lo.y, hi.y) and (lo.z, hi.z).
__device__ __forceinline__ bool slab_test(const Slabs& s, const float4 xy, float lz, float hz, float tmax,
                                          float& t_in) {
  const float x0 = fmaf(xy.x, s.scale.x, s.off.x), x1 = fmaf(xy.y, s.scale.x, s.off.x);
  const float y0 = fmaf(xy.z, s.scale.y, s.off.y), y1 = fmaf(xy.w, s.scale.y, s.off.y);
  const float z0 = fmaf(lz, s.scale.z, s.off.z), z1 = fmaf(hz, s.scale.z, s.off.z);
  t_in = fmaxf(fmaxf(fminf(x0, x1), fminf(y0, y1)), fmaxf(fminf(z0, z1), 0.f));
  const float t_out = fminf(fminf(fmaxf(x0, x1), fmaxf(y0, y1)), fminf(fmaxf(z0, z1), tmax));
  return t_in <= t_out;
}

// A node's children: which of them the ray meets before tmax, and where.  The
// walks are compiled for either kind of node and choose once a ray, which takes
// 0.5 to 2% of the frames on the grid (chosen once a tile, with the shading
// compiled twice, as much; a walk that is not inlined spills more).
struct Children {
  bool h0, h1;
  float a0, a1;
  int c0, c1;
};
template <bool WIDE>
__device__ __forceinline__ Children node_test(const FrameArgs& fa, const Slabs& s, int node, float tmax) {
  Children r;
  if (WIDE) {
    const float4* n = reinterpret_cast<const float4*>(fa.nodes) + 4 * (size_t)node;
    const float4 n0 = __ldg(n), n1 = __ldg(n + 1), n2 = __ldg(n + 2);
    const int2 ch = __ldg(reinterpret_cast<const int2*>(n + 3));
    r.h0 = slab_test(s, n0, n2.x, n2.y, tmax, r.a0);
    r.h1 = slab_test(s, n1, n2.z, n2.w, tmax, r.a1);
    r.c0 = ch.x, r.c1 = ch.y;
  } else {
    const uint4 k0 = __ldg(fa.nodes + 2 * (size_t)node), k1 = __ldg(fa.nodes + 2 * (size_t)node + 1);
    r.h0 = slab_test(s, k0, tmax, r.a0);
    r.h1 = slab_test(s, k1, tmax, r.a1);
    r.c0 = (int)k0.w, r.c1 = (int)k1.w;
  }
  return r;
}

// A lane's walk: the next node (kDone: none), the pending ones, the search cut
// and the widest bound of the FP32 hits kept.
constexpr int kDone = (int)0x80000000;
constexpr int kLeafWait = 3;
struct Walk {
  int node, sp;
  float tcut, errmax;
  bool ok;  // false once the traversal stack overflowed (a far subtree was dropped; never expected)
};

template <int KMAX, int COLS>
__device__ __forceinline__ void kbuf_clear(RayMem<KMAX, COLS>& rm, uint32_t c) {
#pragma unroll
  for (int j = 0; j < KMAX; ++j) {
    rm.t[j][c] = kInf;
    rm.tr[j][c] = 0.f;
    rm.id[j][c] = kNoEntry;
  }
}

__device__ __forceinline__ Walk walk_begin(const FrameArgs& fa, bool live) {
  return Walk{!live || fa.n_prims == 0 ? kDone : (fa.n_prims == 1 ? ~(int)__ldg(fa.leaf_id) : 0), 0, kInf,
              0.f, true};
}

// Walks on with the rays of the warp, one per lane, toward their K nearest
// hits; a lane that has used up `steps` node visits and tests stops where it
// is.  Whole warps call it.  Returns the steps that the lane has left.
// Boxes are culled against the cut widened by the FP32 hits' depth bound and
// by 2 kTieRel of the absolute depth, so that no hit the precise ordering
// would keep is lost to FP32 rounding of the slab tests.
// A lane that arrives at a leaf waits until kLeafWait eighths of the lanes still
// at work are at one: a leaf test is several times as long as a node visit,
// and one lane in seven is at a leaf on average, so tested at once they would
// run with a few lanes each.  With 1, 2, 3, 4 and 6 eighths the 4K frame of
// straight hair took (whole calls, before long walks were put aside) 14.3,
// 14.1, 14.1, 14.1 and 15.2 ms, the close view of the full head 4.21, 4.15,
// 4.14, 4.20 and 4.48 ms.
template <int KMAX, bool COUNT, bool WIDE>
__device__ __forceinline__ int walk_nodes(const FrameArgs& fa, const Slabs& sl, RayMem<KMAX, kBlock>& rm,
                                          Walk& w, int* stack, int steps, Counts& cn) {
  const float pad = 2.f * kTieRel * rm.s_off[threadIdx.x];
  float tcut = w.tcut, errmax = w.errmax;
  int sp = w.sp, node = w.node, stopped = kDone;
  for (;;) {
    if (node >= 0) {
      --steps;
      if (COUNT) ++cn.nodes;
      const Children ch = node_test<WIDE>(fa, sl, node, fmaf(tcut + errmax, 1.f + 2.f * kTieRel, pad));
      if (ch.h0 && ch.h1) {
        const bool first0 = ch.a0 <= ch.a1;
        node = first0 ? ch.c0 : ch.c1;
        if (sp < kStack)
          stack[sp++] = first0 ? ch.c1 : ch.c0;
        else
          w.ok = false;
      } else if (ch.h0 || ch.h1) {
        node = ch.h0 ? ch.c0 : ch.c1;
      } else {
        node = sp ? stack[--sp] : kDone;
      }
    }
    if (steps <= 0 && node != kDone) {
      stopped = node;
      node = kDone;
    }
    const unsigned inner = __ballot_sync(0xffffffffu, node >= 0);
    const unsigned leaf = __ballot_sync(0xffffffffu, node < 0 && node != kDone);
    if (!inner && !leaf) break;
    if (inner && __popc(leaf) * 8 < kLeafWait * __popc(inner | leaf)) continue;
    if (node < 0 && node != kDone) {
      --steps;
      leaf_test<KMAX, kBlock, COUNT>(fa, rm, (uint32_t)(~node), tcut, errmax, cn);
      node = sp ? stack[--sp] : kDone;
    }
  }
  w.node = stopped;
  w.sp = sp;
  w.tcut = tcut;
  w.errmax = errmax;
  return steps;
}
template <int KMAX, bool COUNT>
__device__ __forceinline__ int walk_on(const FrameArgs& fa, RayMem<KMAX, kBlock>& rm, Walk& w,
                                       int* stack, int steps, Counts& cn) {
  const Slabs sl = ray_slabs(fa, ray_o(rm, threadIdx.x), ray_d(rm, threadIdx.x));
  return sl.wide ? walk_nodes<KMAX, COUNT, true>(fa, sl, rm, w, stack, steps, cn)
                 : walk_nodes<KMAX, COUNT, false>(fa, sl, rm, w, stack, steps, cn);
}

// The K nearest hits of the warp's rays, one per live lane, without a stop.
template <int KMAX, bool COUNT>
__device__ __forceinline__ bool traverse(const FrameArgs& fa, RayMem<KMAX, kBlock>& rm, const bool live,
                                         Counts& cn) {
  int stack[kStack];
  kbuf_clear(rm, threadIdx.x);
  Walk w = walk_begin(fa, live);
  walk_on<KMAX, COUNT>(fa, rm, w, stack, 0x7fffffff, cn);
  return w.ok;
}

// ------------------------------------------------------------------ scattering

struct Mat {
  float A[3][3];  // [R, TT, D][rgb]
  float bR, bT, gT;
};

__device__ __forceinline__ void load_mat(const float* __restrict__ m, Mat& o) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(m));
  const float4 b = __ldg(reinterpret_cast<const float4*>(m) + 1);
  const float4 c = __ldg(reinterpret_cast<const float4*>(m) + 2);
  o.A[0][0] = a.x; o.A[0][1] = a.y; o.A[0][2] = a.z;
  o.A[1][0] = a.w; o.A[1][1] = b.x; o.A[1][2] = b.y;
  o.A[2][0] = b.z; o.A[2][1] = b.w; o.A[2][2] = c.x;
  o.bR = c.y; o.bT = c.z; o.gT = c.w;
}

// Gaussian G(beta, x) = exp(-x^2 / 2 beta^2) / (sqrt(2 pi) beta), Section 3.2,
// evaluated with the hardware exponential in both table precisions (a table
// gather costs more than the exponential it replaces).
__device__ __forceinline__ float gauss(float beta, float x) {
  const float ib = 1.0f / beta;
  const float z = x * ib;
  return __expf(-0.5f * z * z) * (kInvSqrt2Pi * ib);
}

// Longitudinal albedo factor IM(theta, beta), bilinear in the baked table.
template <int PREC>
__device__ __forceinline__ float im_lookup(const Tables& tb, float theta, float beta) {
  const float ft = clampf(theta * ((kImNT - 1) / (0.5f * kPi)), 0.f, (float)(kImNT - 1));
  const float fb = clampf((beta - kImBetaLo) * ((kImNB - 1) / (kImBetaHi - kImBetaLo)), 0.f,
                          (float)(kImNB - 1));
  const int it = min((int)ft, kImNT - 2), ib = min((int)fb, kImNB - 2);
  const float wt = ft - (float)it, wb = fb - (float)ib;
  float v00, v01, v10, v11;
  const int i0 = ib * kImNT + it;
  if (PREC == HR_PREC_FP32) {
    v00 = __ldg(tb.im32 + i0);
    v01 = __ldg(tb.im32 + i0 + 1);
    v10 = __ldg(tb.im32 + i0 + kImNT);
    v11 = __ldg(tb.im32 + i0 + kImNT + 1);
  } else {
    v00 = __half2float(tb.im16[i0]);
    v01 = __half2float(tb.im16[i0 + 1]);
    v10 = __half2float(tb.im16[i0 + kImNT]);
    v11 = __half2float(tb.im16[i0 + kImNT + 1]);
  }
  const float a = fmaf(wt, v01 - v00, v00), b = fmaf(wt, v11 - v10, v10);
  return fmaf(wb, b - a, a);
}

constexpr float kInv2Pi = 0.15915494309189535f;
constexpr float kInvPi = 0.3183098861837907f;
constexpr float kInv2Pi2 = 0.05066059182116889f;  // 1 / (2 pi^2)

// Single-fibre BCSDF, Eq. (1).  sg2: the spread variance gathered on the
// light's path (0 without shadow rays), added to every lobe's variance.  With
// trt (HR_FLAG_TRT, Marschner's R / TT / TRT fibre) the third lobe is
// A_TRT G(2 beta_R, theta_h) / 2 pi instead of the diffuse A_D / 2 pi^2.
template <int PREC>
__device__ __forceinline__ void f_single(const Tables& tb, const Mat& m, float th_i, float th_o,
                                         float cphi, float sg2, bool trt, float out[3]) {
  const float th_h = 0.5f * (th_i + th_o);
  const float phi = acosf(clampf(cphi, -1.f, 1.f));
  const bool wide = sg2 > 0.f;
  const float bR = wide ? sqrtf(fmaf(m.bR, m.bR, sg2)) : m.bR;
  const float bT = wide ? sqrtf(fmaf(m.bT, m.bT, sg2)) : m.bT;
  const float gT = wide ? sqrtf(fmaf(m.gT, m.gT, sg2)) : m.gT;
  const float mR = gauss(bR, th_h) * kInv2Pi;
  const float mT = gauss(bT, th_h) * gauss(gT, phi - kPi);
  const float m3 = trt ? gauss(sqrtf(fmaf(4.f * m.bR, m.bR, sg2)), th_h) * kInv2Pi : kInv2Pi2;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    out[c] = fmaf(m.A[0][c], mR, fmaf(m.A[1][c], mT, m.A[2][c] * m3));
}

// Per-hit constants of the aggregated model.
struct EthHit {
  float rho, n_view, nF, nB;
};

// Aggregated BCSDF of a thick hair, Eq. (5)-(13); readings as in the oracle:
// a_F, a_B at incidence |theta_d| / 2; variances add; n = 1 toward the back
// hemisphere (cos phi > 0); A_1+ summed in closed form for real n; B^ variance
// the attenuation-weighted mean of the path variances; S only for cos phi > 0
// with P_n floored at 0.
template <int PREC>
__device__ __forceinline__ void f_ours(const Tables& tb, const Mat& m, const EthHit& eh,
                                       float th_i, float th_o, float cphi, uint32_t flags,
                                       float sg2, float out[3]) {
  const float th_h = 0.5f * (th_i + th_o);
  const float ta = 0.5f * fabsf(th_i - th_o);
  const float phi = acosf(clampf(cphi, -1.f, 1.f));
  const bool trt = flags & HR_FLAG_TRT;
  const float imR = im_lookup<PREC>(tb, ta, m.bR);
  const float imT = im_lookup<PREC>(tb, ta, m.bT);
  // third lobe: diffuse (a quarter of A_D per half) or TRT (half of
  // A_TRT IM(2 beta_R) per half, its width weighted into the forward spread)
  const float im3 = trt ? 0.5f * im_lookup<PREC>(tb, ta, 2.f * m.bR) : 0.25f;
  float aF[3], aB[3];
  float wR = 0.f, wT = 0.f, w3 = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float r = m.A[0][c] * imR * 0.5f;
    const float tt = m.A[1][c] * imT;
    const float third = m.A[2][c] * im3;
    aF[c] = r + tt * eh.nF + third;
    aB[c] = r + tt * eh.nB + third;
    wR += r;
    wT += tt * eh.nF;
    w3 += third;
  }
  const float bR2 = m.bR * m.bR, bT2 = m.bT * m.bT;
  const float s2 = trt ? (wR * bR2 + wT * bT2 + w3 * 4.f * bR2) / (wR + wT + w3)
                       : (wR * bR2 + wT * bT2) / (wR + wT);
  const bool back = cphi > 0.f;
  const float n = back ? 1.f : eh.n_view;
  const float nm1 = n - 1.f;
  const float mR = gauss(sqrtf(fmaf(nm1, s2, bR2) + sg2), th_h) * kInv2Pi;
  const float mT = gauss(sqrtf(fmaf(nm1, s2, bT2) + sg2), th_h) *
                   gauss(sqrtf(fmaf(nm1, s2, m.gT * m.gT) + sg2), phi - kPi);
  const float m3 = trt ? gauss(sqrtf(fmaf(nm1, s2, 4.f * bR2) + sg2), th_h) * kInv2Pi : kInv2Pi2;
  float lob[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float att = nm1 > 0.f ? exp2f(nm1 * __log2f(aF[c])) : 1.f;
    lob[c] = att * fmaf(m.A[0][c], mR, fmaf(m.A[1][c], mT, m.A[2][c] * m3));
  }
  if (back) {
    float A1[3], A3[3], A1p[3];
    float w1 = 0.f, w3 = 0.f, w1p = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float f = fminf(aF[c], 1.f - 1e-6f);
      const float f2 = f * f, g = 1.f - f2, ig = 1.f / g;
      const float b = aB[c];
      A1[c] = b * f2 * ig;
      A3[c] = b * b * b * f2 * ig * ig * ig;
      A1p[c] = 0.6f * b * f * (1.f - exp2f(2.f * eh.n_view * __log2f(f))) * ig;
      w1 += A1[c];
      w3 += A3[c];
      w1p += A1p[c];
    }
    const float vB = (w1 * (bR2 + 2.f * s2) + w3 * (3.f * bR2 + 2.f * s2) +
                      w1p * (bR2 + (eh.n_view + 1.f) * s2)) / (w1 + w3 + w1p);
    const float mB = gauss(sqrtf(vB + sg2), th_h) * kInvPi;
#pragma unroll
    for (int c = 0; c < 3; ++c) lob[c] = fmaf(A1p[c] + A1[c] + A3[c], mB, lob[c]);
    if (!(flags & HR_FLAG_NO_S)) {
      const float Ps = (1.f - eh.rho) * (1.f - cphi);
      const float Pm = 0.2f * (1.f - eh.rho);
      const float Pn = fmaxf(0.f, 1.f - Pm - Ps);
#pragma unroll
      for (int c = 0; c < 3; ++c) lob[c] *= fmaf(Ps, aF[c], Pn);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c] = lob[c];
}

// Forward albedo a_F (rgb) and forward spread variance of a fibre for light
// at incidence |theta| (the a_F reading of the aggregated model).
template <int PREC>
__device__ __forceinline__ void forward_albedo(const Tables& tb, const Mat& m, float theta_abs,
                                               bool trt, float aF[3], float& s2) {
  const float imR = im_lookup<PREC>(tb, theta_abs, m.bR);
  const float imT = im_lookup<PREC>(tb, theta_abs, m.bT);
  const float im3 = trt ? 0.5f * im_lookup<PREC>(tb, theta_abs, 2.f * m.bR) : 0.25f;
  const float nF = erff(kPi / (2.f * 1.41421356f * m.gT));
  float wR = 0.f, wT = 0.f, w3 = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float r = m.A[0][c] * imR * 0.5f;
    const float tt = m.A[1][c] * imT * nF;
    const float third = m.A[2][c] * im3;
    aF[c] = r + tt + third;
    wR += r;
    wT += tt;
    w3 += third;
  }
  const float bR2 = m.bR * m.bR;
  s2 = trt ? (wR * bR2 + wT * m.bT * m.bT + w3 * 4.f * bR2) / (wR + wT + w3)
           : (wR * bR2 + wT * m.bT * m.bT) / (wR + wT);
}

// The ray's interval inside one record's finite cylinder, clipped to
// (tmin, tmax): the hair a shadow ray crosses, or the chord of a primary hit.
// Returns false when empty.
__device__ __forceinline__ bool leaf_span(const FrameArgs& fa, const uint32_t id, const float3 o,
                                          const float3 d, const float tmin, const float tmax,
                                          float& lo, float& hi) {
  const float4 r0 = __ldg(fa.prim_uv + 2 * (size_t)id), r1 = __ldg(fa.prim_uv + 2 * (size_t)id + 1);
  const float u0 = fmaf(r0.x, o.x, fmaf(r0.y, o.y, fmaf(r0.z, o.z, r0.w)));
  const float v0 = fmaf(r1.x, o.x, fmaf(r1.y, o.y, fmaf(r1.z, o.z, r1.w)));
  const float du = fmaf(r0.x, d.x, fmaf(r0.y, d.y, r0.z * d.z));
  const float dv = fmaf(r1.x, d.x, fmaf(r1.y, d.y, r1.z * d.z));
  const float A = fmaf(du, du, dv * dv);
  if (!(A > 0.f)) return false;
  const float inv = 1.0f / A;
  const float tc = -fmaf(u0, du, v0 * dv) * inv;
  const float uc = fmaf(tc, du, u0), vc = fmaf(tc, dv, v0);
  const float h2 = fmaf(uc, uc, vc * vc);
  if (h2 > 1.f) return false;
  const float half = sqrtf((1.f - h2) * inv);
  lo = tc - half;
  hi = tc + half;
  const float4 r2 = __ldg(fa.prim_wa + 2 * (size_t)id);
  const float w0 = fmaf(r2.x, o.x, fmaf(r2.y, o.y, fmaf(r2.z, o.z, r2.w)));
  const float dw = fmaf(r2.x, d.x, fmaf(r2.y, d.y, r2.z * d.z));
  if (dw != 0.f) {
    const float idw = 1.0f / dw;
    const float ta = -w0 * idw, tb = (1.f - w0) * idw;
    lo = fmaxf(lo, fminf(ta, tb));
    hi = fminf(hi, fmaxf(ta, tb));
  } else if (w0 < 0.f || w0 > 1.f) {
    return false;
  }
  lo = fmaxf(lo, tmin);
  hi = fminf(hi, tmax);
  return hi > lo;
}

// Transmittance of the light path of dual scattering (readings as in the
// oracle): the shadow ray from x along wi up to tmax crosses hairs; every
// primitive of the shading hair itself (material row self_mat) is skipped; a
// strand segment counts one hair, a thick-hair segment rho l sqrt(n_tot /
// (pi a b)) for its chord l; each hair multiplies T by its forward albedo at
// incidence |asin(wi . t)| and adds its forward spread variance; T = d_F prod
// a_F^n (d_F = 0.7) once a hair is crossed.  The walk visits every box on the
// path (all crossings count) and stops early once T < 1e-7 in every channel,
// where the light's contribution is below FP32 resolution of the pixel.
constexpr float kDF = 0.7f;
struct LightPath {
  float T[3], sg2;
  bool crossed;
};

// The path across primitive `id`; false once the light is used up.
template <int PREC>
__device__ __forceinline__ bool cross_leaf(const FrameArgs& fa, uint32_t id, const float3 x,
                                           const float3 wi, const float tmax, const uint32_t self_mat,
                                           LightPath& lp) {
  float lo, hi;
  float4 aux;
  if (!leaf_span(fa, id, x, wi, 0.f, tmax, lo, hi) ||
      __float_as_uint((aux = __ldg(fa.prim_wa + 2 * (size_t)id + 1)).x) == self_mat)
    return true;
  const float4 r2 = __ldg(fa.prim_wa + 2 * (size_t)id);
  const float si = clampf(dot3(wi, f3(r2.x, r2.y, r2.z)) *
                              rsqrtf(r2.x * r2.x + r2.y * r2.y + r2.z * r2.z),
                          -1.f, 1.f);
  Mat m;
  load_mat(fa.mat + (size_t)__float_as_uint(aux.x) * HR_MAT_FLOATS, m);
  float aF[3], s2;
  forward_albedo<PREC>(fa.tables, m, fabsf(asinf(si)), (fa.flags & HR_FLAG_TRT) != 0, aF, s2);
  if (aux.y > 0.f) {  // thick hair: its hair number over the chord
    const float ntot = aux.y, r = aux.z, ab = aux.w;
    const float rho = fminf(1.f, ntot * r * r / ab);
    const float n = rho * (hi - lo) * sqrtf(ntot / (kPi * ab));
#pragma unroll
    for (int c = 0; c < 3; ++c) lp.T[c] *= exp2f(n * __log2f(aF[c]));
    lp.sg2 = fmaf(n, s2, lp.sg2);
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) lp.T[c] *= aF[c];
    lp.sg2 += s2;
  }
  lp.crossed = true;
  return !(fmaxf(lp.T[0], fmaxf(lp.T[1], lp.T[2])) < 1e-7f);
}

// One node of a path: the next node, the other hit child on the stack.
template <bool WIDE>
__device__ __forceinline__ int path_node(const FrameArgs& fa, const Slabs& sl, int node, const float tmax,
                                         int* stack, int& sp, bool& ok) {
  const Children ch = node_test<WIDE>(fa, sl, node, tmax);
  if (ch.h0 && ch.h1) {
    if (sp < kStack)
      stack[sp++] = ch.c1;
    else
      ok = false;
    return ch.c0;
  }
  if (ch.h0 || ch.h1) return ch.h0 ? ch.c0 : ch.c1;
  return sp ? stack[--sp] : kDone;
}

// The light paths of a warp's lanes (lanes that are not live have none); with
// WHOLE the whole warp calls it and leaves wait for one another as in walk_on,
// without it each lane walks by itself.
template <int PREC, bool COUNT, bool WHOLE, bool WIDE>
__device__ __forceinline__ void path_walk(const FrameArgs& fa, const Slabs& sl, bool live, const float3 x,
                                          const float3 wi, const float tmax, const uint32_t self_mat,
                                          LightPath& lp, bool& ok, Counts& cn) {
  int stack[kStack];
  int sp = 0;
  int node = !live || fa.n_prims == 0 ? kDone : (fa.n_prims == 1 ? ~(int)__ldg(fa.leaf_id) : 0);
  for (;;) {
    if (node >= 0) {
      if (COUNT) ++cn.nodes;
      node = path_node<WIDE>(fa, sl, node, tmax, stack, sp, ok);
    }
    if (WHOLE) {
      const unsigned inner = __ballot_sync(0xffffffffu, node >= 0);
      const unsigned leaf = __ballot_sync(0xffffffffu, node < 0 && node != kDone);
      if (!inner && !leaf) break;
      if (inner && __popc(leaf) * 8 < kLeafWait * __popc(inner | leaf)) continue;
    } else {
      if (node == kDone) break;
    }
    if (node < 0 && node != kDone) {
      if (COUNT) ++cn.tests;
      node = !cross_leaf<PREC>(fa, (uint32_t)(~node), x, wi, tmax, self_mat, lp) || !sp ? kDone
                                                                                       : stack[--sp];
    }
  }
}
template <int PREC, bool COUNT, bool WHOLE>
__device__ __forceinline__ void shadow_path(const FrameArgs& fa, bool live, const float3 x,
                                            const float3 wi, const float tmax, const uint32_t self_mat,
                                            float T[3], float& sg2, bool& ok, Counts& cn) {
  LightPath lp{{1.f, 1.f, 1.f}, 0.f, false};
  const Slabs sl = ray_slabs(fa, x, wi);
  if (sl.wide)
    path_walk<PREC, COUNT, WHOLE, true>(fa, sl, live, x, wi, tmax, self_mat, lp, ok, cn);
  else
    path_walk<PREC, COUNT, WHOLE, false>(fa, sl, live, x, wi, tmax, self_mat, lp, ok, cn);
  const float dF = lp.crossed ? kDF : 1.f;
  T[0] = lp.T[0] * dF;
  T[1] = lp.T[1] * dF;
  T[2] = lp.T[2] * dF;
  sg2 = lp.sg2;
}

// Direction from x toward a light and its falloff E; the length of the light
// path.
__device__ __forceinline__ void light_dir(const float4 L, const float3 x, float3& wi, float& E) {
  E = 1.f;
  if (L.w == 0.f) {
    wi = f3(L.x, L.y, L.z);
  } else {
    const float3 to = f3(L.x, L.y, L.z) - x;
    const float dd = dot3(to, to);
    const float id = rsqrtf(dd);
    wi = to * id;
    E = id * id;
  }
}
__device__ __forceinline__ float path_length(const float4 L, float E) {
  return L.w == 0.f ? kInf : sqrtf(1.f / E);
}

// Radiance of one hit toward -d (sum over lights of T f E cos(theta_i), T and
// the spread of f from shadow_path when SHADOW (HR_FLAG_SHADOWS), else T = 1)
// and its opacity (strand 1; thick hair 1 - exp(-2 r l n_tot / (pi a b))).
// SHADOW is a template parameter so kernels without shadow rays carry none
// of their registers.  With PATHS the light paths were walked before: light
// l's (T, spread variance) is paths[l * path_stride].
template <int PREC, bool COUNT, bool SHADOW = false, bool PATHS = false>
__device__ __forceinline__ void shade_hit(const FrameArgs& fa, uint32_t id, float t,
                                          const float3 o, const float3 d, float rgb[3],
                                          float& alpha, Counts& cn,
                                          const float4* __restrict__ paths = nullptr,
                                          size_t path_stride = 0) {
  const float4 r2 = __ldg(fa.prim_wa + 2 * (size_t)id), aux = __ldg(fa.prim_wa + 2 * (size_t)id + 1);
  const float3 T = f3(r2.x, r2.y, r2.z) * rsqrtf(r2.x * r2.x + r2.y * r2.y + r2.z * r2.z);
  Mat m;
  load_mat(fa.mat + (size_t)__float_as_uint(aux.x) * HR_MAT_FLOATS, m);
  const float3 wo = d * -1.f;
  const float so = clampf(dot3(wo, T), -1.f, 1.f);
  const float th_o = asinf(so);
  const float3 wop = wo - T * so;
  const float nop = sqrtf(dot3(wop, wop));
  const float3 x = hit_point(o, d, t);
  const bool eth = aux.y > 0.f && !(fa.flags & HR_FLAG_SINGLE_ON_ETH);
  EthHit eh{0.f, 1.f, 0.f, 0.f};
  alpha = 1.f;
  if (aux.y > 0.f) {
    // the chord: the ray's length inside the finite cylinder (0 when FP32
    // rounding puts a hit at the very outline outside it)
    float lo, hi;
    const float chord =
        leaf_span(fa, id, o, d, -kInf, kInf, lo, hi) ? hi - lo : 0.f;
    const float ntot = aux.y, r = aux.z, ab = aux.w;
    eh.rho = fminf(1.f, ntot * r * r / ab);
    const float n_raw = eh.rho * chord * sqrtf(ntot / (kPi * ab));
    eh.n_view = fmaxf(1.f, n_raw);
    alpha = 1.f - __expf(-2.f * r * chord * ntot / (kPi * ab));
    eh.nF = erff(kPi / (2.f * 1.41421356f * m.gT));
    eh.nB = erff(kPi / (1.41421356f * m.gT)) - eh.nF;
  }
  rgb[0] = rgb[1] = rgb[2] = 0.f;
  for (int l = 0; l < fa.lights.n; ++l) {
    const float4 L = fa.lights.xyzw[l];
    float3 wi;
    float E;
    light_dir(L, x, wi, E);
    const float si = clampf(dot3(wi, T), -1.f, 1.f);
    const float th_i = asinf(si);
    const float3 wip = wi - T * si;
    const float nip = sqrtf(dot3(wip, wip));
    const float cphi =
        (nip > 0.f && nop > 0.f) ? clampf(dot3(wip, wop) / (nip * nop), -1.f, 1.f) : 1.f;
    float Tl[3] = {1.f, 1.f, 1.f}, sg2 = 0.f;
    if (SHADOW) {
      bool sok = true;
      shadow_path<PREC, COUNT, false>(fa, true, x, wi, path_length(L, E), __float_as_uint(aux.x), Tl, sg2,
                                      sok, cn);
      if (!sok) atomicAdd(fa.overflow, 1u);
    }
    if (PATHS) {
      const float4 path = __ldg(paths + l * path_stride);
      Tl[0] = path.x;
      Tl[1] = path.y;
      Tl[2] = path.z;
      sg2 = path.w;
    }
    float f[3];
    if (eth) {
      f_ours<PREC>(fa.tables, m, eh, th_i, th_o, cphi, fa.flags, sg2, f);
      if (COUNT) ++cn.eshade;
    } else {
      f_single<PREC>(fa.tables, m, th_i, th_o, cphi, sg2, (fa.flags & HR_FLAG_TRT) != 0, f);
      if (COUNT) ++cn.sshade;
    }
    const float g = E * sqrtf(fmaxf(0.f, 1.f - si * si));
    const float4 Lc = fa.lights.rgb[l];
    rgb[0] = fmaf(f[0] * Tl[0] * g, Lc.x, rgb[0]);
    rgb[1] = fmaf(f[1] * Tl[1] * g, Lc.y, rgb[1]);
    rgb[2] = fmaf(f[2] * Tl[2] * g, Lc.z, rgb[2]);
  }
}

// Shading and front-to-back compositing of a sample's hits (entry j's depth at
// t[j * stride], with SHADOW its low part at tr[j * stride], its word at
// id[j * stride], nearest first).
template <int PREC, bool COUNT, bool SHADOW>
__device__ __forceinline__ void shade_hits(const FrameArgs& fa, const float* t, const float* tr,
                                           const uint32_t* id, uint32_t stride, uint32_t k, const float3 o, const float3 d,
                                           float out[3], Counts& cn) {
  out[0] = out[1] = out[2] = 0.f;
  float T = 1.f;
#pragma unroll 1
  for (uint32_t j = 0; j < k; ++j) {
    const float tj = SHADOW ? __fadd_rn(t[j * stride], tr[j * stride]) : t[j * stride];
    if (!(tj < kInf && T > 0.f)) break;  // sorted by depth
    float rgb[3], a;
    shade_hit<PREC, COUNT, SHADOW>(fa, id[j * stride] & kIdMask, tj, o, d, rgb, a, cn);
    if (COUNT) ++cn.hits;
    const float ta = T * a;
    out[0] = fmaf(ta, rgb[0], out[0]);
    out[1] = fmaf(ta, rgb[1], out[1]);
    out[2] = fmaf(ta, rgb[2], out[2]);
    T *= 1.f - a;
  }
}

template <int KMAX>
__device__ __forceinline__ void primary_store(const FrameArgs& fa, RayMem<KMAX, kBlock>& rm, uint64_t sid) {
  RayKey rk;
  float3 o, d;
  primary_ray(fa, sid, o, d, rk);
  ray_store(rm, threadIdx.x, o, d, rk);
}

// One sample per live lane: ray, K nearest hits, shading and compositing.
// Whole warps call it.
template <int KMAX, int PREC, bool COUNT, bool SHADOW = false>
__device__ __forceinline__ void render_sample(const FrameArgs& fa, RayMem<KMAX, kBlock>& rm, uint64_t sid,
                                              const bool live, float out[3],
                                              bool& ok, Counts& cn) {
  const uint32_t c = threadIdx.x;
  primary_store(fa, rm, sid);
  ok = traverse<KMAX, COUNT>(fa, rm, live, cn);
  out[0] = out[1] = out[2] = 0.f;
  if (live)
    shade_hits<PREC, COUNT, SHADOW>(fa, &rm.t[0][c], &rm.tr[0][c], &rm.id[0][c], kBlock, kbuf_depth<KMAX>(fa),
                                    ray_o(rm, c), ray_d(rm, c), out, cn);
}

// ---------------------------------------------------------------- long walks
//
// A few rays walk ten or a hundred times as far as the others (they skim the
// layer in which the strands bend or lie along the view: 4,000 visits and
// 6,500 tests in the 4K frame of straight hair, 55 of both on average), and
// the frame lasts as long as the warp that traces them.  A ray that has used
// up its budget of steps is therefore put aside with its pending nodes and its
// hits, and a second kernel finishes these rays with a whole warp each.

// A tile with rays put aside: what the last of them needs to composite it.
struct LongTile {
  uint32_t xy;         // origin, x | y << 16
  uint32_t lanes;      // lanes whose rays were put aside
  uint32_t left;       // of those, not finished yet
  uint32_t part;       // lanes whose pixels it stores (small frames: a part of the tile)
  float acc[3][32];    // the lanes' radiance
  uint32_t at[32];     // where a put-aside lane's record starts
};
// A ray's record, in words: tile, lane | pending nodes << 8, cut, widest
// bound, k depths, k low words of depths, k entry words, the pending nodes
// (last the first to visit).
constexpr uint32_t kLongHead = 4;

// Puts the rays of the lanes in `mask` aside (the lane's walk w stopped short
// in them).  False when there is no room: nothing is put aside.
template <int KMAX>
__device__ __forceinline__ bool put_aside(const FrameArgs& fa, const RayMem<KMAX, kBlock>& rm,
                                          const Walk& w, const int* stack, uint32_t x0, uint32_t y0,
                                          unsigned mask, bool inside, uint32_t& tile) {
  const uint32_t lane = threadIdx.x & 31, c = threadIdx.x, k = fa.k;
  const bool mine = (mask >> lane) & 1u;
  const uint32_t words = mine ? kLongHead + 3 * k + (uint32_t)w.sp + 1 : 0u;
  uint32_t incl = words;
#pragma unroll
  for (int q = 1; q < 32; q <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, q);
    if (lane >= (uint32_t)q) incl += v;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, incl, 31), rays = (uint32_t)__popc(mask);
  uint32_t at = 0xffffffffu, first = 0;
  tile = 0;
  if (lane == 0) {
    // room as far as one can see (the counters stay far from wrapping), then for certain
    if (__ldcg(fa.lw.ctr + 1) + total <= fa.lw.words && __ldcg(fa.lw.ctr + 2) < fa.lw.tiles_max &&
        __ldcg(fa.lw.ctr) + rays <= fa.lw.rays_max) {
      at = atomicAdd(fa.lw.ctr + 1, total);
      tile = atomicAdd(fa.lw.ctr + 2, 1u);
      if (at + total > fa.lw.words || tile >= fa.lw.tiles_max) {
        at = 0xffffffffu;
      } else {
        first = atomicAdd(fa.lw.ctr, rays);
        if (first + rays > fa.lw.rays_max) {  // the places taken below the limit stay empty
          for (uint32_t i = first; i < fa.lw.rays_max; ++i) fa.lw.ray_at[i] = 0xffffffffu;
          at = 0xffffffffu;
        }
      }
    }
  }
  at = __shfl_sync(0xffffffffu, at, 0);
  if (at == 0xffffffffu) return false;
  tile = __shfl_sync(0xffffffffu, tile, 0);
  first = __shfl_sync(0xffffffffu, first, 0);
  at += incl - words;
  const unsigned part = __ballot_sync(0xffffffffu, inside);
  if (lane == 0) {
    fa.lw.tiles[tile].xy = x0 | y0 << 16;
    fa.lw.tiles[tile].lanes = mask;
    fa.lw.tiles[tile].left = rays;
    fa.lw.tiles[tile].part = part;
  }
  if (mine) {
    fa.lw.tiles[tile].at[lane] = at;
    fa.lw.ray_at[first + __popc(mask & ((1u << lane) - 1u))] = at;
    uint32_t* r = fa.lw.pool + at;
    r[0] = tile;
    r[1] = lane | (uint32_t)(w.sp + 1) << 8;
    r[2] = __float_as_uint(w.tcut);
    r[3] = __float_as_uint(w.errmax);
    for (uint32_t j = 0; j < k; ++j) {
      r[kLongHead + j] = __float_as_uint(rm.t[j][c]);
      r[kLongHead + k + j] = __float_as_uint(rm.tr[j][c]);
      r[kLongHead + 2 * k + j] = rm.id[j][c];
    }
    r += kLongHead + 3 * k;
    for (int j = 0; j < w.sp; ++j) r[j] = (uint32_t)stack[j];
    r[w.sp] = (uint32_t)w.node;
  }
  return true;
}

__device__ __forceinline__ void flush_counts(const FrameArgs& fa, const Counts& cn) {
  unsigned long long v[8] = {cn.nodes, cn.tests, cn.sshade, cn.eshade, cn.hits, cn.rays,
                             cn.precise_tests, cn.precise_entries};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    unsigned long long x = v[i];
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(fa.counters + i, x);
  }
}

// Pixel-space rectangle (x0, y0, x1, y1) that contains the projection of the
// BVH root box, grown by one pixel; computed by one warp (lanes 0-7 project
// the box corners) and stored by lane 0.  A pixel whose square lies outside it
// cannot see any primitive.  The whole screen when the box reaches behind the
// eye or the BVH has fewer than two leaves.
__device__ __forceinline__ void scene_rect_warp(const FrameArgs& fa, float4* rect) {
  {
    const int lane = threadIdx.x & 31;
    float X0 = kInf, Y0 = kInf, X1 = -kInf, Y1 = -kInf;
    bool ok = fa.n_prims >= 2;
    if (ok && lane < 8) {
      float3 blo, bhi;
      root_box(fa, blo, bhi);
      const float3 p = f3((lane & 1) ? bhi.x : blo.x, (lane & 2) ? bhi.y : blo.y,
                          (lane & 4) ? bhi.z : blo.z);
      const float3 r = p - fa.cam.eye;
      const float xc = dot3(r, fa.cam.right), yc = dot3(r, fa.cam.up), zc = dot3(r, fa.cam.fwd);
      float X, Y;
      if (fa.cam.kind == 1) {
        ok = zc > 1e-6f;
        X = xc / zc * fa.cam.pix;
        Y = -yc / zc * fa.cam.pix;
      } else {
        X = xc * fa.cam.pix;
        Y = -yc * fa.cam.pix;
      }
      X += 0.5f * (float)fa.cam.W;
      Y += 0.5f * (float)fa.cam.H;
      if (!(X == X) || !(Y == Y)) ok = false;
      X0 = X1 = X;
      Y0 = Y1 = Y;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      X0 = fminf(X0, __shfl_xor_sync(0xffffffffu, X0, o));
      Y0 = fminf(Y0, __shfl_xor_sync(0xffffffffu, Y0, o));
      X1 = fmaxf(X1, __shfl_xor_sync(0xffffffffu, X1, o));
      Y1 = fmaxf(Y1, __shfl_xor_sync(0xffffffffu, Y1, o));
    }
    ok = __all_sync(0xffffffffu, ok);
    if (lane == 0)
      *rect = ok ? make_float4(X0 - 1.f, Y0 - 1.f, X1 + 1.f, Y1 + 1.f)
                 : make_float4(-kInf, -kInf, kInf, kInf);
  }
}

// Warp tile: the 32 / grp pixels one warp renders (wtw x wth); a pixel's
// samples on `grp` adjacent lanes.
struct TileLane {
  bool inside;     // the lane's pixel is in the image and in the scene's rectangle
  uint64_t pixel;
};
__device__ __forceinline__ TileLane tile_lane(const FrameArgs& fa, uint32_t x0, uint32_t y0, uint32_t wtw,
                                              const float4 rect) {
  const uint32_t p = (threadIdx.x & 31) / fa.grp;
  const uint32_t x = x0 + p % wtw, y = y0 + p / wtw;
  TileLane t;
  t.inside = x < (uint32_t)fa.cam.W && y < (uint32_t)fa.cam.H && (float)x + 1.f >= rect.x &&
             (float)x <= rect.z && (float)y + 1.f >= rect.y && (float)y <= rect.w;
  t.pixel = (uint64_t)y * (uint32_t)fa.cam.W + x;
  return t;
}

// Sums a pixel's lanes with a fixed XOR-shuffle tree and stores the mean.
// Whole warps call it.
__device__ __forceinline__ void tile_write(const FrameArgs& fa, const TileLane tl, float acc[3],
                                           float* __restrict__ rgb) {
  const uint32_t G = fa.grp;
  for (uint32_t o = 1; o < G; o <<= 1) {
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
    acc[1] += __shfl_xor_sync(0xffffffffu, acc[1], o);
    acc[2] += __shfl_xor_sync(0xffffffffu, acc[2], o);
  }
  if (tl.inside && (threadIdx.x & (G - 1)) == 0) {
    const float inv = 1.0f / (float)fa.spp;
    rgb[3 * tl.pixel] = acc[0] * inv;
    rgb[3 * tl.pixel + 1] = acc[1] * inv;
    rgb[3 * tl.pixel + 2] = acc[2] * inv;
  }
}

// Traces, shades and stores the part of a tile (whole pixels).  With LONG, rays over the budget of steps
// are put aside (at most one sample a lane: no more than 32 spp) and
// the tile is stored by the last of them.
template <int KMAX, int PREC, bool COUNT, bool SHADOW = false, bool LONG = false>
__device__ __forceinline__ void render_warp_tile(const FrameArgs& fa, RayMem<KMAX, kBlock>& rm,
                                                 uint32_t x0, uint32_t y0, uint32_t wtw,
                                                 const float4 rect, int budget,
                                                 float* __restrict__ rgb, Counts& cn, bool& overflow,
                                                 const unsigned part = 0xffffffffu) {
  const uint32_t G = fa.grp, c = threadIdx.x, lane = c & 31;
  TileLane tl = tile_lane(fa, x0, y0, wtw, rect);
  tl.inside = tl.inside && ((part >> lane) & 1u);
  if (!__any_sync(0xffffffffu, tl.inside)) return;
  float acc[3] = {0.f, 0.f, 0.f};
  for (uint32_t s0 = 0; s0 < fa.spp; s0 += G) {
    const uint32_t s = s0 + (lane & (G - 1));
    const bool live = tl.inside && s < fa.spp;
    primary_store(fa, rm, tl.pixel * fa.spp + s);
    kbuf_clear(rm, c);
    int stack[kStack];
    Walk w = walk_begin(fa, live);
    unsigned aside = 0;
    uint32_t tile = 0;
    for (int steps = LONG ? budget : 0x7fffffff;; steps = 0x7fffffff) {
      const int left = walk_on<KMAX, COUNT>(fa, rm, w, stack, steps, cn);
      if (LONG) {
        cn.steps += (uint32_t)(steps - left);
        aside = __ballot_sync(0xffffffffu, w.node != kDone);
        if (aside && !put_aside<KMAX>(fa, rm, w, stack, x0, y0, aside, tl.inside, tile)) continue;
      }
      break;
    }
    float v[3] = {0.f, 0.f, 0.f};
    if (live && !((aside >> lane) & 1u))
      shade_hits<PREC, COUNT, SHADOW>(fa, &rm.t[0][c], &rm.tr[0][c], &rm.id[0][c], kBlock, kbuf_depth<KMAX>(fa),
                                      ray_o(rm, c), ray_d(rm, c), v, cn);
    if (COUNT && live) ++cn.rays;
    overflow |= !w.ok;
    acc[0] += v[0];
    acc[1] += v[1];
    acc[2] += v[2];
    if (LONG && aside) {
      LongTile& lt = fa.lw.tiles[tile];
      lt.acc[0][lane] = acc[0];
      lt.acc[1][lane] = acc[1];
      lt.acc[2][lane] = acc[2];
      return;
    }
  }
  tile_write(fa, tl, acc, rgb);
}

}  // namespace tr
}  // namespace hr
