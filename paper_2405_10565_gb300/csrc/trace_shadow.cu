// Frames with dual-scattering light paths (HR_FLAG_SHADOWS) in three kernels
// a round: the primary rays and their hits, one light path per (hit, light),
// and the shading of the hits with the paths' transmittances.
//
// A light path is a whole BVH walk (the full-head frame makes 840 node visits
// a traced sample for its eight lights, 46 for the primary ray).  Walked
// inside the shading loop they run one after the other per sample, so a frame
// lasts as long as the tile whose lanes walk the most, at the few warps that a
// kernel holding the primary ray's and the shading's state can keep resident:
// 14.2 ms for 100k strands at 1920 x 1080, 8 spp, 8 lights, at a tenth of the
// close view's visits per second.  As independent walks of a lean kernel, 32
// neighbouring hits toward one light per warp, they fill the GPU: 4.5 ms, and
// 4.1 with leaves waiting for one another as in the primary rays' walk.
//
// The hits of a round and their paths go to buffers of kPathBytes at most; the
// primary kernel stops taking tiles once they are full and the next round goes on
// from there.  The host does not know how many rounds a frame needs without
// waiting for it, so it launches up to kMaxRounds and, when the worst case
// would need more, the one-kernel form for whatever tiles are left: a close view
// of the same head (6.4M traced samples) does not fit in the rounds and takes 34
// ms with 8 lights and 70 with 16, a middle view with 8 lights 12 (56, 118 and 21
// with the paths walked in the shading loop throughout).
#include <algorithm>

#include "trace_frame.cuh"

namespace hr {
namespace {

constexpr uint64_t kPathBytes = 448ull << 20;  // 2.5M hits of 8 lights, 13M of one, beside those at work
constexpr uint32_t kMaxRounds = 3;
// A round costs about 25 us more than the one-kernel form where little is
// walked (four launches in a row for one); that form walks a hit's paths one
// after the other, so its time goes with the lights and with the depth of the
// scene.  Rounds / one kernel, us a call at 400 x 300, 2 spp, 1, 2, 4, 8 lights:
// 2.8k segments 109 / 80, 112 / 97, 116 / 142, 120 / 199; 9k segments 197 / 148,
// 197 / 183, 205 / 284, 219 / 479; 44k segments of curls 465 / 357, 509 / 571;
// 96k straight ones 1739 / 3687; 256k 685 / 1134.  So the smallest scenes by
// the number of lights are left to the one kernel, up to the 1M samples measured.
constexpr uint32_t kOneKernelPrims = 49152;  // over the cube of the lights
constexpr uint64_t kOneKernelSamples = 1ull << 20;

struct ShadowTile {
  uint32_t tile;      // index in the frame's warp grid
  uint32_t base;      // first hit of the tile
  uint32_t cnt[8];    // hits of each lane, eight bits each
};

struct ShadowWork {
  uint32_t* ctr;      // [0] hits, [1] tiles with hits (of the round)
  float4* hit;        // [cap] hit position and entry word (id, flags)
  float* depth;       // [cap] depth past the re-based origin
  ShadowTile* tiles;  // [the frame's warp tiles, cap at most]
  float4* path;       // [lights][cap] (T rgb, spread variance)
  uint32_t stop;      // no further tile is taken at this many hits
  uint32_t cap;       // stop plus what the warps at work can still add
};

// Primary rays of the tiles handed out; every hit that shading can reach (up
// to the first opaque one) is listed, a tile's hits together and in lane
// order.
template <int KMAX>
__global__ void __launch_bounds__(kBlock, tr::kTraceBlocks)
    k_shadow_hits(const FrameArgs fa, const float4* __restrict__ rect_p, uint32_t* work,
                  const ShadowWork sw) {
  __shared__ tr::RayMem<KMAX, kBlock> rm;
  const float4 rect = *rect_p;
  const WarpGrid g = warp_grid(rect, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  const uint32_t lane = threadIdx.x & 31, G = fa.grp;
  bool overflow = false;
  for (;;) {
    uint32_t t = 0xffffffffu;
    if (lane == 0 && __ldcg(sw.ctr) < sw.stop) t = atomicAdd(work, 1u);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= g.n) break;
    const uint32_t x0 = g.x0 + (t % g.nx) * g.wtw, y0 = g.y0 + (t / g.nx) * g.wth;
    const tr::TileLane tl = tr::tile_lane(fa, x0, y0, g.wtw, rect);
    const uint32_t s = lane & (G - 1);
    const bool live = tl.inside && s < fa.spp;
    tr::primary_store(fa, rm, tl.pixel * fa.spp + s);
    tr::Counts cn{0, 0, 0, 0, 0, 0, 0, 0};
    overflow |= !tr::traverse<KMAX, false>(fa, rm, live, cn);
    uint32_t cnt = 0;
    if (live)
      for (bool past = false; cnt < fa.k && rm.t[cnt][threadIdx.x] < kInf && !past; ++cnt)
        past = (rm.id[cnt][threadIdx.x] & tr::kOpaque) != 0u;
    uint32_t incl = cnt;
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, q);
      if (lane >= (uint32_t)q) incl += v;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (!total) continue;  // background: the image is cleared
    uint32_t base = 0, rec = 0;
    if (lane == 0) {
      base = atomicAdd(sw.ctr, total);
      rec = atomicAdd(sw.ctr + 1, 1u);
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    rec = __shfl_sync(0xffffffffu, rec, 0);
    if (lane == 0) {
      sw.tiles[rec].tile = t;
      sw.tiles[rec].base = base;
    }
    reinterpret_cast<uint8_t*>(sw.tiles[rec].cnt)[lane] = (uint8_t)cnt;
    const uint32_t h0 = base + incl - cnt;
    for (uint32_t j = 0; j < cnt; ++j) {
      const float t = __fadd_rn(rm.t[j][threadIdx.x], rm.tr[j][threadIdx.x]);
      const float3 x3 = tr::hit_point(tr::ray_o(rm, threadIdx.x), tr::ray_d(rm, threadIdx.x), t);
      sw.hit[h0 + j] = make_float4(x3.x, x3.y, x3.z, __uint_as_float(rm.id[j][threadIdx.x]));
      sw.depth[h0 + j] = t;
    }
  }
  if (overflow) atomicAdd(fa.overflow, 1u);
}

// The light paths: a warp takes 32 consecutive hits and one light.
template <int PREC>
__global__ void __launch_bounds__(kBlock) k_shadow_paths(const FrameArgs fa, const ShadowWork sw) {
  const uint32_t n = *sw.ctr, L = (uint32_t)fa.lights.n;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t tasks = (uint64_t)((n + 31) / 32) * L;
  const uint64_t warps = (uint64_t)gridDim.x * (kBlock / 32);
  for (uint64_t w = ((uint64_t)blockIdx.x * kBlock + threadIdx.x) >> 5; w < tasks; w += warps) {
    const uint32_t l = (uint32_t)(w % L), h = (uint32_t)(w / L) * 32 + lane;
    const bool live = h < n;
    const float4 hit = __ldg(sw.hit + (live ? h : 0));
    const uint32_t id = __float_as_uint(hit.w) & tr::kIdMask;
    const float3 x = tr::f3(hit.x, hit.y, hit.z);
    const float4 light = fa.lights.xyzw[l];
    float3 wi;
    float E;
    tr::light_dir(light, x, wi, E);
    float T[3], sg2;
    bool ok = true;
    tr::Counts cn{0, 0, 0, 0, 0, 0, 0, 0};
    tr::shadow_path<PREC, false, true>(fa, live, x, wi, tr::path_length(light, E),
                                       __float_as_uint(__ldg(&fa.prim_wa[2 * (size_t)id + 1].x)), T, sg2,
                                       ok, cn);
    if (!ok) atomicAdd(fa.overflow, 1u);
    if (live) sw.path[(size_t)l * sw.cap + h] = make_float4(T[0], T[1], T[2], sg2);
  }
}

// Shading and compositing of the listed tiles, one warp each, with the same
// sums as the one-kernel form.
template <int PREC>
__global__ void __launch_bounds__(kBlock)
    k_shadow_shade(const FrameArgs fa, const float4* __restrict__ rect_p, const ShadowWork sw,
                   float* __restrict__ rgb) {
  const float4 rect = *rect_p;
  const WarpGrid g = warp_grid(rect, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  const uint32_t lane = threadIdx.x & 31, G = fa.grp;
  const uint32_t n = sw.ctr[1], warps = gridDim.x * (kBlock / 32);
  for (uint32_t i = (blockIdx.x * kBlock + threadIdx.x) >> 5; i < n; i += warps) {
    const ShadowTile& st = sw.tiles[i];
    const uint32_t t = st.tile, cnt = reinterpret_cast<const uint8_t*>(st.cnt)[lane];
    uint32_t incl = cnt;
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, q);
      if (lane >= (uint32_t)q) incl += v;
    }
    const uint32_t h0 = st.base + incl - cnt;
    const uint32_t x0 = g.x0 + (t % g.nx) * g.wtw, y0 = g.y0 + (t / g.nx) * g.wth;
    const tr::TileLane tl = tr::tile_lane(fa, x0, y0, g.wtw, rect);
    float acc[3] = {0.f, 0.f, 0.f};
    if (cnt) {
      tr::Counts cn{0, 0, 0, 0, 0, 0, 0, 0};
      tr::RayKey rk;
      float3 o, d;
      tr::primary_ray(fa, tl.pixel * fa.spp + (lane & (G - 1)), o, d, rk);
      float T = 1.f;
      for (uint32_t j = 0; j < cnt && T > 0.f; ++j) {
        float c[3], a;
        tr::shade_hit<PREC, false, false, true>(
            fa, __float_as_uint(__ldg(&sw.hit[h0 + j].w)) & tr::kIdMask, __ldg(sw.depth + h0 + j), o, d,
            c, a, cn, sw.path + h0 + j, sw.cap);
        const float ta = T * a;
        acc[0] = fmaf(ta, c[0], acc[0]);
        acc[1] = fmaf(ta, c[1], acc[1]);
        acc[2] = fmaf(ta, c[2], acc[2]);
        T *= 1.f - a;
      }
    }
    tr::tile_write(fa, tl, acc, rgb);
  }
}

int sm_count() {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <typename K>
int resident_grid(K kernel) {
  const int sms = sm_count();
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kBlock, 0) != cudaSuccess || per < 1) {
    cudaGetLastError();
    per = 1;
  }
  return sms * per;
}

template <int KMAX, int PREC>
hr_status launch_rounds(hr_ctx* ctx, const FrameArgs& fa, const float4* rect, uint32_t* work,
                        ShadowWork sw, uint32_t rounds, int g_hits, float* rgb, cudaStream_t st) {
  static const int g_paths = resident_grid(k_shadow_paths<PREC>);
  static const int g_shade = resident_grid(k_shadow_shade<PREC>);
  for (uint32_t r = 0; r < rounds; ++r) {
    HR_CUDA(ctx, cudaMemsetAsync(sw.ctr, 0, 8, st));
    k_shadow_hits<KMAX><<<g_hits, kBlock, 0, st>>>(fa, rect, work, sw);
    HR_LAUNCHED(ctx);
    k_shadow_paths<PREC><<<8 * g_paths, kBlock, 0, st>>>(fa, sw);
    HR_LAUNCHED(ctx);
    k_shadow_shade<PREC><<<g_shade, kBlock, 0, st>>>(fa, rect, sw, rgb);
    HR_LAUNCHED(ctx);
  }
  return HR_OK;
}

template <int PREC>
hr_status launch_rounds_k(hr_ctx* ctx, const FrameArgs& fa, const float4* rect, uint32_t* work,
                          const ShadowWork& sw, uint32_t rounds, int g_hits, float* rgb,
                          cudaStream_t st) {
  switch (kmax_for(fa.k)) {
    case 1: return launch_rounds<1, PREC>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st);
    case 2: return launch_rounds<2, PREC>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st);
    case 4: return launch_rounds<4, PREC>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st);
    default: return launch_rounds<8, PREC>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st);
  }
}

}  // namespace

// The tiles that the rounds take; *left says whether tiles can be left over
// (for the one-kernel form: from *work on, where rounds have *begun).  Nothing
// is launched (and *left is set) for the smallest scenes, where the buffers do
// not fit the context's budget, or where a lane traces more than one sample of
// a pixel (more than 32 spp: its hits would need an order of their own).
hr_status launch_shadow_rounds(hr_ctx* ctx, const FrameArgs& fa, int precision, const float4* rect,
                               uint32_t* work, float* rgb, cudaStream_t st, bool* left, bool* begun) {
  *left = true;
  *begun = false;
  if (fa.spp > fa.grp) return HR_OK;
  const uint64_t L = (uint64_t)fa.lights.n;
  if (L * L * L * fa.n_prims <= kOneKernelPrims &&
      (uint64_t)fa.cam.W * fa.cam.H * fa.spp <= kOneKernelSamples)
    return HR_OK;
  const uint64_t worst = (uint64_t)fa.cam.W * fa.cam.H * fa.spp * fa.k;
  const uint64_t per_hit = sizeof(float4) + sizeof(float) + L * sizeof(float4);
  const uint64_t cap = std::min<uint64_t>(worst, kPathBytes / per_hit);
  // every launched warp can be at a tile of 32 lanes and k hits when the round
  // fills up; nothing is added past the worst case
  const int g_hits = 4 * sm_count();
  const uint64_t at_work = (uint64_t)g_hits * kBlock * fa.k;
  if (cap < worst && cap <= at_work) return HR_OK;
  const uint64_t stop = cap < worst ? cap - at_work : worst;
  const WarpGrid all = warp_grid(make_float4(0.f, 0.f, (float)fa.cam.W, (float)fa.cam.H),
                                 (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  const uint64_t tiles = std::min<uint64_t>(cap, all.n);
  const size_t bytes = 64 + cap * per_hit + tiles * sizeof(ShadowTile);
  char* p = nullptr;
  if (scratch(ctx, kScratchPaths, bytes, (void**)&p) != HR_OK) {
    set_error(ctx, HR_OK, "");
    return HR_OK;
  }
  ShadowWork sw{};
  sw.path = reinterpret_cast<float4*>(p);
  sw.hit = sw.path + L * cap;
  sw.tiles = reinterpret_cast<ShadowTile*>(sw.hit + cap);
  sw.depth = reinterpret_cast<float*>(sw.tiles + tiles);
  sw.ctr = reinterpret_cast<uint32_t*>(sw.depth + cap);
  sw.stop = (uint32_t)stop;
  sw.cap = (uint32_t)cap;
  const uint32_t rounds = (uint32_t)std::min<uint64_t>((worst + stop - 1) / stop, kMaxRounds);
  *left = (uint64_t)rounds * stop < worst;
  *begun = true;
  return precision == HR_PREC_FP16
             ? launch_rounds_k<HR_PREC_FP16>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st)
             : launch_rounds_k<HR_PREC_FP32>(ctx, fa, rect, work, sw, rounds, g_hits, rgb, st);
}

}  // namespace hr
