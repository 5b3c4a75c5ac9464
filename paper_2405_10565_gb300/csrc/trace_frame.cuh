// Frame kernel (hot path of hr_render) and its launcher, shared by the two
// translation units that instantiate it without and with shadow rays (so
// that they compile in parallel).
#pragma once

#include <algorithm>

#include "trace_core.cuh"

namespace hr {
namespace {

// Projected scene rectangle of the frame and cleared work counters, once per
// launch (warp 0).  With a tile schedule (fa.sched), the block also picks
// this frame's heavy tiles among the previous frame's candidates (TileSched):
// those whose slowest lane took at least kHeavyRelPct percent of the steps of
// that frame's slowest tile and more than kHeavyMinSteps, at most kHeavyMax
// of them (the heaviest), stored by their pixel origin heaviest first.  The
// previous frame's warp grid is rebuilt from its scene rectangle, which the
// block then replaces with this frame's, and the candidate threshold of this
// frame is set from the previous frame's largest count.  A previous frame of
// another size or spp, or a frame of more than kHeavyTilesPerWarp tiles per
// resident warp, gives no heavy tiles.  One thread per candidate.
constexpr int kRectThreads = (int)kCandMax;
constexpr uint32_t kLongMinPrims = 2048;
__global__ void __launch_bounds__(kRectThreads) k_scene_rect(const FrameArgs fa, float4* rect,
                                                             uint32_t* work) {
  if (threadIdx.x < 32) tr::scene_rect_warp(fa, rect);
  if (threadIdx.x == 0) *work = 0u;
  if (fa.lw.words && threadIdx.x < 4) fa.lw.ctr[threadIdx.x] = 0u;
  TileSched* sc = fa.sched;
  if (!sc) return;
  __shared__ uint32_t s_hist[256], s_cut, s_n, s_kept;
  __shared__ uint32_t s_tile[kHeavyMax], s_steps[kHeavyMax];
  const uint32_t tid = threadIdx.x;
  const bool have = sc->prev_n > 0 && sc->prev_W == (uint32_t)fa.cam.W &&
                    sc->prev_H == (uint32_t)fa.cam.H && sc->prev_grp == fa.grp;
  const uint32_t M = have ? sc->max_steps : 0u;
  if (tid == 0) {
    s_cut = 0u;
    s_n = 0u;
  }
  if (tid < 256) s_hist[tid] = 0u;
  __syncthreads();
  const float4 rc = *rect;  // written by warp 0 before the barrier
  const WarpGrid g = warp_grid(rc, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  const bool allow = (uint64_t)g.n <= (uint64_t)kHeavyTilesPerWarp * fa.frame_warps;
  const uint32_t nc = have && allow ? min(sc->cand_n, kCandMax) : 0u;
  const bool mine = tid < nc;
  const uint32_t c = mine ? sc->cand_steps[tid] : 0u;
  const uint32_t ct = mine ? sc->cand_tile[tid] : 0u;
  // steps in [lo, M] binned into 256 bins; the cut is the highest bin with
  // at least kHeavyMax candidates at or above it (else bin 0), and those
  // past kHeavyMax in the cut's bin are left out
  const uint32_t lo = max((uint32_t)((uint64_t)M * kHeavyRelPct / 100u), kHeavyMinSteps + 1);
  const uint32_t span = M >= lo ? M - lo + 1 : 1u;
  const bool cand = mine && c >= lo && ct < sc->prev_n;
  const uint32_t b = cand ? (uint32_t)((uint64_t)(min(c, M) - lo) * 256u / span) : 0u;
  if (cand) atomicAdd(&s_hist[b], 1u);
  __syncthreads();
  // suffix sums of the histogram (Hillis-Steele over 256 bins)
  for (uint32_t o = 1; o < 256; o <<= 1) {
    uint32_t v = 0;
    if (tid < 256) v = s_hist[tid] + (tid + o < 256 ? s_hist[tid + o] : 0u);
    __syncthreads();
    if (tid < 256) s_hist[tid] = v;
    __syncthreads();
  }
  if (tid < 256 && s_hist[tid] >= kHeavyMax) atomicMax(&s_cut, tid);
  __syncthreads();
  const uint32_t cut = s_cut;
  // the bins above the cut first (fewer than kHeavyMax candidates), then the cut's
  for (int pass = 0; pass < 2; ++pass) {
    if (cand && (pass == 0 ? b > cut : b == cut)) {
      const uint32_t k = atomicAdd(&s_n, 1u);
      if (k < kHeavyMax) {
        s_tile[k] = ct;
        s_steps[k] = c;
      }
    }
    __syncthreads();
  }
  const uint32_t listed = min(s_n, kHeavyMax);
  if (tid < 32) {
    // a tile listed several times (by parts of it) stays with its heaviest part
    const bool mine_listed = tid < listed;
    const uint32_t t = mine_listed ? s_tile[tid] : 0u, steps = mine_listed ? s_steps[tid] : 0u;
    bool stays = mine_listed;
#pragma unroll 4
    for (uint32_t k = 0; k < kHeavyMax; ++k) {
      const uint32_t kt = __shfl_sync(0xffffffffu, t, k), ks = __shfl_sync(0xffffffffu, steps, k);
      if (k < listed && kt == t && (ks > steps || (ks == steps && k < tid))) stays = false;
    }
    const unsigned heavy = __ballot_sync(0xffffffffu, stays);
    uint32_t r = 0;  // heaviest first (ties by tile index): rank by counting
#pragma unroll 4
    for (uint32_t k = 0; k < kHeavyMax; ++k) {
      const uint32_t kt = __shfl_sync(0xffffffffu, t, k), ks = __shfl_sync(0xffffffffu, steps, k);
      r += ((heavy >> k) & 1u) && (ks > steps || (ks == steps && kt < t));
    }
    if (stays) {
      const WarpGrid pg = warp_grid(sc->prev_rect, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
      sc->heavy[r] = (pg.x0 + (t % pg.nx) * pg.wtw) | ((pg.y0 + (t / pg.nx) * pg.wth) << 16);
    }
    if (tid == 0) s_kept = (uint32_t)__popc(heavy);
  }
  __syncthreads();  // the previous frame's candidates and grid are no longer read
  if (tid == 0) {
    sc->n_heavy = s_kept;
    sc->grp = fa.grp;
    sc->thresh = lo;
    sc->max_steps = 0u;
    sc->cand_n = 0u;
    sc->prev_rect = rc;
    sc->prev_n = g.n;
    sc->prev_W = (uint32_t)fa.cam.W;
    sc->prev_H = (uint32_t)fa.cam.H;
    sc->prev_grp = fa.grp;
  }
}

// Steps (node visits and tests) that a ray may take in k_frame, by the tiles
// per resident warp.  Finishing a ray with a whole warp costs several times
// the warp time of its share in a full warp, so it pays only where a long walk
// would outlast the frame: with less than a tile per warp that is any walk
// longer than usual, with many tiles only walks many times as long.  Budgets
// of 64, 128, 256, 512 steps and none: the far view of the full head (1.6
// tiles per warp; 55 steps a ray on average, 570 at most) 1.47, 1.28, 1.37,
// 1.51, 1.63 ms a call; the curled clusters (4.8; 133, 583) 2.58, 2.55, 1.83,
// 1.59, 1.39; a thumbnail (0.09) 0.29, 0.32, 0.38, 0.38, 0.40; the 4K frame of
// straight hair (39; 100, 10,600) 11.0, 11.1, 10.0, 9.9, 14.5; the close view
// (55; 44, 1,200) 6.2, 4.4, 3.91, 3.85, 3.83.
// Below a tile per warp, where parts of tiles are handed out, 40, 64 and 96
// steps: 262, 271, 277 us at 0.09 tiles per warp, 379, 360, 361 at 0.19,
// 760, 739, 728 and 301, 292, 304 at half a tile, 341, 327, 335 at 0.9.
__device__ __forceinline__ int step_budget(uint32_t tiles, uint32_t warps) {
  const float per = (float)tiles / (float)warps;
  return (int)fminf(fmaxf(64.f * per * per, per < 0.125f ? 40.f : 64.f), 1024.f);
}

// Small frames hand out parts of a tile, 2^n of them of whole pixels, as far as
// there are warps for them: a warp's lanes go through nodes and leaves
// together, so the fewer rays share a warp, the sooner its last one is done
// (a 94 x 70 frame of 2,812 strands 387 us a call whole, 379 in parts and 360
// with the budget that this allows; with shadow rays, 203 strands at 78 x 48,
// 132 and 86).
__device__ __forceinline__ uint32_t tile_split(uint32_t tiles, uint32_t warps, uint32_t grp) {
  uint32_t ls = 0;
  while ((grp << (ls + 1)) <= 32u && ((uint64_t)tiles << (ls + 1)) <= warps) ++ls;
  return ls;
}

// Persistent frame kernel.  The image has been cleared to background; the
// warp tiles (32 / grp pixels each) that overlap the projected scene rectangle
// are handed out one at a time through an atomic counter, so the few tiles
// that see hair spread over every warp of the GPU and a warp that drew cheap
// tiles takes more.  With a schedule, the hand-outs start with the heavy tiles
// (TileSched); rays over the budget of steps go to k_long_rays.  No warp ever
// waits for another.
template <int KMAX, int PREC, bool COUNT, bool SHADOW>
__global__ void __launch_bounds__(kBlock, SHADOW ? 1 : tr::kTraceBlocks)
    k_frame(const FrameArgs fa, const float4* __restrict__ rect_p, uint32_t* work,
            float* __restrict__ rgb) {
  constexpr bool LONG = !COUNT && !SHADOW;
  __shared__ tr::RayMem<KMAX, kBlock> rm;
  const float4 rect = *rect_p;
  const WarpGrid g = warp_grid(rect, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  tr::Counts cn{0, 0, 0, 0, 0, 0, 0, 0};
  bool overflow = false;
  const uint32_t lane = threadIdx.x & 31;
  if (COUNT && fa.tile_log && blockIdx.x == 0 && threadIdx.x == 0) *fa.tile_count = g.n;
  TileSched* sc = LONG ? fa.sched : nullptr;
  const uint32_t nh = sc && sc->grp == fa.grp ? min(sc->n_heavy, kHeavyMax) : 0u;
  const uint32_t thresh = sc ? sc->thresh : 0u;
  uint32_t wmax = 0;  // the warp's largest tile step count
  const int budget = LONG && fa.lw.words ? step_budget(g.n, fa.frame_warps) : 0x7fffffff;
  const uint32_t ls = COUNT ? 0u : tile_split(g.n, fa.frame_warps, fa.grp);
  for (;;) {
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(work, 1u);
    t = __shfl_sync(0xffffffffu, t, 0);
    uint32_t x0, y0;
    const unsigned part = (0xffffffffu >> (32u - (32u >> ls))) << ((t & ((1u << ls) - 1u)) * (32u >> ls));
    t >>= ls;
    if (t < nh) {  // a tile of the previous frame's grid; one that is not of this grid is skipped
      const uint32_t xy = sc->heavy[t];
      x0 = xy & 0xffffu, y0 = xy >> 16;
      const uint32_t gx = (x0 - g.x0) / g.wtw, gy = (y0 - g.y0) / g.wth;
      if (x0 < g.x0 || y0 < g.y0 || (x0 - g.x0) % g.wtw || (y0 - g.y0) % g.wth || gx >= g.nx ||
          gy * g.nx + gx >= g.n)
        continue;
      t = gy * g.nx + gx;
    } else {
      t -= nh;
      if (t >= g.n) break;
      x0 = g.x0 + (t % g.nx) * g.wtw, y0 = g.y0 + (t / g.nx) * g.wth;
      if (nh && __any_sync(0xffffffffu, lane < nh && sc->heavy[lane] == (x0 | (y0 << 16)))) continue;
    }
    const uint32_t steps0 = cn.steps;
    uint64_t t0 = 0;
    uint32_t nodes0 = 0, tests0 = 0;
    if (COUNT && fa.tile_log) {
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
      nodes0 = cn.nodes;
      tests0 = cn.tests;
    }
    tr::render_warp_tile<KMAX, PREC, COUNT, SHADOW, LONG>(fa, rm, x0, y0, g.wtw, rect, budget,
                                                          rgb, cn, overflow, part);
    if (sc) {
      // the tile's slowest-lane steps: the warp's maximum, and a candidate for
      // the next frame's heavy tiles at or above the threshold
      const uint32_t st = __reduce_max_sync(0xffffffffu, cn.steps - steps0);
      wmax = max(wmax, st);
      if (lane == 0 && st >= thresh && __ldcg(&sc->cand_n) < kCandMax) {  // no atomics once full
        const uint32_t k = atomicAdd(&sc->cand_n, 1u);
        if (k < kCandMax) {
          sc->cand_tile[k] = t;
          sc->cand_steps[k] = st;
        }
      }
    }
    if (COUNT && fa.tile_log) {
      const uint32_t dn = __reduce_max_sync(0xffffffffu, cn.nodes - nodes0);
      const uint32_t dt = __reduce_max_sync(0xffffffffu, cn.tests - tests0);
      uint64_t t1;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
      if (lane == 0 && t < fa.tile_cap) {
        uint32_t sm;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
        fa.tile_log[t] = hr_tile_record{t0, t1, t, sm, dn, dt};
      }
    }
  }
  if (sc && lane == 0 && wmax) atomicMax(&sc->max_steps, wmax);
  if (COUNT) tr::flush_counts(fa, cn);
  if (overflow) atomicAdd(fa.overflow, 1u);
}

// The rays put aside, a warp each.  Nodes come off the warp's stack up to 32
// at a time, one a lane, the nearest subtrees first; the boxes they hit go
// back on it, a lane's nearer child above its farther one and nearer lanes'
// above farther ones', and hit leaves onto a list that is tested as soon as it
// fills a warp (or no node is left).  Hits are kept one after the other in
// lane order, so a ray's result does not depend on when or where it is
// finished.  The last ray of a tile shades the tile's rays (one a lane) and
// stores it.
constexpr int kLongStack = 512;  // one node at a time once fewer than 64 places are left
constexpr int kLongLeaves = 96;
template <int KMAX, int PREC>
__global__ void __launch_bounds__(kBlock, 6)
    k_long_rays(const FrameArgs fa, const float4* __restrict__ rect_p, float* __restrict__ rgb) {
  constexpr int kWarps = kBlock / 32;
  __shared__ tr::RayMem<KMAX, kWarps> rm;
  __shared__ int s_node[kWarps][kLongStack];
  __shared__ uint32_t s_leaf[kWarps][kLongLeaves];
  const uint32_t lane = threadIdx.x & 31, c = threadIdx.x >> 5, k = fa.k;
  const uint32_t above = lane == 31 ? 0u : 0xffffffffu << (lane + 1);
  const uint32_t n_rays = min(__ldcg(fa.lw.ctr), fa.lw.rays_max);
  const float4 rect = *rect_p;
  const WarpGrid g = warp_grid(rect, (uint32_t)fa.cam.W, (uint32_t)fa.cam.H, fa.grp);
  tr::Counts cn{0, 0, 0, 0, 0, 0, 0, 0};
  int* nodes = s_node[c];
  uint32_t* leaves = s_leaf[c];
  // lane 0 takes the next ray while the warp works on this one
  constexpr uint32_t kNone = 0xffffffffu, kEnd = 0xfffffffeu;
  auto take = [&]() {
    const uint32_t i = atomicAdd(fa.lw.ctr + 3, 1u);
    return i < n_rays ? __ldg(fa.lw.ray_at + i) : kEnd;
  };
  uint32_t following = lane == 0 ? take() : 0u;
  for (;;) {
    const uint32_t at = __shfl_sync(0xffffffffu, following, 0);
    if (at == kEnd) break;
    if (lane == 0) following = take();
    if (at == kNone) continue;
    uint32_t* r = fa.lw.pool + at;
    tr::LongTile& lt = fa.lw.tiles[r[0]];
    const uint32_t xy = lt.xy, owner = r[1] & 0xffu;
    int n = (int)(r[1] >> 8);
    const uint32_t x0 = xy & 0xffffu, y0 = xy >> 16;
    float tcut = __uint_as_float(r[2]), errmax = __uint_as_float(r[3]);
    for (uint32_t j = lane; j < k; j += 32) {
      rm.t[j][c] = __uint_as_float(r[tr::kLongHead + j]);
      rm.tr[j][c] = __uint_as_float(r[tr::kLongHead + k + j]);
      rm.id[j][c] = r[tr::kLongHead + 2 * k + j];
    }
    for (int j = (int)lane; j < n; j += 32) nodes[j] = (int)r[tr::kLongHead + 3 * k + j];
    float3 o, d;
    {
      const uint32_t p = owner / fa.grp;
      const uint64_t pixel = (uint64_t)(y0 + p / g.wtw) * (uint32_t)fa.cam.W + x0 + p % g.wtw;
      tr::RayKey rk;
      tr::primary_ray(fa, pixel * fa.spp + (owner & (fa.grp - 1)), o, d, rk);
      if (lane == 0) tr::ray_store(rm, c, o, d, rk);
    }
    __syncwarp();
    const tr::Slabs sl = tr::ray_slabs(fa, o, d);
    const float pad = 2.f * tr::kTieRel * rm.s_off[c], M = rm.M[c];
    int nl = 0;
    while (n > 0 || nl > 0) {
      if (n > 0 && nl < 32) {
        const int m = max(1, min(min(n, 32), kLongStack - 64 - n));
        const bool mine = (int)lane < m;
        const int node = mine ? nodes[n - 1 - (int)lane] : tr::kDone;
        n -= m;
        __syncwarp();
        bool h0 = false, h1 = false, swap = false;
        int c0 = 0, c1 = 0;
        if (node >= 0) {
          const float tb = fmaf(tcut + errmax, 1.f + 2.f * tr::kTieRel, pad);
          const tr::Children ch =
              sl.wide ? tr::node_test<true>(fa, sl, node, tb) : tr::node_test<false>(fa, sl, node, tb);
          h0 = ch.h0, h1 = ch.h1;
          swap = ch.a1 < ch.a0;
          c0 = ch.c0, c1 = ch.c1;
        } else if (mine) {  // a leaf that was pending when the ray was put aside
          h0 = true;
          c0 = node;
        }
        const bool n0 = h0 && c0 >= 0, n1 = h1 && c1 >= 0;
        const unsigned b0 = __ballot_sync(0xffffffffu, n0), b1 = __ballot_sync(0xffffffffu, n1);
        int q = n + __popc(b0 & above) + __popc(b1 & above);
        if (n0 && n1) {
          nodes[q] = swap ? c0 : c1;
          nodes[q + 1] = swap ? c1 : c0;
        } else if (n0 || n1) {
          nodes[q] = n0 ? c0 : c1;
        }
        n += __popc(b0) + __popc(b1);
        const bool l0 = h0 && c0 < 0, l1 = h1 && c1 < 0;
        const unsigned e0 = __ballot_sync(0xffffffffu, l0), e1 = __ballot_sync(0xffffffffu, l1);
        q = nl + __popc(e0 & above) + __popc(e1 & above);
        if (l0) leaves[q++] = (uint32_t)~c0;
        if (l1) leaves[q] = (uint32_t)~c1;
        nl += __popc(e0) + __popc(e1);
        __syncwarp();
        continue;
      }
      const int ml = min(nl, 32);
      const bool leaf = (int)lane < ml;
      const uint32_t id = leaf ? leaves[nl - 1 - (int)lane] : 0u;
      nl -= ml;
      float th = 0.f, terr = 0.f;
      int hit = tr::kMiss;
      if (leaf)
        hit = tr::intersect32(fa, id, __ldg(fa.prim_uv + 2 * (size_t)id),
                              __ldg(fa.prim_uv + 2 * (size_t)id + 1), o, d, M, tcut + errmax, th, terr);
      unsigned hits = __ballot_sync(0xffffffffu, hit != tr::kMiss);
      while (hits) {
        const int l = __ffs(hits) - 1;
        hits &= hits - 1;
        if ((int)lane == l && th - terr <= tcut + errmax)
          tr::keep_hit<KMAX, kWarps, false>(fa, rm, c, id, hit, th, terr, tcut, errmax, cn);
        __syncwarp();
        tcut = __shfl_sync(0xffffffffu, tcut, l);
        errmax = __shfl_sync(0xffffffffu, errmax, l);
      }
      __syncwarp();
    }
    for (uint32_t j = lane; j < k; j += 32) {
      r[tr::kLongHead + j] = __float_as_uint(rm.t[j][c]);
      r[tr::kLongHead + 2 * k + j] = rm.id[j][c];
    }
    __syncwarp();
    uint32_t left = 0;
    if (lane == 0) {
      __threadfence();
      left = atomicSub(&lt.left, 1u);
    }
    left = __shfl_sync(0xffffffffu, left, 0);
    if (left != 1u) continue;
    __threadfence();
    // the tile's last ray: shade the lanes put aside and store the tile
    tr::TileLane tl = tr::tile_lane(fa, x0, y0, g.wtw, rect);
    tl.inside = (lt.part >> lane) & 1u;
    float acc[3] = {__ldcg(&lt.acc[0][lane]), __ldcg(&lt.acc[1][lane]), __ldcg(&lt.acc[2][lane])};
    if ((lt.lanes >> lane) & 1u) {
      const uint32_t* rec = fa.lw.pool + lt.at[lane];
      uint32_t id[KMAX];
      float t[KMAX];
#pragma unroll
      for (int j = 0; j < KMAX; ++j) {
        t[j] = j < (int)k ? __uint_as_float(__ldcg(rec + tr::kLongHead + j)) : 0.f;
        id[j] = j < (int)k ? __ldcg(rec + tr::kLongHead + 2 * k + j) : 0u;
      }
      tr::RayKey rk;
      float3 ro, rd;
      tr::primary_ray(fa, tl.pixel * fa.spp + (lane & (fa.grp - 1)), ro, rd, rk);
      tr::shade_hits<PREC, false, false>(fa, t, nullptr, id, 1u, k, ro, rd, acc, cn);
    }
    tr::tile_write(fa, tl, acc, rgb);
  }
}

template <int KMAX, int PREC, bool COUNT, bool SHADOW>
int frame_grid() {
  static int grid = 0;
  if (!grid) {
    int dev = 0, sms = 1, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_frame<KMAX, PREC, COUNT, SHADOW>, kBlock,
                                                      0) != cudaSuccess) {
      cudaGetLastError();
      per = 4;
    }
    grid = sms * (per > 0 ? per : 1);
  }
  return grid;
}

// Room for the rays put aside: up to 64 MB of records, less for small images;
// no words (no ray is put aside) where it does not fit the context's memory
// budget, for more than 32 spp and for small scenes, whose walks are short.
inline void long_work(hr_ctx* ctx, FrameArgs& fa) {
  fa.lw = LongWork{};
  if (fa.spp > fa.grp || fa.n_prims < kLongMinPrims) return;
  const uint64_t samples = (uint64_t)fa.cam.W * fa.cam.H * fa.spp;
  const uint64_t words = std::min<uint64_t>(16u << 20, samples * 16 + 4096);
  const uint64_t rays = words / (tr::kLongHead + 8), tiles = std::min<uint64_t>(rays, 65536);
  char* p = nullptr;
  if (scratch(ctx, kScratchLong, 64 + tiles * sizeof(tr::LongTile) + (words + rays) * 4, (void**)&p) != HR_OK) {
    set_error(ctx, HR_OK, "");
    return;
  }
  fa.lw.tiles = reinterpret_cast<tr::LongTile*>(p + 64);
  fa.lw.ctr = reinterpret_cast<uint32_t*>(p);
  fa.lw.pool = reinterpret_cast<uint32_t*>(fa.lw.tiles + tiles);
  fa.lw.ray_at = fa.lw.pool + words;
  fa.lw.words = (uint32_t)words;
  fa.lw.rays_max = (uint32_t)rays;
  fa.lw.tiles_max = (uint32_t)tiles;
}

template <int KMAX, int PREC, bool SHADOW>
hr_status launch_k(hr_ctx* ctx, const FrameArgs& fa, bool count, float* rgb, cudaStream_t st) {
  const uint32_t tiles = tiles_for(fa.cam.W, fa.cam.H, fa.spp);
  float4* rect = nullptr;
  HR_TRY(scratch(ctx, 47, 2 * sizeof(float4), (void**)&rect));
  uint32_t* work = reinterpret_cast<uint32_t*>(rect + 1);
  HR_CUDA(ctx, cudaMemsetAsync(rgb, 0, (size_t)fa.cam.W * fa.cam.H * 3 * sizeof(float), st));
  // the counting kernel keeps the plain hand-out order (its tile log is indexed
  // by it), and so do frames with shadow rays
  FrameArgs f = fa;
  if (count || SHADOW)
    f.sched = nullptr;
  else
    long_work(ctx, f);
  f.frame_warps = (uint32_t)frame_grid<KMAX, PREC, false, SHADOW>() * (kBlock / 32);
  k_scene_rect<<<1, kRectThreads, 0, st>>>(f, rect, work);
  HR_LAUNCHED(ctx);
  if (count) {
    const int g = (int)std::min<uint32_t>(tiles, frame_grid<KMAX, PREC, true, SHADOW>());
    k_frame<KMAX, PREC, true, SHADOW><<<g, kBlock, 0, st>>>(f, rect, work, rgb);
  } else {
    if (SHADOW) {  // the one-kernel form takes what the rounds leave over
      bool left = true, begun = false;
      HR_TRY(launch_shadow_rounds(ctx, f, PREC, rect, work, rgb, st, &left, &begun));
      if (!left) return HR_OK;
      if (begun) f.frame_warps = 0;  // *work counts whole tiles: no parts
    }
    // up to 32 parts a tile, four warps a block
    const int g = (int)std::min<uint64_t>(8ull * tiles, (uint64_t)frame_grid<KMAX, PREC, false, SHADOW>());
    k_frame<KMAX, PREC, false, SHADOW><<<g, kBlock, 0, st>>>(f, rect, work, rgb);
  }
  HR_LAUNCHED(ctx);
  if (f.lw.words) {
    static const int long_grid = [] {
      int dev = 0, sms = 1;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      return 6 * sms;
    }();
    k_long_rays<KMAX, PREC><<<long_grid, kBlock, 0, st>>>(f, rect, rgb);
    HR_LAUNCHED(ctx);
  }
  return HR_OK;
}

template <int PREC, bool SHADOW>
hr_status launch_p(hr_ctx* ctx, const FrameArgs& fa, bool count, float* rgb, cudaStream_t st) {
  switch (kmax_for(fa.k)) {
    case 1: return launch_k<1, PREC, SHADOW>(ctx, fa, count, rgb, st);
    case 2: return launch_k<2, PREC, SHADOW>(ctx, fa, count, rgb, st);
    case 4: return launch_k<4, PREC, SHADOW>(ctx, fa, count, rgb, st);
    default: return launch_k<8, PREC, SHADOW>(ctx, fa, count, rgb, st);
  }
}

template <bool SHADOW>
hr_status launch_frame_t(hr_ctx* ctx, const FrameArgs& fa, int precision, bool count,
                         float* rgb_dev, cudaStream_t st) {
  if (fa.cam.W <= 0 || fa.cam.H <= 0) return HR_OK;
  return precision == HR_PREC_FP16 ? launch_p<HR_PREC_FP16, SHADOW>(ctx, fa, count, rgb_dev, st)
                                   : launch_p<HR_PREC_FP32, SHADOW>(ctx, fa, count, rgb_dev, st);
}

}  // namespace
}  // namespace hr
