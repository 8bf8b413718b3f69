// render.cu -- wavefront MARS path tracer.  Per depth wave d (rays in
// [base[d], base[d] + count[d]) of the tile's arena):
//
//   k_trace  (wave d)  closest hit of every ray (camera rays for d = 1)
//   k_shade  (wave d)  emission reached by the ray, weighted against NEE
//                      (multi-sample balance heuristic, Sec. 3.1); at a vertex
//                      x_d with d <= D-1 the sampling half of the secondary
//                      estimator: counts beta_t from the cache (T(x)/I_px x q,
//                      three cases, clamp; Sec. 3.1 "Optimization", Sec. 4.1),
//                      Alg. 1, NEE samples written as shadow rays, BSDF / guided
//                      children appended to wave d+1 (warp-aggregated
//                      allocation)
//   k_shadow (wave d)  one thread per NEE shadow ray: any hit zeroes the sample
//
// then deepest first
//
//   k_reverse (wave d) every ray's sample value
//                        <L_r,t> = f|cos|/p_t (Le w_dir + w_ind <L_r(child vertex)>)
//                      and cost (rays in its subtree, counting itself), the
//                      vertex's <L_r> = sum_t 1/beta_t sum_s <L_r,t> (Sec. 3.1
//                      "Secondary estimator"), and the local statistics of
//                      Sec. 4.1 "Local estimates" (per cell and technique: n,
//                      sum v, sum v^2, sum cost), pre-reduced over runs of equal
//                      cells in a warp before float64 atomics.
//
// A tile whose arena overflowed commits nothing.
#include <algorithm>

#include "wave.cuh"

namespace mars {

namespace {

__global__ void k_tile_init(DevCounters* ctr, const IterArgs* __restrict__ itp) {
  const unsigned long long n0 = (unsigned long long)(itp->tile_end - itp->tile_begin);
  const int t = threadIdx.x;
  if (t < MAXD + 2) {
    ctr->base[t] = 0;
    ctr->count[t] = (t == 1) ? n0 : 0ull;
    ctr->sbase[t] = 0;
    ctr->scount[t] = 0;
    ctr->slcount[t] = 0;
    ctr->lbase[t] = 0;
    ctr->lcount[t] = 0;
    ctr->vcount[t] = 0;
    ctr->trace_next[t] = 0;
    ctr->shadow_next[t] = 0;
  }
  if (t == 0) {
    ctr->overflow = 0;
    ctr->demand = n0;
  }
}

// One warp, lane d - 1 for depth wave d: the wave's counters are loaded side by
// side (one thread that added them up took a round trip to memory after another,
// 7 us at D = 12).
__global__ void k_tile_finish(DevCounters* ctr, unsigned int* tile_status, const IterArgs* __restrict__ itp, int D) {
  const int lane = threadIdx.x, d = lane + 1;
  const bool on = d <= D;
  const unsigned overflow = ctr->overflow;
  const unsigned long long cnt = on ? ctr->count[d] : 0ull;
  unsigned long long v[5] = {cnt, on ? ctr->scount[d] : 0ull, on ? ctr->slcount[d] : 0ull, on ? ctr->lcount[d] : 0ull,
                             on ? ctr->vcount[d] : 0ull};
  const unsigned long long wave_total = on ? ctr->wave_total[d] : 0ull;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] += __shfl_xor_sync(FULL, v[k], off);
  }
  if (!overflow && on) ctr->wave_total[d] = wave_total + cnt;
  if (lane != 0) return;
  // every ray of the tile, drawn by whichever kernels: the waves lie one after the
  // other, and k_tail counts its rays by depth without placing its waves
  ctr->demand = v[0];
  if (!overflow) {
    // fire-and-forget additions; nobody else writes these while the tile ends
    atomicAdd(&ctr->entries, v[0]);
    atomicAdd(&ctr->shadow_entries, v[1]);
    atomicAdd(&ctr->shadow_traced, v[2]);
    atomicAdd(&ctr->light_entries, v[3]);
    atomicAdd(&ctr->light_vertex_entries, v[4]);
  }
  tile_status[itp->tile_slot] = overflow;
  if (overflow) ctr->any_overflow = 1;
}

// Totals of a second tile lane's counters into the first's (added, then cleared
// in the source, so that a later merge adds only what came after).  One warp; a
// lane moves the counters of its number, so that they are loaded side by side.
__global__ void k_merge_lanes(DevCounters* dst, DevCounters* src) {
  const int lane = threadIdx.x;
  unsigned long long* const from[] = {&src->shadow_entries, &src->shadow_traced, &src->rays, &src->vertices,
                                      &src->est_vertices, &src->entries, &src->light_entries,
                                      &src->light_vertex_entries, &src->light_rays, &src->conn_rays};
  unsigned long long* const to[] = {&dst->shadow_entries, &dst->shadow_traced, &dst->rays, &dst->vertices,
                                    &dst->est_vertices, &dst->entries, &dst->light_entries,
                                    &dst->light_vertex_entries, &dst->light_rays, &dst->conn_rays};
  constexpr int N = sizeof(from) / sizeof(from[0]);
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (lane == k) {
      const unsigned long long v = *from[k];
      *from[k] = 0;
      atomicAdd(to[k], v);
    }
  if (lane < MAXD + 2) {
    const unsigned long long v = src->wave_total[lane];
    src->wave_total[lane] = 0;
    atomicAdd(&dst->wave_total[lane], v);
  }
  if (lane >= 20 && lane < 28) {
    const int k = (lane - 20) >> 2, q = (lane - 20) & 3;
    const unsigned long long v = src->trace_work[k][q];
    src->trace_work[k][q] = 0;
    atomicAdd(&dst->trace_work[k][q], v);
  }
  if (lane >= 28 && lane < 28 + NT) {
    const int t = lane - 28;
    const double v = src->sum_beta[t];
    src->sum_beta[t] = 0.0;
    atomicAdd(&dst->sum_beta[t], v);
  }
  if (lane == 31) {
    if (src->any_overflow) dst->any_overflow = 1;
    src->any_overflow = 0;
    if (src->check_flags) atomicOr(&dst->check_flags, src->check_flags);
    src->check_flags = 0;
    atomicMax(&dst->demand, src->demand);
  }
}

template <int MINB>
__global__ void __launch_bounds__(MAX_WAVE_THREADS, MINB) k_trace(const DevScene s, const DevCache c, const Arena a,
                                                         const IterArgs* __restrict__ itp, const int d) {
  const IterArgs it = *itp;
  DevCounters* ctr = c.ctr;
  // after an overflow some slots of this wave were never written: stop, the
  // tile is re-rendered in smaller pieces
  if (overflowed(ctr)) return;
  extern __shared__ RayStage ray_stage[];
  const Wave w = wave_of(ctr, a, d);
  TraceWork tw;
  closest_hits(s, c, a, it, WaveSlots{w.base, (uint32_t)it.tile_begin, d == 1}, (unsigned)w.n,
               d == 1 ? 0u : (unsigned)w.n, &ctr->trace_next[d],
               (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5,
               ray_stage + (threadIdx.x >> 5), tw);
  flush_work(tw, ctr->trace_work[0], ctr);
}

// a wave of the tile in the whole arena, allocated from by every block of the grid
struct GridWave {
  using Index = unsigned long long;
  static constexpr bool MIXED = false;
  WaveSlots slots;
  Index n;                        // the wave's rays
  Index base_next, sbase, lbase;  // first slots of its children, NEE samples and light connection samples
  Index cap, scap, lcap;          // ends of the regions
  Index first, stride;            // the block's first ray of the wave, and its step
  DevCounters* ctr;
  int d;
  __device__ __forceinline__ void alloc(int te, int ts, int tl, Index b[3]) {
    b[0] = te > 0 ? atomicAdd(&ctr->count[d + 1], (Index)te) : 0;
    b[1] = ts > 0 ? atomicAdd(&ctr->scount[d], (Index)ts) : 0;
    b[2] = tl > 0 ? atomicAdd(&ctr->lcount[d], (Index)tl) : 0;
  }
  __device__ __forceinline__ Index list(int n_) { return atomicAdd(&ctr->slcount[d], (Index)n_); }
  __device__ __forceinline__ void overflow() { atomicOr(&ctr->overflow, OVER_ARENA); }
};

template <int MINB, bool BD>
__global__ void __launch_bounds__(MAX_WAVE_THREADS, MINB) k_shade(const DevScene s, const DevCache c, const Arena a,
                                                         const IterArgs* __restrict__ itp, const int d) {
  const IterArgs it = *itp;
  DevCounters* ctr = c.ctr;
  // block-level allocation synchronises the block: decide the early exit once
  // per block (other blocks may raise the overflow flag meanwhile)
  __shared__ unsigned int blk_exit;
  __shared__ ShadeBlock<unsigned long long> blk;
  extern __shared__ ShadeWarpCtx shade_ctx[];
  if (threadIdx.x == 0) blk_exit = ctr->overflow;
  __syncthreads();
  if (blk_exit) return;
  const Wave w = wave_of(ctr, a, d);
  const unsigned long long cnt = ctr->count[d];
  GridWave io;
  io.slots = WaveSlots{w.base, (uint32_t)it.tile_begin, d == 1};
  io.n = w.n;
  io.base_next = w.base + cnt < a.cap ? w.base + cnt : a.cap;
  io.sbase = d == 1 ? 0ull : ctr->sbase[d - 1] + ctr->scount[d - 1];
  io.lbase = d == 1 ? 0ull : ctr->lbase[d - 1] + ctr->lcount[d - 1];
  io.cap = a.cap;
  io.scap = a.scap;
  io.lcap = a.lcap;
  io.first = blockIdx.x * (unsigned long long)blockDim.x;
  io.stride = gridDim.x * (unsigned long long)blockDim.x;
  io.ctr = ctr;
  io.d = d;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctr->base[d + 1] = io.base_next;
    ctr->sbase[d] = io.sbase;
    if (BD) ctr->lbase[d] = io.lbase;
  }
  shade_wave<BD>(s, c, a, it, d, io, shade_ctx + (threadIdx.x >> 5), blk);
}

// ----------------------------------------------------------------- shadow
// the listed shadow rays of the waves d..d1: SH0, SH1[sbase, sbase + slcount) of
// each (at most scount of them), each with the slot of its sample's value
template <int MINB>
__global__ void __launch_bounds__(MAX_WAVE_THREADS, MINB) k_shadow(const DevScene s, const DevCache c, const Arena a,
                                                           const int d, const int d1) {
  DevCounters* ctr = c.ctr;
  if (overflowed(ctr)) return;
  extern __shared__ RayStage ray_stage[];
  TraceWork tw;
  for (int e = d; e <= d1; ++e) {
    const unsigned long long sb = ctr->sbase[e], sl = ctr->slcount[e];
    const unsigned long long n = sl < a.scap - sb ? sl : a.scap - sb;
    if (n > 0)
      shadow_hits(s, c, a, sb, (unsigned)n, &ctr->shadow_next[e], (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                  (gridDim.x * blockDim.x) >> 5, ray_stage + (threadIdx.x >> 5), tw);
  }
  flush_work(tw, ctr->trace_work[1], ctr);
}

template <int MINB, bool BD>
__global__ void __launch_bounds__(MAX_WAVE_THREADS, MINB) k_reverse(const DevScene s, const DevCache c, const Arena a,
                                                             const IterArgs* __restrict__ itp, const int d) {
  const IterArgs it = *itp;
  if (c.ctr->overflow) return;  // the tile is re-rendered; commit nothing
  const Wave w = wave_of(c.ctr, a, d);
  const unsigned long long gw = (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) >> 5;
  const unsigned long long nw = (gridDim.x * (unsigned long long)blockDim.x) >> 5;
  RevSums acc;
  reverse_wave<BD, unsigned long long>(s, c, a, it, WaveSlots{w.base, (uint32_t)it.tile_begin, d == 1}, w.n, gw * 32,
                                       nw * 32, acc);
  flush_sums(c, acc, BD || (c.techniques & MARS_TECH_GUIDED));
}

size_t trace_smem(int threads) { return (size_t)(threads / 32) * sizeof(RayStage); }
size_t shade_smem(int threads) { return (size_t)(threads / 32) * sizeof(ShadeWarpCtx); }

// Register-cap variants of every wave kernel, compiled with
// __launch_bounds__(256, MINB): trace and shadow 64 or 40 registers, shade 80 or
// 64, reverse the compiler's choice (110), 80 or 64.  Variant 0, what a cache
// starts with, is the 64, 80 and 64 register one for trace, shade and shadow:
// uncapped they take 88, 144 and 77, and the kernels, which wait on loads most of
// the time, lose more to the warps that then do not fit than they gain
// (iterations with the caps against without, both before the pools of rays: guided
// room 512^2 0.94 -> 0.89 ms in the warm-up and 1.44 -> 1.25 with given counts, 131k
// triangles at 1024^2 3.62 -> 2.97, 524k at 2048^2 13.4 -> 11.7).  k_reverse keeps its registers
// (capped at 80, 512^2 warm-up 0.86 -> 0.91 ms).
using TraceFn = void (*)(const DevScene, const DevCache, const Arena, const IterArgs*, const int);
using ShadowFn = void (*)(const DevScene, const DevCache, const Arena, const int, const int);
TraceFn trace_fn(int v) { return v == 2 ? k_trace<6> : k_trace<4>; }
TraceFn shade_fn(int v, bool bd = false) {
  if (bd) return v == 2 ? k_shade<4, true> : k_shade<3, true>;
  return v == 2 ? k_shade<4, false> : k_shade<3, false>;
}
ShadowFn shadow_fn(int v) { return v == 2 ? k_shadow<6> : k_shadow<4>; }
TraceFn reverse_fn(int v, bool bd = false) {
  if (bd) return v == 2 ? k_reverse<4, true> : (v == 1 ? k_reverse<3, true> : k_reverse<1, true>);
  return v == 2 ? k_reverse<4, false> : (v == 1 ? k_reverse<3, false> : k_reverse<1, false>);
}

}  // namespace

int wave_variants(int) { return 3; }
bool wave_variant_repeats(int kernel, int v, int techniques) {
  return v == 1 && kernel != WK_REVERSE && !(kernel == WK_SHADOW && (techniques & MARS_TECH_LIGHT));
}
int wave_variant_registers(int kernel, int v) {
  if (v == 0) return 0;
  if (kernel == WK_SHADE || kernel == WK_REVERSE) return v == 1 ? 80 : 64;
  return v == 1 ? 64 : 40;
}

cudaError_t wave_occupancy(const int threads[WAVE_KERNELS], const int variant[WAVE_KERNELS],
                           int blocks_per_sm[WAVE_KERNELS]) {
  cudaError_t e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[WK_TRACE], trace_fn(variant[WK_TRACE]),
                                                         threads[WK_TRACE], trace_smem(threads[WK_TRACE]))) != cudaSuccess)
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[WK_SHADE], shade_fn(variant[WK_SHADE]),
                                                         threads[WK_SHADE], shade_smem(threads[WK_SHADE]))) !=
      cudaSuccess)
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[WK_SHADOW], shadow_fn(variant[WK_SHADOW]),
                                                         threads[WK_SHADOW], trace_smem(threads[WK_SHADOW]))) != cudaSuccess)
    return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm[WK_REVERSE], reverse_fn(variant[WK_REVERSE]),
                                                       threads[WK_REVERSE], 0);
}

bool wave_threads_ok(int threads) { return threads >= 32 && threads <= MAX_WAVE_THREADS && threads % 32 == 0; }

// Whether the shadow and light connection kernels launched after wave d's shading
// take the waves up to d that earlier launches left.  With light connections the
// waves from `tail` on, all small, go three at a time: a launch of the light
// kernels lasts as long as its longest subpath (up to five traversals one after
// the other, 150 us and more) however few samples a wave has, and the launches of
// one stream follow one another.  Heightfield of 131k triangles, wave by wave -> in
// threes: 128^2 1.15 -> 0.83 ms, 256^2 1.45 -> 1.12, 512^2 2.08 -> 1.76, 1024^2 4.41 ->
// 4.23; in twos 0.85, 1.12, 1.83 and 4.22, all in one 0.98, 1.28, 1.84 and 4.29 (they
// then start late).
static bool side_batch_ends(int d, int D, int tail) {
  return tail <= 0 || d < tail || (d - tail) % 3 == 2 || d == D - 2 || d == D - 1;
}

cudaError_t launch_tile(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs* it, const WaveLaunch& L,
                        int64_t tile_pixels, int tail, int tail_blocks, cudaStream_t st, cudaStream_t side, cudaStream_t side2, const cudaEvent_t* sync,
                        cudaEvent_t* ev) {
  k_tile_init<<<1, 32, 0, st>>>(c.ctr, it);
  const int D = c.max_depth;
  const int tT = L.threads[WK_TRACE], tS = L.threads[WK_SHADE], tH = L.threads[WK_SHADOW], tR = L.threads[WK_REVERSE];
  // The persistent grid, but no more blocks than four rays per pixel of the
  // tile fill: a block without work still costs its launch (64^2 box 0.150 ->
  // 0.147 ms, 128^2 room 0.605 -> 0.596 ms; two rays per pixel 0.617, one 0.667:
  // the second and third waves hold more rays than there are pixels)
  auto G = [&](int k, int) {
    const int64_t most = (4 * tile_pixels + L.threads[k] - 1) / L.threads[k];
    return (int)std::max<int64_t>(1, std::min<int64_t>(L.grid[k], most));
  };
  const size_t smS = shade_smem(tS);
  const bool nee = (c.techniques & MARS_TECH_NEE) != 0;
  const bool bd = (c.techniques & MARS_TECH_LIGHT) != 0;
  // The NEE shadow rays of wave d run on the side stream and its light
  // connection samples on a second one (side2, else the side stream too),
  // overlapped with the forward kernels of the next waves and with each other
  // (disjoint data); the reverse pass, their only consumer, waits for all of
  // them.
  // sync: D + 2 events without timing (after shade(d); after the last shadow
  // kernel; after the last light kernel).  ev (optional, 7 D + 2 timing
  // events): ev[0] start; ev[2(d-1)+1],
  // ev[2(d-1)+2] after wave d's trace and shade; ev[2D + 2(d-1) + 1 .. 2] around
  // its shadow kernel on the side stream; ev[5D + 1] when the reverse pass may
  // start; ev[4D + k] after the k-th reverse kernel; ev[5D + 2 + 2(d-1) .. + 1]
  // around its light connection kernel on the side stream.
  if (ev) cudaEventRecord(ev[0], st);
  cudaStream_t lside = side2 ? side2 : side;
  bool any_shadow = false, any_light = false;
  const int last = !bd && tail > 0 ? tail - 1 : D;  // the deepest wave of the wave kernels
  int first = 1;
  for (int d = 1; d <= last; ++d) {
    trace_fn(L.variant[WK_TRACE])<<<G(WK_TRACE, d), tT, trace_smem(tT), st>>>(s, c, a, it, d);
    if (ev) cudaEventRecord(ev[2 * (d - 1) + 1], st);
    shade_fn(L.variant[WK_SHADE], bd)<<<G(WK_SHADE, d), tS, smS, st>>>(s, c, a, it, d);
    if (ev) cudaEventRecord(ev[2 * (d - 1) + 2], st);
    if (!side_batch_ends(d, D, bd ? tail : 0)) continue;
    // the side kernels of the waves first..d
    const bool shadow = first <= D - 1 && nee, light = bd && first <= D - 2;
    if (shadow || light) cudaEventRecord(sync[d - 1], st);
    if (shadow) {
      cudaStreamWaitEvent(side, sync[d - 1], 0);
      any_shadow = true;
      if (ev) cudaEventRecord(ev[2 * D + 2 * (d - 1) + 1], side);
      shadow_fn(L.variant[WK_SHADOW])<<<G(WK_SHADOW, d), tH, trace_smem(tH), side>>>(s, c, a, first, std::min(d, D - 1));
      if (ev) cudaEventRecord(ev[2 * D + 2 * (d - 1) + 2], side);
    }
    if (light) {
      if (lside != side || !shadow) cudaStreamWaitEvent(lside, sync[d - 1], 0);
      any_light = true;
      if (ev) cudaEventRecord(ev[5 * D + 2 + 2 * (d - 1)], lside);
      cudaError_t e = launch_light(s, c, a, it, L.variant[WK_SHADOW], G(WK_SHADOW, d), tH, first, std::min(d, D - 2), lside);
      if (e != cudaSuccess) return e;
      if (ev) cudaEventRecord(ev[5 * D + 2 + 2 * (d - 1) + 1], lside);
    }
    first = d + 1;
  }
  if (!bd && tail > 0) launch_tail(s, c, a, it, tail, tail_blocks, st);
  if (any_shadow) {
    cudaEventRecord(sync[D], side);
    cudaStreamWaitEvent(st, sync[D], 0);
  }
  if (any_light && lside != side) {
    cudaEventRecord(sync[D + 1], lside);
    cudaStreamWaitEvent(st, sync[D + 1], 0);
  } else if (any_light && !any_shadow) {
    cudaEventRecord(sync[D], side);
    cudaStreamWaitEvent(st, sync[D], 0);
  }
  if (ev) cudaEventRecord(ev[5 * D + 1], st);
  if (!bd && tail > 0) launch_tail_reverse(s, c, a, it, tail, tail_blocks, st);
  for (int d = last; d >= 1; --d) {
    reverse_fn(L.variant[WK_REVERSE], bd)<<<G(WK_REVERSE, d), tR, 0, st>>>(s, c, a, it, d);
    if (ev) cudaEventRecord(ev[4 * D + (D - d + 1)], st);
  }
  k_tile_finish<<<1, 32, 0, st>>>(c.ctr, c.tile_status, it, D);
  return cudaGetLastError();
}

cudaError_t launch_merge_lanes(DevCounters* dst, DevCounters* src, cudaStream_t st) {
  k_merge_lanes<<<1, 32, 0, st>>>(dst, src);
  return cudaGetLastError();
}

int tile_launches(int max_depth, int techniques, int tail) {
  const bool nee = (techniques & MARS_TECH_NEE) != 0, bd = (techniques & MARS_TECH_LIGHT) != 0;
  const int D = max_depth, last = !bd && tail > 0 ? tail - 1 : D;
  int n = 2 + 3 * last + (last < D ? 2 : 0);  // begin and end, trace, shade, reverse, the tail kernels
  for (int d = 1, first = 1; d <= last; ++d) {
    if (!side_batch_ends(d, D, bd ? tail : 0)) continue;
    if (nee && first <= D - 1) ++n;
    if (bd && first <= D - 2) n += 2;  // light subpaths, connections
    first = d + 1;
  }
  return n;
}

}  // namespace mars
