// tail.cu -- the waves from depth k on in two kernels, one forward (closest
// hits, shading, shadow rays) and one in reverse, instead of four launches a
// depth.  A small wave costs a launch and the slowest ray's chain of steps
// whatever its size (20 to 40 us for the closest hits alone), and the depths that
// follow wait for it.  Here a block takes its share of wave k's rays, the roots
// (camera rays for k = 1), and renders their subtrees by itself, in rounds: the
// children of the last round's rays and, up to TAIL_TARGET rays, new roots --
// closest hits of the round's rays beside the shadow rays of the last round's
// samples, then shading.  Other blocks' rounds fill the SM while one waits.  A
// block allocates from its own slice of the arena that the waves before left,
// without global counters.  The rounds (their rays) are written down for the
// reverse kernel, which runs them backwards; a child's round always comes after
// its parent's.  A slice that overflows raises the tile's overflow flag like a
// wave.  The device functions are the wave kernels' own, with the compiler's
// fused multiply-adds there spelled out, so that an image does not depend on
// which of the two rendered it.
// Bound by latency: the chain of the slowest ray of each round.  Measured per
// iteration, wave kernels alone -> with the tail: 64^2 box 0.150 -> 0.123 ms,
// 128^2 room of 459 spheres 0.575 -> 0.482, 317 x 203 room 0.532 -> 0.519, 128^2 and
// 256^2 heightfield of 131k triangles 0.75 -> 0.39 and 0.96 -> 0.59, 524k triangles
// at 256^2 1.38 -> 0.93; from a deeper wave on 512^2 room's warm-up 0.847 -> 0.824, with
// given counts 1.170 -> 1.159, heightfield at 1024^2 2.65 -> 2.43.
#define MARS_PIN_FMA
#include "wave.cuh"

namespace mars {

namespace {

// The block's share of a wave's rays, its roots: groups of ROOT_GROUP
// neighbouring rays dealt round-robin to the blocks, so that a cheap and a dear
// part of the image are spread over all of them (groups of 16 and 32 leave small
// images unevenly dealt: 64^2 room 0.40, 0.42 and 0.45 ms).
constexpr unsigned ROOT_GROUP = 8;
struct Roots {
  unsigned base;        // the wave's first slot
  unsigned blocks, block;
  __device__ __forceinline__ unsigned at(unsigned j) const {  // the wave's ray that is the block's root j
    return (j / ROOT_GROUP * blocks + block) * ROOT_GROUP + j % ROOT_GROUP;
  }
  // blocks of `blocks` that have roots in a wave of n rays: the first ones
  __device__ __forceinline__ static unsigned sharers(unsigned n, unsigned blocks) {
    return max(1u, min(blocks, (n + ROOT_GROUP - 1) / ROOT_GROUP));
  }
  __device__ __forceinline__ unsigned count(unsigned n) const {  // of a wave of n rays
    const unsigned groups = (n + ROOT_GROUP - 1) / ROOT_GROUP;
    if (block >= groups) return 0;
    const unsigned mine = (groups - 1 - block) / blocks + 1;
    return mine * ROOT_GROUP - ((groups - 1) % blocks == block ? groups * ROOT_GROUP - n : 0u);
  }
};
// The rays of a block's round: n_child children of the last round at `base`,
// then the roots from j0 on.
struct RoundSlots {
  unsigned base, n_child, j0;
  Roots roots;
  uint32_t px0;
  bool first_wave;  // the roots are camera rays
  __device__ __forceinline__ unsigned record(unsigned li) const {
    return li < n_child ? base + li : roots.base + roots.at(j0 + (li - n_child));
  }
  __device__ __forceinline__ bool camera(unsigned li) const { return first_wave && li >= n_child; }
  __device__ __forceinline__ uint32_t pixel(unsigned li) const { return px0 + roots.at(j0 + (li - n_child)); }
};
// the io of a block's round: children in the block's slice of the arena, counted
// in shared memory
struct BlockWave {
  using Index = unsigned;
  static constexpr bool MIXED = true;
  RoundSlots slots;
  Index n, base_next, sbase, lbase, cap, scap, lcap, first, stride;
  unsigned *count, *scount, *slcount, *over, *depth;  // shared memory; depth[d]: rays of depth d
  __device__ __forceinline__ void alloc(int te, int ts, int, Index b[3]) {
    b[0] = te > 0 ? atomicAdd(count, (unsigned)te) : 0u;
    b[1] = ts > 0 ? atomicAdd(scount, (unsigned)ts) : 0u;
    b[2] = 0;
  }
  __device__ __forceinline__ Index list(int n_) { return atomicAdd(slcount, (unsigned)n_); }
  __device__ __forceinline__ void overflow() { *over = OVER_SLICE; }
};
constexpr int TAIL_WARPS = TAIL_THREADS / 32;
// four blocks an SM: 126 registers and no spills (five blocks at 96 registers:
// 128^2 room 0.48 -> 0.52 ms; the chain of one thread's instructions is what
// takes the time here)
constexpr int TAIL_BLOCKS = 4;
constexpr unsigned TAIL_TARGET = 2 * TAIL_THREADS;  // 1, 4 and 8 times measure within 1 to 3 %

struct TailShared {
  IterArgs it;
  unsigned next[2][2];  // rays taken from the closest-hit and shadow pools (of even and odd rounds)
  unsigned count[2], scount[2], slcount[2];
  unsigned over;
  unsigned depth[MAXD + 2];
  unsigned long long work[2][4], shadow_entries, shadow_traced;
  ShadeBlock<unsigned> blk;
};
union TailScratch {
  ShadeWarpCtx ctx;
  RayStage stage;
};

// a warp's traversal counters into the block's
__device__ __forceinline__ void add_work(const TraceWork& w, unsigned long long* dst, DevCounters* ctr) {
#ifdef MARS_CHECKED
  if (w.bad) atomicOr(&ctr->check_flags, w.bad);
#else
  (void)ctr;
#endif
  const unsigned v[4] = {w.nodes, w.quads, w.spheres, w.tris};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned t = __reduce_add_sync(FULL, v[k]);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(dst + k, (unsigned long long)t);
  }
}

__global__ void __launch_bounds__(TAIL_THREADS, TAIL_BLOCKS) k_tail(const DevScene s, const DevCache c, const Arena a,
                                                             const IterArgs* __restrict__ itp, const int k) {
  __shared__ TailShared sh;
  __shared__ TailScratch scratch[TAIL_WARPS];
  const int tid = threadIdx.x, warp = tid >> 5;
  DevCounters* ctr = c.ctr;
  const Wave w = wave_of(ctr, a, k);
  if (tid == 0) {
    sh.it = *itp;
    sh.over = ctr->overflow;  // raised by an earlier wave, or by another block meanwhile
    sh.shadow_entries = sh.shadow_traced = 0;
  }
  if (tid < 8) sh.work[tid >> 2][tid & 3] = 0;
  if (tid < MAXD + 2) sh.depth[tid] = 0;
  if (tid < 2) sh.count[tid] = sh.scount[tid] = sh.slcount[tid] = sh.next[0][tid] = sh.next[1][tid] = 0;
  __syncthreads();
  const IterArgs& it = sh.it;
  // the block's slices of what the waves up to k left of the two regions, shared by
  // the blocks that have roots
  const unsigned sharers = Roots::sharers((unsigned)w.n, gridDim.x);
  const unsigned long long start = w.base + w.n, sstart = k == 1 ? 0ull : ctr->sbase[k - 1] + ctr->scount[k - 1];
  const bool sharer = blockIdx.x < sharers;
  const unsigned slice = sharer ? (unsigned)((a.cap - start) / sharers) : 0u;
  const unsigned sslice = sharer && sstart < a.scap ? (unsigned)((a.scap - sstart) / sharers) : 0u;
  RoundSlots rs;
  rs.base = (unsigned)start + blockIdx.x * slice;
  rs.n_child = rs.j0 = 0;
  rs.roots = Roots{(unsigned)w.base, gridDim.x, blockIdx.x};
  rs.px0 = (uint32_t)it.tile_begin;
  rs.first_wave = k == 1;
  const unsigned n_roots = rs.roots.count((unsigned)w.n), cap = rs.base + slice;
  unsigned sbase = (unsigned)sstart + blockIdx.x * sslice, prev_sbase = sbase, n_listed = 0;
  const unsigned scap = sbase + sslice;
  int r = 0;
  while (!sh.over) {
    // all the roots that are left when the rounds run out
    const unsigned room = r >= TAIL_ROUNDS - MAXD - 2 ? 0xffffffffu
                                                      : (rs.n_child < TAIL_TARGET ? TAIL_TARGET - rs.n_child : 0u);
    const unsigned n = rs.n_child + min(room, n_roots - rs.j0);
    if (n == 0 && n_listed == 0) break;
    const int e = r & 1;
    if (n > 0) {
      TraceWork tw;
      closest_hits(s, c, a, it, rs, n, k == 1 ? rs.n_child : n, &sh.next[e][0], (unsigned)warp, (unsigned)TAIL_WARPS,
                   &scratch[warp].stage, tw);
      add_work(tw, sh.work[0], ctr);
    }
    if (n_listed > 0) {
      TraceWork sw;
      shadow_hits(s, c, a, prev_sbase, n_listed, &sh.next[e][1], (unsigned)warp, (unsigned)TAIL_WARPS,
                  &scratch[warp].stage, sw);
      add_work(sw, sh.work[1], ctr);
    }
    __syncthreads();
    if (n == 0) break;
    if (tid == 0) {
      c.tail_rounds[(size_t)blockIdx.x * TAIL_ROUNDS + r] = make_uint4(rs.base, n, rs.n_child, rs.j0);
      sh.next[e ^ 1][0] = sh.next[e ^ 1][1] = 0;
      sh.count[e ^ 1] = sh.scount[e ^ 1] = sh.slcount[e ^ 1] = 0;
    }
    BlockWave io;
    io.slots = rs;
    io.n = n;
    io.base_next = rs.base + rs.n_child;
    io.sbase = sbase;
    io.lbase = 0;
    io.cap = cap;
    io.scap = scap;
    io.lcap = 0;
    io.first = 0;
    io.stride = TAIL_THREADS;
    io.count = &sh.count[e];
    io.scount = &sh.scount[e];
    io.slcount = &sh.slcount[e];
    io.over = &sh.over;
    io.depth = sh.depth;
    shade_wave<false>(s, c, a, it, k, io, &scratch[warp].ctx, sh.blk);
    __syncthreads();
    ++r;
    rs.j0 += n - rs.n_child;
    rs.base += rs.n_child;
    rs.n_child = sh.count[e];
    prev_sbase = sbase;
    sbase += sh.scount[e];
    n_listed = sh.slcount[e];
    if (tid == 0) {
      sh.shadow_entries += sh.scount[e];
      sh.shadow_traced += n_listed;
    }
  }
  __syncthreads();
  if (tid == 0) {
    c.tail_rounds[(size_t)gridDim.x * TAIL_ROUNDS + blockIdx.x] = make_uint4((unsigned)r, 0u, 0u, 0u);
    if (sh.over & OVER_SLICE) atomicOr(&ctr->overflow, OVER_SLICE);
    if (sh.shadow_entries) atomicAdd(&ctr->scount[k], sh.shadow_entries);
    if (sh.shadow_traced) atomicAdd(&ctr->slcount[k], sh.shadow_traced);
  }
  if (tid < 8 && sh.work[tid >> 2][tid & 3]) atomicAdd(&ctr->trace_work[tid >> 2][tid & 3], sh.work[tid >> 2][tid & 3]);
  if (tid >= 32 && tid < 32 + MAXD + 2 && sh.depth[tid - 32])
    atomicAdd(&ctr->count[tid - 32], (unsigned long long)sh.depth[tid - 32]);
}

// the same grid as k_tail's
__global__ void __launch_bounds__(TAIL_THREADS, TAIL_BLOCKS) k_tail_reverse(const DevScene s, const DevCache c, const Arena a,
                                                                     const IterArgs* __restrict__ itp, const int k) {
  if (c.ctr->overflow) return;  // the tile is re-rendered; commit nothing
  const IterArgs it = *itp;
  const int rounds = (int)c.tail_rounds[(size_t)gridDim.x * TAIL_ROUNDS + blockIdx.x].x;
  RoundSlots rs;
  rs.roots = Roots{(unsigned)c.ctr->base[k], gridDim.x, blockIdx.x};
  rs.px0 = (uint32_t)it.tile_begin;
  rs.first_wave = k == 1;
  RevSums acc;
  for (int r = rounds - 1; r >= 0; --r) {
    const uint4 q = c.tail_rounds[(size_t)blockIdx.x * TAIL_ROUNDS + r];
    rs.base = q.x;
    rs.n_child = q.z;
    rs.j0 = q.w;
    reverse_wave<false, unsigned>(s, c, a, it, rs, q.y, threadIdx.x & ~31u, (unsigned)TAIL_THREADS, acc);
    __syncthreads();
  }
  flush_sums(c, acc, (c.techniques & MARS_TECH_GUIDED) != 0);
}

}  // namespace

// resident blocks of k_tail per SM
int tail_occupancy() {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_tail, TAIL_THREADS, 0) != cudaSuccess) return 0;
  return b;
}

void launch_tail(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs* it, int k, int blocks,
                 cudaStream_t st) {
  k_tail<<<blocks, TAIL_THREADS, 0, st>>>(s, c, a, it, k);
}
void launch_tail_reverse(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs* it, int k, int blocks,
                         cudaStream_t st) {
  k_tail_reverse<<<blocks, TAIL_THREADS, 0, st>>>(s, c, a, it, k);
}

}  // namespace mars
