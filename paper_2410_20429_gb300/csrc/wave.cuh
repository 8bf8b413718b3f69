// wave.cuh -- what a wave's rays go through: closest and any hits by pools of
// rays, shading and sampling, and the reverse pass, as device functions of the
// wave kernels (render.cu) and of the kernels that render the deep waves of a
// tile together (tail.cu).
#pragma once

#include "device.cuh"

namespace mars {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// software prefetch of one line into L2 (no register result, no wait)
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// every wave kernel accepts blocks of up to MAX_WAVE_THREADS threads; the launch
// shape (threads per block, grid) is a per-cache setting (WaveLaunch)
constexpr int MAX_WAVE_THREADS = 256;

__device__ __forceinline__ float4 f4(f3 a, float w) { return make_float4(a.x, a.y, a.z, w); }
__device__ __forceinline__ f3 fmin3(f3 a, f3 b) { return mk3(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z)); }

// NEE density (solid angle at x) of reaching point y on light l along wi; HIT: y
// is where a ray hit the light (its squared distance then fuses in another order)
template <bool HIT>
__device__ __forceinline__ float nee_pdf(const DevScene& s, int l, f3 x, f3 y, f3 wi) {
  const float4 l1 = __ldg(s.lights + 5 * l + 1), l2 = __ldg(s.lights + 5 * l + 2), l3 = __ldg(s.lights + 5 * l + 3);
  const float cosl = -dot(xyz(l3), wi);
  if (cosl <= 0.0f) return 0.0f;
  const f3 dv = y - x;
  return l1.w * (HIT ? length2_hit(dv) : dot(dv, dv)) / (l2.w * cosl);
}

// pinhole camera ray of pixel px with box-filter jitter (W/p = 1)
__device__ __forceinline__ void camera_ray(const DevScene& s, const Rng& rng, uint32_t px, f3& o, f3& dir) {
  const float4 u = rng.u4(px, DIM_CAMERA, 0);
  const int ix = (int)(px % (uint32_t)s.width), iy = (int)(px / (uint32_t)s.width);
  const float sx = (2.0f * ((float)ix + u.x) / (float)s.width - 1.0f) * s.tanh_half * s.aspect;
  const float sy = (1.0f - 2.0f * ((float)iy + u.y) / (float)s.height) * s.tanh_half;
  const f3 cf = mk3(s.cam_f[0], s.cam_f[1], s.cam_f[2]);
  const f3 cr = mk3(s.cam_r[0], s.cam_r[1], s.cam_r[2]);
  const f3 cu = mk3(s.cam_u[0], s.cam_u[1], s.cam_u[2]);
  dir = normalize(cf + span2(cr, sx, cu, sy));
  o = mk3(s.cam_o[0], s.cam_o[1], s.cam_o[2]);
}

// slots [base, base + n) of wave d, clamped to the arena
struct Wave {
  unsigned long long base, n;
};
__device__ __forceinline__ Wave wave_of(const DevCounters* ctr, const Arena& a, int d) {
  const unsigned long long base = ctr->base[d], cnt = ctr->count[d];
  return {base, cnt < a.cap - base ? cnt : a.cap - base};
}

// A warp's allocation from a shared counter: its slots are contiguous, in lane
// order: lane l owns [base + incl - n, base + incl).
template <class Index>
struct WarpAlloc {
  Index base;  // first slot of the warp (relative to the counter's origin)
  int incl;                 // inclusive prefix of the counts up to this lane
  int total;                // slots of the whole warp
};

// inclusive warp scan of a per-lane count; returns (inclusive prefix, warp total)
__device__ __forceinline__ int2 warp_scan(int n, int lane) {
  int incl = n;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(FULL, incl, off);
    if (lane >= off) incl += y;
  }
  return make_int2(incl, __shfl_sync(FULL, incl, 31));
}

// lane owning item k of a warp block: the smallest l with incl[l] > k
__device__ __forceinline__ int owner_lane(const int* incl, int k) {
  int lo = 0, hi = 31;
#pragma unroll
  for (int it = 0; it < 5; ++it) {
    const int mid = (lo + hi) >> 1;
    if (incl[mid] > k) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// warp sum of a thread's traversal counters, one atomic per counter and warp
__device__ __forceinline__ void flush_work(TraceWork w, unsigned long long* dst, DevCounters* ctr) {
#ifdef MARS_CHECKED
  if (w.bad) atomicOr(&ctr->check_flags, w.bad);
#else
  (void)ctr;
#endif
  unsigned long long v[4] = {w.nodes, w.quads, w.spheres, w.tris};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], off);
  }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (v[k]) atomicAdd(dst + k, v[k]);
  }
}

// ------------------------------------------------------------------ trace
// The rays of a wave as its warps take them: chunks of 32, the first the warp's
// own, the others from a counter that the grid's warps share.  The two records
// of a chunk's rays are copied to shared memory one chunk ahead (cp.async), so
// that a lane that takes a ray does not wait for device memory.
struct RayStage {
  float4 r[2][2][32];  // [buffer][record][ray of the chunk]
};
template <class Counter, class Slots>
struct RayPool {
  const float4 *g0, *g1;  // the rays' records
  Slots slots;            // slots.record(k): where ray k's records are
  Counter* counter;
  RayStage* st;
  unsigned n, nrec;                      // rays; the first nrec have records
  unsigned base, cnt, off, nbase, ncnt;  // current chunk (rays used: off), next chunk
  unsigned warps;                           // warps that share the wave
  int buf;

  __device__ __forceinline__ void load(unsigned b, unsigned c, int which, int lane) {
    if ((unsigned)lane < c && b + lane < nrec) {
      const auto at = slots.record(b + lane);
      const unsigned d0 = (unsigned)__cvta_generic_to_shared(&st->r[which][0][lane]);
      const unsigned d1 = (unsigned)__cvta_generic_to_shared(&st->r[which][1][lane]);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d0), "l"(g0 + at) : "memory");
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d1), "l"(g1 + at) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void grab(int lane) {
    const Counter own = (Counter)warps * 32;
    nbase = ncnt = 0;
    if (n > own) {
      Counter b = 0;
      if (lane == 0) b = atomicAdd(counter, (Counter)32);
      b = own + __shfl_sync(FULL, b, 0);
      if (b < n) {
        nbase = (unsigned)b;
        ncnt = min(32u, n - nbase);
      }
    }
  }
  // warp, warps: the warp's number among those that share the wave
  __device__ __forceinline__ RayPool(const float4* g0_, const float4* g1_, Slots slots_, unsigned n_, unsigned nrec_,
                                     Counter* counter_, unsigned warp, unsigned warps_, RayStage* st_, int lane)
      : g0(g0_), g1(g1_), slots(slots_), counter(counter_), st(st_), n(n_), nrec(nrec_), off(0), warps(warps_), buf(0) {
    const unsigned b = warp * 32u;
    base = b < n ? b : 0u;
    cnt = b < n ? min(32u, n - base) : 0u;
    load(base, cnt, 0, lane);
    grab(lane);
    load(nbase, ncnt, 1, lane);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
  }
  __device__ __forceinline__ bool dry() const { return off >= cnt && ncnt == 0; }
  // a ray of the current chunk for every lane of `want`, as far as the chunk
  // goes: its index in the chunk, or -1
  __device__ __forceinline__ int take(unsigned want, int lane) {
    if (off >= cnt && ncnt > 0) {
      __syncwarp();
      base = nbase;
      cnt = ncnt;
      off = 0;
      grab(lane);
      load(nbase, ncnt, buf, lane);
      buf ^= 1;
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
    }
    const unsigned k = off + (unsigned)__popc(want & ((1u << lane) - 1u));
    off = min(cnt, off + (unsigned)__popc(want));
    return ((want >> lane) & 1u) && k < cnt ? (int)k : -1;
  }
};

// Traversal of the pool's rays, a warp's lanes each on a ray of their own.
// Divergence and the latency of a step's chain of loads and comparisons bound
// it, not arithmetic or bandwidth: rays of a wave need between a few and a
// hundred steps, and inner nodes and primitives run other code.  So lanes whose
// ray has ended take new rays as soon as REFILL of them wait (the others go on
// meanwhile), and each turn runs one kind of step: primitives when more than a
// third of the busy lanes are at one, else nodes (primitives shorten the rays
// they hit; any turn's kind left to the nodes alone was 25 % slower).
// Against one ray per thread from start to end over the binary hierarchy:
// guided room 512^2, first bounce, 0.67M rays: 12.0 -> 16.9 active lanes per
// instruction, 76.6M -> 66.6M warp instructions, 117 -> 108 us; iterations of
// the 524k-triangle scene at 2048^2 11.7 -> 10.8 ms, of the bidirectional
// 131k-triangle scene at 1024^2 4.9 -> 4.3 ms.  REFILL 4 to 16 measure alike,
// 24 and 32 slower on large scenes (11.6 and 11.1 ms).
// start(k, o4, d4, ray) prepares ray k of the wave and returns whether it is
// traced; done(k, ray) stores its result.
constexpr int REFILL = 8;
template <class Ray, class Pool, class Entry, class Start, class Done>
__device__ __forceinline__ void trace_pool(const DevScene& s, Pool& pool, Entry* stack, TraceWork& tw, int lane,
                                           Start start, Done done) {
  Ray q;
  q.cur = TRAV_DONE;
  unsigned li = 0;
  while (true) {
    const unsigned idle = __ballot_sync(FULL, q.cur == TRAV_DONE);
    if (idle == FULL || (__popc(idle) >= REFILL && !pool.dry())) {
      const int k = pool.take(idle, lane);
      if (k >= 0) {
        li = pool.base + (unsigned)k;
        if (!start(li, pool.st->r[pool.buf][0][k], pool.st->r[pool.buf][1][k], q)) q.cur = TRAV_DONE;
      }
      if (pool.dry() && __ballot_sync(FULL, q.cur != TRAV_DONE) == 0u) break;
    }
    const unsigned nodes = __ballot_sync(FULL, q.cur >= 0);
    const unsigned leaves = __ballot_sync(FULL, q.cur < 0 && q.cur != TRAV_DONE);
    if (__popc(nodes) >= 2 * __popc(leaves)) {
      if (q.cur >= 0) {
        q.node_step(s, stack, tw);
        if (q.cur == TRAV_DONE) done(li, q);
      }
    } else if (q.cur < 0 && q.cur != TRAV_DONE) {
      q.leaf_step(s, stack, tw);
      if (q.cur == TRAV_DONE) done(li, q);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Slots of a wave whose rays lie one after the other; those of the first wave
// are the camera rays of the pixels from px0 on.
struct WaveSlots {
  unsigned long long base;
  uint32_t px0;
  bool first_wave;
  __device__ __forceinline__ unsigned long long record(unsigned long long li) const { return base + li; }
  __device__ __forceinline__ bool camera(unsigned long long) const { return first_wave; }
  __device__ __forceinline__ uint32_t pixel(unsigned long long li) const { return px0 + (uint32_t)li; }
};

// closest hits of n rays into their hit records: distance and primitive, -1
// traced and missed, -2 not traced
template <class Counter, class Slots>
__device__ __forceinline__ void closest_hits(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs& it,
                                             const Slots& slots, unsigned n, unsigned nrec, Counter* counter,
                                             unsigned warp, unsigned warps, RayStage* st, TraceWork& tw) {
  const int lane = threadIdx.x & 31;
  const Rng rng{it.seed, it.job, it.iteration};
  uint2 stack[STACK];
  RayPool<Counter, Slots> pool(a.R[0], a.R[1], slots, n, nrec, counter, warp, warps, st, lane);
  trace_pool<ClosestRay>(
      s, pool, stack, tw, lane,
      [&](unsigned li, float4 r0, float4 r1, ClosestRay& q) {
        if (!chk(slots.record(li) < a.cap, MARS_CHECK_ARENA, c.ctr)) return false;
        f3 o = xyz(r0), dir = xyz(r1);
        if (slots.camera(li)) {
          camera_ray(s, rng, slots.pixel(li), o, dir);
        } else if (!(r1.w > 0.0f)) {  // A = beta_t p_t is 0 for a drawn sample that is not traced
          a.H[slots.record(li)] = make_float2(0.0f, __int_as_float(-2));
          return false;
        }
        q.start(o, dir);
        return true;
      },
      [&](unsigned li, const ClosestRay& q) {
        a.H[slots.record(li)] = make_float2(q.t_best, __int_as_float(q.best));
      });
}

// any hits of the n listed shadow rays at `sbase`: an occluded sample's value is zeroed
template <class Counter>
__device__ __forceinline__ void shadow_hits(const DevScene& s, const DevCache& c, const Arena& a,
                                            unsigned long long sbase, unsigned n, Counter* counter, unsigned warp,
                                            unsigned warps, RayStage* st, TraceWork& tw) {
  const int lane = threadIdx.x & 31;
  int stack[STACK];
  unsigned j = 0;
  RayPool<Counter, WaveSlots> pool(a.SH[0], a.SH[1], WaveSlots{sbase, 0u, false}, n, n, counter, warp, warps, st, lane);
  trace_pool<AnyRay>(
      s, pool, stack, tw, lane,
      [&](unsigned, float4 s0, float4 s1, AnyRay& q) {
        j = __float_as_uint(s1.w);
        if (!(s0.w > 0.0f)) return false;
        q.start(xyz(s0), xyz(s1), s0.w);
        return true;
      },
      [&](unsigned, const AnyRay& q) {
        if (q.hit && chk(j < a.scap, MARS_CHECK_SHADOW, c.ctr)) a.SH[2][j] = make_float4(0.f, 0.f, 0.f, 0.f);
      });
}

// ------------------------------------------------------------------ shade
// Per-warp staging area of k_shade: the context of the 32 vertices of a chunk,
// structure of arrays [field][lane], read by the lanes that draw their samples.
// C_Y and C_GP are used with light connections only (see k_shade<., true>).
enum {
  C_XO = 0, C_NS = 3, C_WO = 6, C_MTYPE = 9, C_ALPHA = 10, C_COL = 11, C_CELL = 14, C_PX = 15, C_LIN = 16,
  C_T = 18, C_B0 = 21, C_B1 = 22, C_B2 = 23, C_G0 = 24, C_MULT = 25, C_Y = 26, C_GP = 31, C_FIELDS = 32
};
struct ShadeWarpCtx {
  float f[C_FIELDS][32];
  int incl_ext[32];
  int incl_sh[32];
  int incl_lc[32];
};

// Whole-path weights with light connections (the bidirectional application,
// Sec. 5): the balance heuristic over every strategy of a full path z_1..z_n
// (z_n on a light) -- the camera path, NEE at z_{n-1}, light connection at
// z_i (i <= n - 2, n - 1 - i <= LIGHT_MAX light vertices) -- each strategy's
// density times its expected sample count.  Relative to the camera prefix
// C_k = prod_{j<k} bw_B(x_j) P->_j (P->_j: area density of x_{j+1} by BSDF
// sampling at x_j) the strategies that split the path before x_k add up to the
// window Y_k[l] = bw_L(x_{k-l}) prod_{m=k-l+1}^{k-2} P<-_m / prod_{m=k-l}^{k-1}
// bw_B P->_m (P<-_m: area density of x_m on a light subpath), which a ray
// carries forward as Z (Y of its parent times the parent's P<- towards the
// grandparent, Z[1] = the parent's light connection count) and the hit divides
// by the last step's bw_B P->.  The term of a light connection l vertices back
// at x_k is W_k[l] = Y_k[1] for l = 1 and Y_k[l] P<-_{k-1} for l >= 2 (P<-_{k-1}
// depends on the direction x_k continues in); a child carries Z[l] = W[l - 1].
// Emission hit at x_n from x_{n-1}:
//   w = bw_B P->_{n-1} / (bw_B P->_{n-1} + bw_N(x_{n-1}) pN + pN P<-_{n-1} sum_{l>=2} Z[l]);
// NEE at x_k towards y: w = bw_N pN / (bw_N pN + bw_B P->_k + pN P<-_k sum_l W_k[l]);
// light connections: the light kernel (bdpt.cu).
// Who shares a wave and where its rays and their children lie is the `io` of
// shade_wave: slots (record(li): ray li's slot; camera(li), pixel(li)), n rays,
// the first slots of children, NEE and light connection samples (base_next,
// sbase, lbase) and the ends of their regions (cap, scap, lcap), the block's
// first ray and its step, alloc() and list() from the shared counters, and MIXED:
// rays of any depth.
// a block's allocation of a chunk: per-warp counts, then their first slots
template <class Index>
struct ShadeBlock {
  int n[3][MAX_WAVE_THREADS / 32];
  Index base[3][MAX_WAVE_THREADS / 32];
};

// Shading and sampling of a wave by the blocks (or the block) that share it.
template <bool BD, class IO>
__device__ __forceinline__ void shade_wave(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs& it,
                                           const int d, IO& io, ShadeWarpCtx* ctx, ShadeBlock<typename IO::Index>& blk) {
  using Index = typename IO::Index;
  DevCounters* ctr = c.ctr;
  const Index base_next = io.base_next, sbase = io.sbase, lbase = io.lbase;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int D = c.max_depth;
  const bool on_b = c.techniques & MARS_TECH_BSDF, on_n = c.techniques & MARS_TECH_NEE,
             on_g = !BD && (c.techniques & MARS_TECH_GUIDED);
  // light connections are drawn at vertices of depth <= D - 2
  const bool on_l = BD && d <= D - 2;
  const Rng rng{it.seed, it.job, it.iteration};
  const float inf = __int_as_float(0x7f800000);

  // block-sized chunks (uniform trip count over the block); warp k of the block
  // takes the k-th 32 slots of the chunk
  for (Index b0 = io.first; b0 < io.n; b0 += io.stride) {
    const Index li = b0 + threadIdx.x;
    const Index i = io.slots.record(li);
    const bool active = li < io.n && chk(i < a.cap, MARS_CHECK_ARENA, ctr);
    const bool camera = io.slots.camera(li);
    bool est_depth = d <= D - 1;
    int depth = d;
    if (!IO::MIXED && d > 1) {
      // the ray record of this thread's next slot, fetched into L2 meanwhile
      const Index ln = li + io.stride;
      if (ln < io.n) {
        const Index in = io.slots.record(ln);
#pragma unroll
        for (int k = 0; k < NR; ++k) prefetch_l2(a.R[k] + in);
      }
    }

    // ---- the ray of this slot and its hit
    f3 o = mk3(0.f, 0.f, 0.f), dir = mk3(0.f, 0.f, 1.f), T = mk3(1.f, 1.f, 1.f), fcp = mk3(1.f, 1.f, 1.f);
    float A = 1.0f, S_ind = 1.0f, bwN = 0.0f, invSb = 0.0f;
    uint64_t lin = 0;
    uint32_t px = 0, parent_cell = 0;
    float th = 0.0f, mult = 1.0f;
    int prim = -2;
    float Z[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // light connections: whole-path weight window
    if (active) {
      if (camera) {
        px = io.slots.pixel(li);
        camera_ray(s, rng, px, o, dir);
      } else {
        mult = a.M[i];
        const float4 r0 = a.R[0][i], r1 = a.R[1][i], r2 = a.R[2][i], r3 = a.R[3][i], r4 = a.R[4][i];
        o = xyz(r0);
        px = __float_as_uint(r0.w);
        dir = xyz(r1);
        A = r1.w;
        T = xyz(r2);
        S_ind = r2.w;   // light connections: |cos| at the parent
        fcp = xyz(r3);
        bwN = r3.w;
        lin = (uint64_t)__float_as_uint(r4.x) | ((uint64_t)__float_as_uint(r4.y) << 32);
        if (BD) {
          const float4 r5 = a.R5[i];
          Z[0] = r4.z; Z[1] = r4.w; Z[2] = r5.x; Z[3] = r5.y; Z[4] = r5.z; Z[5] = r5.w;
        } else {
          parent_cell = __float_as_uint(r4.z);
          invSb = r4.w;
        }
      }
      // a ray's depth is the number of its lineage's digits and one
      if constexpr (IO::MIXED) {
        depth = 1 + (64 - __clzll((long long)lin) + c.bits - 1) / c.bits;
        est_depth = depth <= D - 1;
      }
      const float2 h = a.H[i];
      th = h.x;
      prim = __float_as_int(h.y);
    }

    f3 E = mk3(0.f, 0.f, 0.f);
    float Le_lum = 0.0f;
    const f3 G = camera ? mk3(1.f, 1.f, 1.f)
                        : (BD ? fcp : (S_ind > 0.0f ? fcp * (A / S_ind) : mk3(0.f, 0.f, 0.f)));
    uint32_t flags = prim >= -1 ? F_TRACED : 0u;
    int gam[NT] = {0, 0, 0};
    float beta[NT] = {0.f, 0.f, 0.f};
    float Y[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // light connections: Y_k[1..5]
    float gprev = 0.0f;                        // |cos| at the parent / t^2
    int cell = 0;
    f3 p = mk3(0.f, 0.f, 0.f), ns = mk3(0.f, 0.f, 1.f), wo = mk3(0.f, 0.f, 1.f);
    f3 climit = mk3(inf, inf, inf);
    Mat mat;
    mat.type = 0;
    mat.alpha = 1.0f;
    mat.col = mk3(0.f, 0.f, 0.f);
    if (prim >= 0 && chk(prim < s.n_prims, MARS_CHECK_PRIM, ctr)) {
      p = o + dir * th;
      const f3 ng = prim_normal(s.prims, prim, p);
      wo = dir * -1.0f;
      int m = prim_material(s.prims, prim);
      if (!chk(m >= 0 && m < s.n_mats, MARS_CHECK_MATERIAL, ctr)) m = 0;
      const float4 m0 = __ldg(s.mats + 3 * m), m1 = __ldg(s.mats + 3 * m + 1), m2 = __ldg(s.mats + 3 * m + 2);
      const float cosg = dot(ng, wo);
      // the last step's bw_B P-> (area density of this hit from the parent)
      const float inv_t2 = 1.0f / (th * th);
      const float cp_prev = BD && !camera ? A * fabsf(cosg) * inv_t2 : 0.0f;
      if (cosg > 0.0f && m0.w > 0.0f) {
        float w_dir = 1.0f;
        if (!camera && BD) {
          float sz = Z[1] + Z[2] + Z[3] + Z[4] + Z[5];
          float pN = 0.0f;
          if (prim < s.n_quads) {
            const int l = __float_as_int(__ldg(&s.prims[4 * prim + 3].w));
            if (l >= 0 && chk(l < s.n_lights, MARS_CHECK_LIGHT, ctr))
              pN = __ldg(&s.lights[5 * l + 1].w) / __ldg(&s.lights[5 * l + 2].w);
          }
          const float lpe = cosg * INV_PI_F * S_ind * inv_t2;   // P<-_{n-1}: cosine emission towards the parent
          const float den = cp_prev + bwN * pN + pN * lpe * sz;
          w_dir = den > 0.0f ? cp_prev / den : 0.0f;
        } else if (!camera) {
          float pn = 0.0f;
          if (bwN > 0.0f && prim < s.n_quads) {
            const int l = __float_as_int(__ldg(&s.prims[4 * prim + 3].w));
            if (l >= 0) pn = nee_pdf<true>(s, l, o, p, dir);
          }
          const float den = S_ind + bwN * pn;
          w_dir = den > 0.0f ? A / den : 0.0f;
        }
        const f3 Le = xyz(m2);
        E = mul(fcp, Le * w_dir);
        Le_lum = lum(Le);
      }
      if (est_depth && m0.z > 0.0f) {
        // ---- budgets and Alg. 1 at vertex x_d
        flags |= F_EST;
        ns = cosg >= 0.0f ? ng : ng * -1.0f;
        cell = c.oct_nodes ? octree_cell(s, c.oct_nodes, p) : cell_of(s, c.grid_n, p);
        if (!chk(cell >= 0 && cell < c.n_cells, MARS_CHECK_CELL, ctr)) cell = 0;
        if (!chk(px < (uint32_t)c.n_pixels, MARS_CHECK_PIXEL, ctr)) px = 0;
        mat.type = (int)m0.x;
        mat.alpha = m0.y;
        mat.col = xyz(m1);
        const float4 est = it.has_estimate ? c.est[px] : make_float4(1.f, 1.f, 1.f, 0.f);
        if (!BD && it.collect && it.has_estimate) {
          climit.x = T.x > 0.0f ? it.outlier * est.x / T.x : inf;
          climit.y = T.y > 0.0f ? it.outlier * est.y / T.y : inf;
          climit.z = T.z > 0.0f ? it.outlier * est.z / T.z : inf;
        }
        // counts without learned statistics: one NEE (and light connection)
        // sample and one continuation sample split evenly over BSDF and guided
        // sampling
        const float base_cont = (on_b && on_g) ? 0.5f : 1.0f;
        const unsigned on_mask = (on_b ? 1u : 0u) | (on_n ? 2u : 0u) | ((on_g || on_l) ? 4u : 0u);
        vertex_budgets(c, it, cell, T, est, mult, on_mask, base_cont, BD ? 1.0f : base_cont, beta);
        if (BD && !camera) {
          const float icp = cp_prev > 0.0f ? 1.0f / cp_prev : 0.0f;
#pragma unroll
          for (int l = 0; l < 5; ++l) Y[l] = Z[l] * icp;
          gprev = S_ind * inv_t2;
        }
        // Alg. 1: one uniform decides the rounding of every technique
        float r = rng.u4(px, DIM_ROUND, lin).x;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          if (!((on_mask >> t) & 1u)) continue;
          const float sm = beta[t] + r;
          const int g = (int)floorf(sm);
          gam[t] = g;
          r = sm - (float)g;
        }
      }
    }

    // ---- slots for the children (wave d+1), the NEE shadow rays and the light
    // connection samples: warp scans, then one atomic per counter and block
    // (every block of the grid allocates from the same counters)
    const int n_ext = BD ? gam[0] : gam[0] + gam[2], n_sh = gam[1], n_lc = BD ? gam[2] : 0;
    const int2 se = warp_scan(n_ext, lane), ss = warp_scan(n_sh, lane);
    const int2 sl = BD ? warp_scan(n_lc, lane) : make_int2(0, 0);
    if constexpr (IO::MIXED) {
      // rays drawn per depth, for the iteration's wave sizes
      unsigned left = __ballot_sync(FULL, n_ext > 0);
      while (left) {
        const int lead = __ffs(left) - 1;
        const int d0 = __shfl_sync(FULL, depth, lead);
        const unsigned same = __ballot_sync(FULL, n_ext > 0 && depth == d0);
        const unsigned drawn = __reduce_add_sync(FULL, depth == d0 ? (unsigned)n_ext : 0u);
        if (lane == 0) atomicAdd(&io.depth[d0 + 1], drawn);
        left &= ~same;
      }
    }
    if (lane == 31) {
      blk.n[0][warp] = se.y;
      blk.n[1][warp] = ss.y;
      blk.n[2][warp] = sl.y;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int te = 0, ts = 0, tl = 0;
      for (int k = 0; k < nwarps; ++k) {
        const int e = blk.n[0][k], h = blk.n[1][k], q = blk.n[2][k];
        blk.n[0][k] = te;
        blk.n[1][k] = ts;
        blk.n[2][k] = tl;
        te += e;
        ts += h;
        tl += q;
      }
      Index b[3];
      io.alloc(te, ts, BD ? tl : 0, b);
      for (int k = 0; k < nwarps; ++k) {
        blk.base[0][k] = b[0] + (Index)blk.n[0][k];
        blk.base[1][k] = b[1] + (Index)blk.n[1][k];
        blk.base[2][k] = b[2] + (Index)blk.n[2][k];
      }
    }
    __syncthreads();
    const WarpAlloc<Index> ae{blk.base[0][warp], se.x, se.y};
    const WarpAlloc<Index> as{blk.base[1][warp], ss.x, ss.y};
    const WarpAlloc<Index> al{blk.base[2][warp], sl.x, sl.y};
    const Index first = base_next + ae.base + (Index)(ae.incl - n_ext);
    const Index sfirst = sbase + as.base + (Index)(as.incl - n_sh);
    const Index lfirst = lbase + al.base + (Index)(al.incl - n_lc);
    const bool fits = first + (Index)n_ext <= io.cap && sfirst + (Index)n_sh <= io.scap &&
                      (!BD || lfirst + (Index)n_lc <= io.lcap);
    if ((n_ext > 0 || n_sh > 0 || n_lc > 0) && !fits) io.overflow();

    // ---- vertex record of this slot
    if (active) {
      flags |= (uint32_t)gam[0] | ((uint32_t)gam[1] << 8) | ((uint32_t)gam[2] << 16);
      a.V[0][i] = f4(E, __uint_as_float(flags));
      if (flags & F_EST) {
        a.V[1][i] = f4(G, 0.0f);
        a.V[2][i] = f4(climit, __uint_as_float((uint32_t)cell));
        a.V[3][i] = make_float4(beta[0], beta[1], beta[2], __uint_as_float((uint32_t)(fits && BD ? lfirst : 0ull)));
        // the hit record is dead from here on: keep the first child and first
        // shadow-ray slots in it for the reverse pass
        a.H[i] = make_float2(__uint_as_float((uint32_t)(fits ? first : 0ull)),
                             __uint_as_float((uint32_t)(fits ? sfirst : 0ull)));
      }
      if (on_g && it.collect && !camera && (flags & F_TRACED))
        a.V[4][i] = make_float4(Le_lum, invSb, __uint_as_float(parent_cell), __int_as_float(guide_bin(dir)));
    }
    if (ae.total == 0 && as.total == 0 && al.total == 0) continue;  // warp-uniform; no block barrier follows

    // ---- stage the vertex context of every lane for the cooperative loops
    {
      const Frame fr = make_frame(ns);
      const f3 wol = fr.to_local(wo);
      const f3 xo = p + ns * s.eps;
      float* cx = ctx->f[0];
      cx[C_XO * 32 + lane] = xo.x; cx[(C_XO + 1) * 32 + lane] = xo.y; cx[(C_XO + 2) * 32 + lane] = xo.z;
      cx[C_NS * 32 + lane] = ns.x; cx[(C_NS + 1) * 32 + lane] = ns.y; cx[(C_NS + 2) * 32 + lane] = ns.z;
      cx[C_WO * 32 + lane] = wol.x; cx[(C_WO + 1) * 32 + lane] = wol.y; cx[(C_WO + 2) * 32 + lane] = wol.z;
      cx[C_MTYPE * 32 + lane] = __int_as_float(mat.type);
      cx[C_ALPHA * 32 + lane] = mat.alpha;
      cx[C_COL * 32 + lane] = mat.col.x; cx[(C_COL + 1) * 32 + lane] = mat.col.y; cx[(C_COL + 2) * 32 + lane] = mat.col.z;
      cx[C_CELL * 32 + lane] = __int_as_float(cell);
      cx[C_PX * 32 + lane] = __uint_as_float(px);
      cx[C_LIN * 32 + lane] = __uint_as_float((uint32_t)lin);
      cx[(C_LIN + 1) * 32 + lane] = __uint_as_float((uint32_t)(lin >> 32));
      cx[C_T * 32 + lane] = T.x; cx[(C_T + 1) * 32 + lane] = T.y; cx[(C_T + 2) * 32 + lane] = T.z;
      cx[C_B0 * 32 + lane] = beta[0];
      cx[C_B1 * 32 + lane] = beta[1];
      cx[C_B2 * 32 + lane] = beta[2];
      cx[C_G0 * 32 + lane] = __int_as_float(gam[0]);
      cx[C_MULT * 32 + lane] = mult;
      if (BD) {
#pragma unroll
        for (int l = 0; l < 5; ++l) cx[(C_Y + l) * 32 + lane] = Y[l];
        cx[C_GP * 32 + lane] = gprev;
      }
      ctx->incl_ext[lane] = ae.incl;
      ctx->incl_sh[lane] = as.incl;
      ctx->incl_lc[lane] = al.incl;
    }
    __syncwarp();
    const float* cx = ctx->f[0];

    // NEE samples (primary estimators of NEE), one per lane and pass; the value
    // assumes the light is visible (the shadow kernel zeroes it otherwise)
    for (int k0 = 0; k0 < as.total; k0 += 32) {
      const int k = k0 + lane;
      const Index j = sbase + as.base + (Index)k;
      bool trace = false;
      f3 xo = mk3(0.f, 0.f, 0.f), wi = mk3(0.f, 0.f, 1.f);
      float tmax = -1.0f;
      if (k < as.total && j < io.scap) {
        const int L = owner_lane(ctx->incl_sh, k);
        const int sidx = k - (L > 0 ? ctx->incl_sh[L - 1] : 0);
        xo = mk3(cx[C_XO * 32 + L], cx[(C_XO + 1) * 32 + L], cx[(C_XO + 2) * 32 + L]);
        const f3 vns = mk3(cx[C_NS * 32 + L], cx[(C_NS + 1) * 32 + L], cx[(C_NS + 2) * 32 + L]);
        const f3 wol = mk3(cx[C_WO * 32 + L], cx[(C_WO + 1) * 32 + L], cx[(C_WO + 2) * 32 + L]);
        Mat m;
        m.type = __float_as_int(cx[C_MTYPE * 32 + L]);
        m.alpha = cx[C_ALPHA * 32 + L];
        m.col = mk3(cx[C_COL * 32 + L], cx[(C_COL + 1) * 32 + L], cx[(C_COL + 2) * 32 + L]);
        const uint32_t vpx = __float_as_uint(cx[C_PX * 32 + L]);
        const uint64_t vlin = (uint64_t)__float_as_uint(cx[C_LIN * 32 + L]) |
                              ((uint64_t)__float_as_uint(cx[(C_LIN + 1) * 32 + L]) << 32);
        const float bB = cx[C_B0 * 32 + L], bN = cx[C_B1 * 32 + L], bG = cx[C_B2 * 32 + L];
        const float bwB = on_b ? (it.aware ? bB : 1.0f) : 0.0f;
        const float bwNv = on_n ? (it.aware ? bN : 1.0f) : 0.0f;
        const float bwG = on_g ? (it.aware ? bG : 1.0f) : 0.0f;
        const float4 u = rng.u4(vpx, 32u + (uint32_t)sidx, vlin);
        int l = s.n_lights - 1;
        for (int q = 0; q < s.n_lights; ++q)
          if (u.x < __ldg(&s.lights[5 * q].w)) { l = q; break; }
        const float4 l0 = __ldg(s.lights + 5 * l), l1 = __ldg(s.lights + 5 * l + 1),
                     l2 = __ldg(s.lights + 5 * l + 2), l4 = __ldg(s.lights + 5 * l + 4);
        const f3 y = xyz(l0) + span2(xyz(l1), u.y, xyz(l2), u.z);
        const f3 dv = y - xo;
        const float dist = sqrtf(dot(dv, dv));
        wi = dv * (1.0f / dist);
        const float pn = nee_pdf<false>(s, l, xo, y, wi);
        const float ci = dot(vns, wi);
        f3 v = mk3(0.f, 0.f, 0.f);
        if (pn > 0.0f && ci > 0.0f) {
          const Frame fr = make_frame(vns);
          float pb;
          const f3 wil = fr.to_local(wi);
          const f3 fc = bsdf_eval(m, wol, wil, pb);
          const float pg = on_g ? guide_pdf(c.guide_cdf + (size_t)__float_as_int(cx[C_CELL * 32 + L]) * GUIDE_BINS, wi)
                                : 0.0f;
          if (nonzero(fc)) {
            if (BD) {
              // the full path x_1..x_d, y: weight over every strategy
              const float4 l3 = __ldg(s.lights + 5 * l + 3);
              const float pN = l1.w / l2.w;
              const float cosl = -dot(xyz(l3), wi);
              const float id2 = 1.0f / (dist * dist);
              const float t_nee = bwNv * pN;
              const float t_cam = bwB * pb * cosl * id2;
              // light connections l vertices back: W[1] = Y[1], W[l] = Y[l] P<-_{d-1} (l >= 2)
              const float y1 = cx[C_Y * 32 + L];
              float sy = 0.0f;
#pragma unroll
              for (int q = 1; q < 5; ++q) sy += cx[(C_Y + q) * 32 + L];
              float t_lc = 0.0f;
              if (y1 > 0.0f || sy > 0.0f) {
                float lp = 0.0f;
                if (sy > 0.0f) {
                  float prev;
                  const f3 frev = bsdf_eval(m, wil, wol, prev);   // at x_d, light arriving along wi
                  const float qx = prev > 0.0f ? fminf(1.0f, max_channel(frev) / prev) : 0.0f;
                  lp = prev * qx * cx[C_GP * 32 + L];
                }
                t_lc = pN * (cosl * INV_PI_F * ci * id2) * (y1 + lp * sy);
              }
              const float den = t_nee + t_cam + t_lc;
              const float sc = den > 0.0f ? t_nee / (den * pn) : 0.0f;
              v = mk3(fc.x * l4.x * sc, fc.y * l4.y * sc, fc.z * l4.z * sc);
            } else {
              // f|cos| Le / p_N times the balance weight beta_N p_N / den: p_N cancels
              const float den = sum3(bwB, pb, bwG, pg, bwNv, pn);
              const float sc = bwNv / den;
              v = mk3(fc.x * l4.x * sc, fc.y * l4.y * sc, fc.z * l4.z * sc);
            }
          }
        }
        a.SH[2][j] = f4(v, 0.0f);
        // a sample of value 0 needs no shadow ray
        trace = nonzero(v);
        tmax = dist - s.eps;
      }
      // compacted list of the shadow rays to trace: one atomic per warp
      const unsigned need = __ballot_sync(FULL, trace);
      if (need) {
        Index lb = 0;
        if (lane == 0) lb = io.list(__popc(need));
        lb = __shfl_sync(FULL, lb, 0);
        if (trace) {
          const Index pos = sbase + lb + (Index)__popc(need & ((1u << lane) - 1u));
          if (pos < io.scap) {
            a.SH[0][pos] = f4(xo, tmax);
            a.SH[1][pos] = f4(wi, __uint_as_float((unsigned int)j));
          }
        }
      }
    }

    // BSDF and guided children (primary estimators that continue the path);
    // a vertex's BSDF children come first, then its guided children
    for (int k0 = 0; k0 < ae.total; k0 += 32) {
      const int k = k0 + lane;
      const Index j = base_next + ae.base + (Index)k;
      if (k < ae.total && j < io.cap) {
        const int L = owner_lane(ctx->incl_ext, k);
        const int kk = k - (L > 0 ? ctx->incl_ext[L - 1] : 0);
        const int g0 = __float_as_int(cx[C_G0 * 32 + L]);
        const int t = kk < g0 ? 0 : 2;
        const int sidx = t == 0 ? kk : kk - g0;
        const f3 xo = mk3(cx[C_XO * 32 + L], cx[(C_XO + 1) * 32 + L], cx[(C_XO + 2) * 32 + L]);
        const f3 vns = mk3(cx[C_NS * 32 + L], cx[(C_NS + 1) * 32 + L], cx[(C_NS + 2) * 32 + L]);
        const f3 wol = mk3(cx[C_WO * 32 + L], cx[(C_WO + 1) * 32 + L], cx[(C_WO + 2) * 32 + L]);
        Mat m;
        m.type = __float_as_int(cx[C_MTYPE * 32 + L]);
        m.alpha = cx[C_ALPHA * 32 + L];
        m.col = mk3(cx[C_COL * 32 + L], cx[(C_COL + 1) * 32 + L], cx[(C_COL + 2) * 32 + L]);
        const int vcell = __float_as_int(cx[C_CELL * 32 + L]);
        const uint32_t vpx = __float_as_uint(cx[C_PX * 32 + L]);
        const uint64_t vlin = (uint64_t)__float_as_uint(cx[C_LIN * 32 + L]) |
                              ((uint64_t)__float_as_uint(cx[(C_LIN + 1) * 32 + L]) << 32);
        const f3 vT = mk3(cx[C_T * 32 + L], cx[(C_T + 1) * 32 + L], cx[(C_T + 2) * 32 + L]);
        const float bB = cx[C_B0 * 32 + L], bN = cx[C_B1 * 32 + L], bG = cx[C_B2 * 32 + L];
        const float bwB = on_b ? (it.aware ? bB : 1.0f) : 0.0f;
        const float bwNv = on_n ? (it.aware ? bN : 1.0f) : 0.0f;
        const float bwG = on_g ? (it.aware ? bG : 1.0f) : 0.0f;
        const float bt = t == 0 ? bB : bG;
        const float* cdf = on_g ? c.guide_cdf + (size_t)vcell * GUIDE_BINS : nullptr;
        const Frame fr = make_frame(vns);
        const float4 u = rng.u4(vpx, (uint32_t)(t * 32 + sidx), vlin);
        f3 wi = mk3(0.f, 0.f, 1.f);
        bool ok;
        float pt = 0.0f;
        if (t == 0) {
          f3 wl;
          ok = bsdf_sample(m, wol, u.x, u.y, wl);
          if (ok) wi = fr.to_world(wl);
        } else {
          int b = guide_pick(cdf, u.x);
          if (!chk(b >= 0 && b < GUIDE_BINS, MARS_CHECK_BIN, ctr)) b = 0;
          wi = guide_dir(b, u.y, u.z);
          pt = guide_bin_prob(cdf, b) * (GUIDE_BINS / (4.0f * PI_F));
          ok = dot(wi, vns) > 0.0f;
        }
        float cA = 0.0f, cS = 0.0f, cinvSb = 0.0f;
        f3 cf = mk3(0.f, 0.f, 0.f), cT = mk3(0.f, 0.f, 0.f);
        float cz[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (ok) {
          float pb;
          const f3 wil = fr.to_local(wi);
          const f3 fc = bsdf_eval(m, wol, wil, pb);
          const float pg = on_g ? guide_pdf(cdf, wi) : 0.0f;
          if (t == 0) pt = pb;
          if (pt > 0.0f && nonzero(fc)) {
            const float ipt = 1.0f / pt;
            cf = mk3(fc.x * ipt, fc.y * ipt, fc.z * ipt);
            cA = (t == 0 ? bwB : bwG) * pt;
            if (BD) {
              // no MIS weight on the continuation; the ray carries |cos| here and
              // the whole-path window
              const float wb = 1.0f / bt;
              cT = mk3(vT.x * cf.x * wb, vT.y * cf.y * wb, vT.z * cf.z * wb);
              cS = dot(vns, wi);
              // Z of the child: Z[1] = bw_L here, Z[l] = W[l - 1] (W[1] = Y[1], W[l] = Y[l] P<-_{d-1})
              cz[0] = on_l ? (it.aware ? bG : 1.0f) : 0.0f;
              cz[1] = cx[C_Y * 32 + L];
              float sy = 0.0f;
#pragma unroll
              for (int q = 1; q < 5; ++q) sy += cx[(C_Y + q) * 32 + L];
              if (sy > 0.0f) {
                float prev;
                const f3 frev = bsdf_eval(m, wil, wol, prev);   // P<- of the parent towards its parent
                const float qx = prev > 0.0f ? fminf(1.0f, max_channel(frev) / prev) : 0.0f;
                const float lp = prev * qx * cx[C_GP * 32 + L];
#pragma unroll
                for (int q = 1; q < 5; ++q) cz[q + 1] = cx[(C_Y + q) * 32 + L] * lp;
              }
            } else {
              cS = sum2(bwB, pb, bwG, pg);
              const float w_ind = cA / cS;
              const float wb = w_ind / bt;
              cT = mk3(vT.x * cf.x * wb, vT.y * cf.y * wb, vT.z * cf.z * wb);
              const float sb = bB * pb + (on_g ? bG * pg : 0.0f);
              cinvSb = sb > 0.0f ? 1.0f / sb : 0.0f;
            }
          }
        }
        const uint64_t digit = (uint64_t)(t == 0 ? sidx + 1 : 32 + sidx + 1);
        const uint64_t clin = (vlin << c.bits) | digit;
        a.R[0][j] = f4(xo, __uint_as_float(vpx));
        a.R[1][j] = f4(wi, cA);
        a.R[2][j] = f4(cT, cS);
        a.R[3][j] = f4(cf, bwNv);
        if (BD) {
          a.R[4][j] = make_float4(__uint_as_float((uint32_t)clin), __uint_as_float((uint32_t)(clin >> 32)), cz[0], cz[1]);
          a.R5[j] = make_float4(cz[2], cz[3], cz[4], cz[5]);
        } else {
          a.R[4][j] = make_float4(__uint_as_float((uint32_t)clin), __uint_as_float((uint32_t)(clin >> 32)),
                                  __uint_as_float((uint32_t)vcell), cinvSb);
        }
        a.M[j] = cx[C_MULT * 32 + L] * bt;
      }
    }

    // light connection samples: the camera vertex's context for the light kernel
    if (BD) {
      for (int k0 = 0; k0 < al.total; k0 += 32) {
        const int k = k0 + lane;
        const Index j = lbase + al.base + (Index)k;
        if (k < al.total && j < io.lcap) {
          const int L = owner_lane(ctx->incl_lc, k);
          const int sidx = k - (L > 0 ? ctx->incl_lc[L - 1] : 0);
          const f3 vns = mk3(cx[C_NS * 32 + L], cx[(C_NS + 1) * 32 + L], cx[(C_NS + 2) * 32 + L]);
          const f3 wow = make_frame(vns).to_world(mk3(cx[C_WO * 32 + L], cx[(C_WO + 1) * 32 + L],
                                                      cx[(C_WO + 2) * 32 + L]));
          const float bB = cx[C_B0 * 32 + L], bN = cx[C_B1 * 32 + L], bL = cx[C_B2 * 32 + L];
          a.LJ[0][j] = make_float4(cx[C_XO * 32 + L], cx[(C_XO + 1) * 32 + L], cx[(C_XO + 2) * 32 + L],
                                   cx[C_PX * 32 + L]);
          a.LJ[1][j] = f4(vns, __uint_as_float((uint32_t)__float_as_int(cx[C_MTYPE * 32 + L]) |
                                               ((uint32_t)sidx << 8) | ((uint32_t)d << 16)));
          a.LJ[2][j] = make_float4(cx[C_COL * 32 + L], cx[(C_COL + 1) * 32 + L], cx[(C_COL + 2) * 32 + L],
                                   cx[C_ALPHA * 32 + L]);
          a.LJ[3][j] = f4(wow, cx[C_MULT * 32 + L]);
          a.LJ[4][j] = make_float4(cx[C_T * 32 + L], cx[(C_T + 1) * 32 + L], cx[(C_T + 2) * 32 + L], bB);
          a.LJ[5][j] = make_float4(it.aware ? bB : 1.0f, on_n ? (it.aware ? bN : 1.0f) : 0.0f,
                                   it.aware ? bL : 1.0f, cx[C_GP * 32 + L]);
          a.LJ[6][j] = make_float4(cx[C_Y * 32 + L], cx[(C_Y + 1) * 32 + L], cx[(C_Y + 2) * 32 + L],
                                   cx[(C_Y + 3) * 32 + L]);
          a.LJ[7][j] = make_float4(cx[C_LIN * 32 + L], cx[(C_LIN + 1) * 32 + L], 0.0f, 0.0f);
        }
      }
    }
    __syncwarp();  // the context is overwritten by the next chunk
  }
}

// ---------------------------------------------------------------- reverse
// inclusive scan restricted to runs of equal keys (start = first lane of the run)
__device__ __forceinline__ float seg_scan(float v, int lane, int start) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float u = __shfl_up_sync(FULL, v, off);
    if (lane - off >= start) v += u;
  }
  return v;
}

// iteration counters of a thread's slots: one warp reduction and one atomic per
// counter and warp at the end, not per chunk (every warp of the grid adds to the
// same few addresses)
struct RevSums {
  unsigned n_traced = 0, n_est = 0, n_rays = 0;
  double sb0 = 0.0, sb1 = 0.0, sb2 = 0.0;
};

// Values, costs and statistics of n rays, 32 at a time: this warp's chunks start
// at c0 and step by `step`.
template <bool BD, class Index, class Slots>
__device__ __forceinline__ void reverse_wave(const DevScene& s, const DevCache& c, const Arena& a, const IterArgs& it,
                                             const Slots& slots, const Index n, Index c0, const Index step,
                                             RevSums& acc) {
  DevCounters* ctr = c.ctr;
  const int lane = threadIdx.x & 31;
  const bool on_g = !BD && (c.techniques & MARS_TECH_GUIDED);
  const bool collect = it.collect != 0;
  for (; c0 < n; c0 += step) {
    const Index li = c0 + lane;
    const Index i = slots.record(li);
    const bool active = li < n && chk(i < a.cap, MARS_CHECK_ARENA, ctr);
    const bool camera = slots.camera(li);
    {
      // the records of this thread's next slot, fetched into L2 while this one
      // is processed (the reverse pass reads them long after they were written)
      const Index ln = li + step;
      if (ln < n) {
        const Index in = slots.record(ln);
        prefetch_l2(a.V[0] + in);
        prefetch_l2(a.H + in);
        prefetch_l2(a.V[1] + in);
        prefetch_l2(a.V[2] + in);
        prefetch_l2(a.V[3] + in);
      }
    }
    uint32_t flags = 0;
    f3 E = mk3(0.f, 0.f, 0.f), Lr = mk3(0.f, 0.f, 0.f);
    uint32_t csub = 0;
    uint32_t key = 0xffffffffu;
    float st[NT][NSTAT];
#pragma unroll
    for (int t = 0; t < NT; ++t)
#pragma unroll
      for (int k = 0; k < NSTAT; ++k) st[t][k] = 0.0f;
    float bt[NT] = {0.f, 0.f, 0.f};
    if (active) {
      // one round trip for the flags and the first child / shadow-ray slots,
      // then every other load of the vertex is issued before any is used
      const float4 v0 = a.V[0][i];
      const float2 fs = a.H[i];
      E = xyz(v0);
      flags = __float_as_uint(v0.w);
      const bool guide_dep = on_g && collect && !camera && (flags & F_TRACED);
      float4 v4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (guide_dep) v4 = a.V[4][i];
      if (flags & F_EST) {
        int gB = flags & 0xff, gN = (flags >> 8) & 0xff, gG = (flags >> 16) & 0xff;
        // with light connections slot 2 holds the light connection samples,
        // which are not children
        int gL = BD ? gG : 0;
        if (BD) gG = 0;
        int ne = gB + gG;
        Index first = __float_as_uint(fs.x), sf = __float_as_uint(fs.y);
        // the children and NEE values lie inside the arena (else read none)
        const bool in_a = chk(first + (Index)ne <= a.cap, MARS_CHECK_ARENA, ctr);
        const bool in_s = chk(sf + (Index)gN <= a.scap, MARS_CHECK_SHADOW, ctr);
        if (!in_a) { first = 0; ne = 0; gB = 0; gG = 0; }
        if (!in_s) { sf = 0; gN = 0; }
        const float4 v1 = a.V[1][i], v2 = a.V[2][i], v3 = a.V[3][i];
        float4 pn[4], pe[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          pn[q] = q < gN ? a.SH[2][sf + q] : make_float4(0.f, 0.f, 0.f, 0.f);
          pe[q] = q < ne ? a.S[first + q] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        bt[0] = v3.x; bt[1] = v3.y; bt[2] = v3.z;
        const f3 climit = xyz(v2);
        key = __float_as_uint(v2.w);
        if (!chk(key < (uint32_t)c.n_cells, MARS_CHECK_CELL, ctr)) key = 0xffffffffu;
        if (gN > 0) {
          f3 sum = mk3(0.f, 0.f, 0.f);
          for (int k = 0; k < gN; k += 4) {
            if (k > 0) {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                pn[q] = k + q < gN ? a.SH[2][sf + k + q] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (k + q >= gN) break;
              const f3 v = xyz(pn[q]);
              sum = sum + v;
              const f3 vc = fmin3(v, climit);
              st[1][1] += vc.x; st[1][2] += vc.y; st[1][3] += vc.z;
              st[1][4] += vc.x * vc.x; st[1][5] += vc.y * vc.y; st[1][6] += vc.z * vc.z;
            }
          }
          const float ib1 = 1.0f / bt[1];
          Lr = mk3(sum.x * ib1, sum.y * ib1, sum.z * ib1);
          csub += (uint32_t)gN;
          st[1][0] = (float)gN;
          st[1][7] = (float)gN;
        }
        // 1 / beta once per technique, not one division per child value
        const float ib0 = gB > 0 ? 1.0f / bt[0] : 0.0f, ib2 = gG > 0 ? 1.0f / bt[2] : 0.0f;
        for (int k = 0; k < ne; k += 4) {
          if (k > 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) pe[q] = k + q < ne ? a.S[first + k + q] : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (k + q >= ne) break;
            const float4 sv = pe[q];
            const int t = k + q < gB ? 0 : 2;
            const float ib = t == 0 ? ib0 : ib2;
            Lr = Lr + mk3(sv.x * ib, sv.y * ib, sv.z * ib);
            const uint32_t cc = __float_as_uint(sv.w);
            csub += cc;
            const f3 vc = fmin3(xyz(sv), climit);
            if (t == 0) {
              st[0][0] += 1.0f; st[0][1] += vc.x; st[0][2] += vc.y; st[0][3] += vc.z;
              st[0][4] += vc.x * vc.x; st[0][5] += vc.y * vc.y; st[0][6] += vc.z * vc.z; st[0][7] += (float)cc;
            } else {
              st[2][0] += 1.0f; st[2][1] += vc.x; st[2][2] += vc.y; st[2][3] += vc.z;
              st[2][4] += vc.x * vc.x; st[2][5] += vc.y * vc.y; st[2][6] += vc.z * vc.z; st[2][7] += (float)cc;
            }
          }
        }
        if (BD && gL > 0) {
          // light connection samples: the sum of the sample's connections (in
          // the order of its light vertices) and its cost from the light kernels
          unsigned long long lf = __float_as_uint(v3.w);
          if (!chk(lf + (unsigned long long)gL <= a.lcap, MARS_CHECK_ARENA, ctr)) gL = 0;
          const float ib = 1.0f / bt[2];
          for (int q = 0; q < gL; ++q) {
            const float4 lr = a.LR[lf + q];
            const unsigned long long vf = __float_as_uint(lr.x);
            int m = (int)__float_as_uint(lr.y);
            if (!chk(m <= LIGHT_MAX && vf + (unsigned long long)m <= a.vcap, MARS_CHECK_ARENA, ctr)) m = 0;
            f3 v = mk3(0.f, 0.f, 0.f);
            for (int k = 0; k < m; ++k) v = v + xyz(a.LC[vf + k]);
            const uint32_t cc = (uint32_t)lr.w;
            Lr = Lr + mk3(v.x * ib, v.y * ib, v.z * ib);
            csub += cc;
            st[2][0] += 1.0f; st[2][1] += v.x; st[2][2] += v.y; st[2][3] += v.z;
            st[2][4] += v.x * v.x; st[2][5] += v.y * v.y; st[2][6] += v.z * v.z; st[2][7] += (float)cc;
          }
        }
        const f3 G = xyz(v1);
        E = E + mul(G, Lr);
      }
      const uint32_t cost = 1u + csub;
      a.S[i] = f4(E, __uint_as_float(cost));
      if (camera && chk(slots.pixel(li) < (uint32_t)c.n_pixels, MARS_CHECK_PIXEL, ctr))
        c.img[slots.pixel(li)] = f4(E, (float)cost);  // w: rays of the pixel's path tree
      if (guide_dep) {
        const float wdep = (v4.x + lum(Lr)) * v4.y;
        if (wdep > 0.0f && chk(__float_as_uint(v4.z) < (uint32_t)c.n_cells, MARS_CHECK_CELL, ctr) &&
            chk(__float_as_int(v4.w) >= 0 && __float_as_int(v4.w) < GUIDE_BINS, MARS_CHECK_BIN, ctr)) {
          const uint32_t pc = __float_as_uint(v4.z);
          atomicAdd(c.guide_hist + (size_t)pc * GUIDE_BINS + __float_as_int(v4.w), wdep);
          c.guide_dirty[pc] = 1;
        }
      }
    }

    // ---- iteration counters, kept per thread over all chunks of the launch
    if (active && (flags & F_TRACED)) ++acc.n_traced;
    if (active && (flags & F_EST)) {
      ++acc.n_est;
      acc.sb0 += bt[0];
      acc.sb1 += bt[1];
      acc.sb2 += bt[2];
    }
    if (active && camera) acc.n_rays += 1u + csub;

    // ---- local statistics: reduce runs of equal cells, then float64 atomics
    if (collect) {
      const unsigned any = __ballot_sync(FULL, key != 0xffffffffu);
      if (any) {
        const uint32_t prev = __shfl_up_sync(FULL, key, 1);
        const bool head = lane == 0 || prev != key;
        const unsigned heads = __ballot_sync(FULL, head);
        // a run of two or more lanes with statistics is the only case that needs
        // the segmented scan (in deep waves neighbouring vertices rarely share a cell)
        const bool pairs = __any_sync(FULL, !head && key != 0xffffffffu);
        const unsigned below = lane == 31 ? FULL : ((2u << lane) - 1u);
        const int start = 31 - __clz(heads & below);
        const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          if (!slot_on(c.techniques, t)) continue;
          // skip a technique no lane drew, and the scan when every run is one lane
          if (!__any_sync(FULL, st[t][0] > 0.0f)) continue;
          if (pairs) {
#pragma unroll
            for (int k = 0; k < NSTAT; ++k) st[t][k] = seg_scan(st[t][k], lane, start);
          }
          if (tail && key != 0xffffffffu && st[t][0] > 0.0f) {
            if (c.stats32) {
              float4* dst = reinterpret_cast<float4*>(c.stats32 + ((size_t)key * NT + t) * NSTAT);
              atomicAdd(dst, make_float4(st[t][0], st[t][1], st[t][2], st[t][3]));
              atomicAdd(dst + 1, make_float4(st[t][4], st[t][5], st[t][6], st[t][7]));
            } else {
              // structure of arrays: the 8 sums of a record sit in 8 different
              // cache lines, so their atomics do not queue on one line
              const size_t plane = (size_t)c.n_cells * NT;
              double* dst = c.stats + (size_t)key * NT + t;
#pragma unroll
              for (int k = 0; k < NSTAT; ++k) atomicAdd(dst + k * plane, (double)st[t][k]);
            }
          }
        }
      }
    }
  }
}

// the sums of a warp's threads to the iteration's counters
__device__ __forceinline__ void flush_sums(const DevCache& c, const RevSums& acc, bool third) {
  DevCounters* ctr = c.ctr;
  unsigned long long n_traced = acc.n_traced, n_est = acc.n_est, n_rays = acc.n_rays;
  double sb0 = acc.sb0, sb1 = acc.sb1, sb2 = acc.sb2;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    n_traced += __shfl_xor_sync(FULL, n_traced, off);
    n_est += __shfl_xor_sync(FULL, n_est, off);
    n_rays += __shfl_xor_sync(FULL, n_rays, off);
    sb0 += __shfl_xor_sync(FULL, sb0, off);
    sb1 += __shfl_xor_sync(FULL, sb1, off);
    sb2 += __shfl_xor_sync(FULL, sb2, off);
  }
  if ((threadIdx.x & 31) == 0) {
    if (n_traced) atomicAdd(&ctr->vertices, n_traced);
    if (n_est) {
      atomicAdd(&ctr->est_vertices, n_est);
      atomicAdd(&ctr->sum_beta[0], sb0);
      if (c.techniques & MARS_TECH_NEE) atomicAdd(&ctr->sum_beta[1], sb1);
      if (third) atomicAdd(&ctr->sum_beta[2], sb2);
    }
    if (n_rays) atomicAdd(&ctr->rays, n_rays);
  }
}

}  // namespace

}  // namespace mars
