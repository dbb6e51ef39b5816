// piko_batch.cu -- many scenes in one pass.
//
// All scenes of a batch share one index space per phase: vertices,
// triangles, bins and tiles of scene s follow those of scenes 0..s-1, and a
// work item finds its scene by binary search over the prefix counts.  The
// phases are those of the single-scene forward (vertex stage, setup and
// counts, scan, scatter, Process), a launch each, or one persistent cooperative
// launch whose CTAs meet at grid barriers between phases.  The Piko paper's
// runtime is multi-kernel and names a persistent kernel as the alternative it
// did not take (Sec. 5); the per-scene bin size and schedule
// are the knobs its Sec. 7.2 explores by hand.
//
// Every wait (grid barrier, scan look-back) is bounded by a clock budget;
// on expiry PIKO_ERR_TIMEOUT is recorded and every later phase is skipped.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <string>
#include <vector>

#include "piko_direct.cuh"
#include "piko_scan.cuh"
#include "piko_bwd_tile.cuh"

namespace piko {

struct BatchScene {
  RasterGeom g;
  int V, T, mode, schedule;
  int vtx_base, tri_base, bin_base;
  int direct;         // small triangles are rasterized by the count pass (piko_direct.cuh)
  unsigned key_base;  // into the direct keys
  int unclamped;  // Lambert without the clamp (the handle's option)
  const float4* pos;
  const int* tris;
  const float* mvp;
  const float* color;
  const float* normal;
  const float* light;
  unsigned long long* key_out;
  float4* rgba_out;
  uint2* gnorm_out;
  uint2* galb_out;
  // backward
  const float4* dl;
  float4* acc;  // the gradient sums of the scene's vertices (NULL: no gradients wanted)
  int copies;   // of acc, V apart
  const float4* attr;  // colour and n . L of the vertices for the backward (Lambert)
};

struct BatchSync {
  unsigned count;     // CTAs arrived at the current grid barrier
  unsigned gen;       // barrier generation
  unsigned dyn_head;  // dynamic tile queue
  unsigned epoch;     // tag of the scan's chunk states; each count phase advances it (never cleared)
};

struct BatchParams {
  int n;
  const BatchScene* sc;    // [n]
  const int* vtx_prefix;   // [n+1] each
  const int* tri_prefix;
  const int* bin_prefix;
  const int* stat_prefix;  // tiles of static scenes
  const int* dyn_prefix;   // tiles of dynamic scenes
  const int* pblock_prefix;  // 16 x 2 pixel blocks (backward)
  int total_pblocks;
  int total_v, total_t, total_bins, total_static, total_dyn;
  int4* vtx;
  float4* vattr;  // colour and n . L per vertex (Lambert; the colour only where the scene has one)
  float* invw;  // 1 / clip w per vertex (perspective-correct attributes), else NULL
  BinRect* rect;
  unsigned char* marks;  // a byte per 32 triangles: 1 where some of them have bin entries (else their rects are not written)
  unsigned long long* dkeys;  // a key per pixel of the scenes with direct rasterization
  unsigned total_dkeys;
  unsigned* cnt;  // 2 * total_bins, zero between frames
  unsigned* bin_off;
  unsigned* cursor;
  unsigned long long* chunk_state;
  unsigned* bin_tris;
  unsigned long long capacity;
  DevStatus* st;
  BatchSync* sync;
  int max_bin_px;
  long long wait_budget;  // clock cycles a device-side wait may take before PIKO_ERR_TIMEOUT
  int withhold;           // test hooks: TEST_WITHHOLD_* bits (piko_scan.cuh)
};

// largest s with prefix[s] <= i (prefix[n] > i)
__device__ __forceinline__ int find_scene(const int* __restrict__ prefix, int n, int i) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(prefix + mid) <= i) lo = mid;
    else hi = mid;
  }
  return lo;
}

// find_scene for the item base + lane of a warp: one search, of the warp's
// first item with every lane reading the same words, and a step per scene
// boundary inside the warp (base is below the batch's total)
__device__ __forceinline__ int find_scene_lane(const int* __restrict__ prefix, int n, int base, int i) {
  int s = find_scene(prefix, n, base);
  while (s + 1 < n && __ldg(prefix + s + 1) <= i) ++s;
  return s;
}

__device__ __forceinline__ bool skip_flags(const DevStatus* st) {
  return (*reinterpret_cast<const volatile unsigned*>(&st->flags) & STATUS_SKIP_MASK) != 0u;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid barrier of a co-resident grid.  Returns false (for every thread of
// the CTA) when the frame must stop: a wait ran out of its budget or an
// earlier phase recorded a condition that makes later phases unsafe.
// skip_arrival (a test hook) makes this CTA wait without arriving, so that
// every CTA's wait runs out.
__device__ bool grid_barrier(BatchSync* sync, DevStatus* st, long long budget, bool skip_arrival = false) {
  __shared__ int s_go;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned gen = ld_acquire_u32(&sync->gen);
    __threadfence();
    if (!skip_arrival && atomicAdd(&sync->count, 1u) == gridDim.x - 1) {
      sync->count = 0u;
      __threadfence();
      st_release_u32(&sync->gen, gen + 1u);
    } else {
      const long long t0 = clock64();
      while (ld_acquire_u32(&sync->gen) == gen) {
        if (clock64() - t0 > budget) {
          record_error(st, PIKO_ERR_TIMEOUT);
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
    s_go = skip_flags(st) ? 0 : 1;  // one read per CTA: every thread takes the same branch
  }
  __syncthreads();
  return s_go != 0;
}

// The same stop test outside a barrier, uniform over the CTA.
__device__ bool cta_should_stop(const DevStatus* st) {
  __shared__ int s_stop;
  __syncthreads();
  if (threadIdx.x == 0) s_stop = skip_flags(st) ? 1 : 0;
  __syncthreads();
  return s_stop != 0;
}

// ------------------------------------------------------------------ phases
template <bool PERSP>
__device__ void phase_vertex(const BatchParams& b) {
  if (b.total_dkeys) clear_keys(b.dkeys, b.total_dkeys);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < b.total_v; i += gridDim.x * blockDim.x) {
    const int s = find_scene_lane(b.vtx_prefix, b.n, i & ~31, i);
    const BatchScene& d = b.sc[s];
    const int v = i - d.vtx_base;
    if (PERSP) {
      float w;
      b.vtx[i] = snap_vertex(__ldg(d.pos + v), d.mvp, (float)d.g.W, (float)d.g.H, &w);
      b.invw[i] = w > 0.0f ? __fdiv_rn(1.0f, w) : 0.0f;
    } else {
      b.vtx[i] = snap_vertex(__ldg(d.pos + v), d.mvp, (float)d.g.W, (float)d.g.H);
    }
    if (d.mode == PIKO_SHADE_LAMBERT && d.normal) {  // (without triangles there may be no normals)
      const float* n = d.normal + 3 * (size_t)v;
      const float* c = d.color + 3 * (size_t)v;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      if (d.color) a = make_float4(__ldg(c), __ldg(c + 1), __ldg(c + 2), 0.f);
      a.w = __ldg(n) * __ldg(d.light) + __ldg(n + 1) * __ldg(d.light + 1) + __ldg(n + 2) * __ldg(d.light + 2);
      b.vattr[i] = a;
    }
  }
}

struct LaneBins {
  bool valid, single;
  int bx0, by0, bx1, by1;
  int nbx, bin_base;
  unsigned dentries;  // bin entries a directly rasterized triangle would have had
};

__device__ __forceinline__ LaneBins no_bins() {
  LaneBins r;
  r.valid = false; r.single = false;
  r.bx0 = 0; r.by0 = 0; r.bx1 = -1; r.by1 = -1; r.nbx = 1; r.bin_base = 0;
  r.dentries = 0u;
  return r;
}

__device__ __forceinline__ LaneBins lane_setup(const BatchParams& b, int t, int lane) {
  LaneBins r = no_bins();
  if (t >= b.total_t) return r;
  const int s = find_scene_lane(b.tri_prefix, b.n, t - lane, t);
  const BatchScene& d = b.sc[s];
  r.nbx = d.g.nbx;
  r.bin_base = d.bin_base;
  const int tl = t - d.tri_base;
  const int3 id = tri_indices(d.tris, (unsigned)tl);
  if ((unsigned)id.x >= (unsigned)d.V || (unsigned)id.y >= (unsigned)d.V || (unsigned)id.z >= (unsigned)d.V) {
    record_error(b.st, PIKO_ERR_BAD_INDEX);
    return r;
  }
  const int4* vtx = b.vtx + d.vtx_base;
  const int4 p0 = __ldg(vtx + id.x), p1 = __ldg(vtx + id.y), p2 = __ldg(vtx + id.z);
  if (!(p0.w & p1.w & p2.w)) return r;
  const int minx = min(p0.x, min(p1.x, p2.x)), maxx = max(p0.x, max(p1.x, p2.x));
  const int miny = min(p0.y, min(p1.y, p2.y)), maxy = max(p0.y, max(p1.y, p2.y));
  int px0, px1, py0, py1;
  centre_range(minx, maxx, 0, d.g.W - 1, px0, px1);
  centre_range(miny, maxy, 0, d.g.H - 1, py0, py1);
  if (px0 > px1 || py0 > py1) return r;
  r.bx0 = px0 >> d.g.bshift_x; r.bx1 = px1 >> d.g.bshift_x;
  r.by0 = py0 >> d.g.bshift_y; r.by1 = py1 >> d.g.bshift_y;
  if (d.direct && direct_small(maxx - minx, maxy - miny, px0, px1, py0, py1, DIRECT_MAX_PX)) {
    if (direct_triangle(p0, p1, p2, (unsigned)tl, px0, px1, py0, py1, d.g.W, b.dkeys + d.key_base))
      r.dentries = (unsigned)((r.bx1 - r.bx0 + 1) * (r.by1 - r.by0 + 1));
    return r;  // no bin entries
  }
  r.valid = (long long)(p1.x - p0.x) * (p2.y - p0.y) - (long long)(p2.x - p0.x) * (p1.y - p0.y) != 0;
  if (!r.valid) return r;
  r.single = r.bx0 == r.bx1 && r.by0 == r.by1;
  return r;
}

// Pairs (triangle, bin) of multi-bin triangles, spread over the warp.
template <typename F>
__device__ __forceinline__ void for_multi_pairs(const LaneBins& r, int lane, F&& f) {
  const int bw = r.bx1 - r.bx0 + 1;
  const int nb = (r.valid && !r.single) ? bw * (r.by1 - r.by0 + 1) : 0;
  int incl = nb;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(FULL_MASK, incl, o);
    if (lane >= o) incl += u;
  }
  const int total = __shfl_sync(FULL_MASK, incl, 31);
  for (int k0 = 0; k0 < total; k0 += 32) {
    const int k = k0 + lane;
    const int kk = k < total ? k : total - 1;
    int owner = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const int v = __shfl_sync(FULL_MASK, incl, owner + s - 1);
      if (v <= kk) owner += s;
    }
    const int ox = __shfl_sync(FULL_MASK, r.bx0, owner), oy = __shfl_sync(FULL_MASK, r.by0, owner);
    const int obw = __shfl_sync(FULL_MASK, bw, owner);
    const int first = __shfl_sync(FULL_MASK, incl - nb, owner);
    const int onbx = __shfl_sync(FULL_MASK, r.nbx, owner), obase = __shfl_sync(FULL_MASK, r.bin_base, owner);
    if (k < total) {
      const int local = k - first;
      const int yy = local / obw;
      f(owner, obase + (oy + yy) * onbx + ox + (local - yy * obw));
    }
  }
}

__device__ void phase_count(const BatchParams& b) {
  const int lane = threadIdx.x & 31;
  unsigned dentries = 0u;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int warps_total = gridDim.x * (blockDim.x >> 5);
  for (int base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < b.total_t;
       base += warps_total * 32) {
    const int t = base + lane;
    const LaneBins r = lane_setup(b, t, lane);
    dentries += r.dentries;
    const bool any = __any_sync(FULL_MASK, r.valid);
    if (lane == 0) b.marks[base >> 5] = any ? 1 : 0;
    if (!any) continue;  // nothing to bin
    const unsigned bin = r.single ? (unsigned)(r.bin_base + r.by0 * r.nbx + r.bx0) : 0xFFFFFFFFu;
    const unsigned grp = __match_any_sync(FULL_MASK, bin);
    const int leader = __ffs(grp) - 1;
    unsigned slot = 0;
    if (r.single && lane == leader) slot = atomicAdd(b.cnt + bin, (unsigned)__popc(grp));
    slot = __shfl_sync(FULL_MASK, slot, leader) + __popc(grp & lt_mask);
    if (t < b.total_t) {
      BinRect q;
      if (!r.valid) {
        q.lo = 0xFFFFFFFFu; q.hi = 0u;
      } else if (r.single) {
        q.lo = (unsigned)r.bx0 | ((unsigned)r.by0 << 16) | 0x8000u; q.hi = slot;
      } else {
        q.lo = (unsigned)r.bx0 | ((unsigned)r.by0 << 16); q.hi = (unsigned)r.bx1 | ((unsigned)r.by1 << 16);
      }
      b.rect[t] = q;
    }
    for_multi_pairs(r, lane, [&](int, int gbin) { atomicAdd(b.cnt + b.total_bins + gbin, 1u); });
  }
  const unsigned long long sum = __reduce_add_sync(FULL_MASK, dentries);
  if (lane == 0 && sum) atomicAdd(&b.st->direct_entries, sum);
}

// By one thread, before the launch or barrier that the scan waits for.
__device__ void prepare_scan(const BatchParams& b) {
  b.st->scan_ticket = 0u;
  b.sync->epoch += 1u;
}

__device__ void phase_scan(const BatchParams& b, ScanSmem& sm) {
  const int chunk_bins = (int)blockDim.x * SCAN_PER;
  const int nchunks = (b.total_bins + chunk_bins - 1) / chunk_bins;
  // tickets only grow, so a CTA takes at most nchunks + 1 of them; the cap
  // turns a broken ticket counter into a recorded error instead of a spin
  for (int iter = 0;; ++iter) {
    if (threadIdx.x == 0) {
      sm.chunk = (int)atomicAdd(&b.st->scan_ticket, 1u);
      if (iter > nchunks) {
        record_error(b.st, PIKO_ERR_TIMEOUT);
        sm.chunk = nchunks;
      }
    }
    __syncthreads();
    const int chunk = sm.chunk;
    if (chunk < 0 || chunk >= nchunks) break;
    scan_chunk(chunk, nchunks, b.total_bins, b.cnt, b.bin_off, b.cursor, b.capacity, b.st, b.chunk_state, &b.sync->epoch,
               sm, &b.sync->dyn_head, b.wait_budget, b.withhold);
    __syncthreads();  // sm.chunk is rewritten for the next ticket
  }
}

// Bin entries of the 32 triangles from base on.
__device__ __forceinline__ void scatter_triangles(const BatchParams& b, int base, int lane) {
  const int t = base + lane;
  LaneBins r = no_bins();
  if (t < b.total_t) {
    const BinRect q = b.rect[t];
    if (q.lo != 0xFFFFFFFFu) {
      const BatchScene& d = b.sc[find_scene_lane(b.tri_prefix, b.n, base, t)];
      r.valid = true;
      r.nbx = d.g.nbx;
      r.bin_base = d.bin_base;
      if (q.lo & 0x8000u) {
        r.single = true;
        const int gbin = d.bin_base + (int)(q.lo >> 16) * d.g.nbx + (int)(q.lo & 0x7FFFu);
        const unsigned pos = __ldg(b.bin_off + gbin) + q.hi;
        if (pos < b.capacity) b.bin_tris[pos] = (unsigned)t;
      } else {
        r.bx0 = q.lo & 0xFFFF; r.by0 = q.lo >> 16; r.bx1 = q.hi & 0xFFFF; r.by1 = q.hi >> 16;
      }
    }
  }
  for_multi_pairs(r, lane, [&](int owner, int gbin) {
    const unsigned pos = atomicAdd(b.cursor + gbin, 1u);
    if (pos < b.capacity) b.bin_tris[pos] = (unsigned)(base + owner);
  });
}

__device__ void phase_scatter(const BatchParams& b) {
  const int lane = threadIdx.x & 31;
  const int step = gridDim.x * (blockDim.x >> 5) * 32;
  // the marks of the warp's next 32 batches of triangles in one load; unmarked ones are skipped
  for (long long base0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base0 < b.total_t;
       base0 += 32LL * step) {
    const long long mine = base0 + (long long)lane * step;
    for (unsigned m = __ballot_sync(FULL_MASK, mine < b.total_t && __ldcg(b.marks + (mine >> 5)) != 0); m != 0u;
         m &= m - 1u) {
      scatter_triangles(b, (int)(base0 + (long long)(__ffs(m) - 1) * step), lane);
    }
  }
}

struct ProcessShared {
  TileScene sc;
  int tile, scene;
  unsigned nbig;
};

__device__ void load_tile_scene(const BatchParams& b, int s, TileScene& t) {
  const BatchScene& d = b.sc[s];
  t.g = d.g;
  t.mode = d.mode;
  t.unclamped = d.unclamped;
  t.small_px = 32;
  t.tri_base = d.tri_base;
  t.tris = d.tris;
  t.vtx = b.vtx + d.vtx_base;
  t.color = d.color;
  t.normal = d.normal;
  t.light = d.light;
  t.vdot = nullptr;
  t.vattr = b.vattr + d.vtx_base;
  t.invw = b.invw ? b.invw + d.vtx_base : nullptr;
  t.T = d.T;
  t.clip_tris = nullptr;  // batches do not clip
  t.clip_orig = nullptr;
  t.pos = nullptr;
  t.mvp = nullptr;
  t.dkeys = d.direct ? b.dkeys + d.key_base : nullptr;
  t.key_out = d.key_out;
  t.rgba_out = d.rgba_out;
  t.gnorm_out = d.gnorm_out;
  t.galb_out = d.galb_out;
}

template <bool PERSP>
__device__ void process_one(const BatchParams& b, const int* prefix, int i, ProcessShared& ps, const TileSmem& sm,
                            unsigned& big_base) {
  if (threadIdx.x == 0) {
    const int s = find_scene(prefix, b.n, i);
    if (s != ps.scene) {
      load_tile_scene(b, s, ps.sc);
      ps.scene = s;
    }
    ps.tile = i - __ldg(prefix + s);
  }
  __syncthreads();
  const TileScene& sc = ps.sc;
  const int gbin = b.sc[ps.scene].bin_base + ps.tile;
  TileStats st = {0ull, 0ull, 0ull};
  const unsigned beg = __ldg(b.bin_off + gbin), end = __ldg(b.bin_off + gbin + 1);
  if (beg > end || (unsigned long long)end > b.capacity) {  // same for every thread: skip the tile
    if (threadIdx.x == 0) record_error(b.st, PIKO_ERR_OVERFLOW);
    __syncthreads();
    return;
  }
  if (sc.dkeys && beg == end) shade_direct_tile<PERSP, false>(sc, ps.tile);
  process_tile<false, PERSP>(sc, ps.tile, beg, end, b.bin_tris, sm, big_base, st);
}

template <bool PERSP>
__device__ void phase_process(const BatchParams& b, ProcessShared& ps, const TileSmem& sm) {
  for (int i = threadIdx.x; i < b.max_bin_px; i += blockDim.x) sm.skey[i] = KEY_EMPTY;
  if (threadIdx.x == 0) {
    ps.scene = -1;
    *sm.s_nbig = 0u;
  }
  __syncthreads();
  unsigned big_base = 0u;
  // DirectMap scenes: tiles dealt round robin; then LoadBalance scenes from the queue
  for (int i = blockIdx.x; i < b.total_static; i += gridDim.x) process_one<PERSP>(b, b.stat_prefix, i, ps, sm, big_base);
  __shared__ int s_next;
  for (int iter = 0;; ++iter) {
    if (threadIdx.x == 0) {
      s_next = (int)atomicAdd(&b.sync->dyn_head, 1u);
      if (iter > b.total_dyn) {  // the queue only grows: at most total_dyn + 1 takes
        record_error(b.st, PIKO_ERR_TIMEOUT);
        s_next = b.total_dyn;
      }
    }
    __syncthreads();
    const int i = s_next;
    __syncthreads();  // s_next is rewritten for the next tile
    if (i < 0 || i >= b.total_dyn) break;
    process_one<PERSP>(b, b.dyn_prefix, i, ps, sm, big_base);
  }
}

#ifndef PIKO_BATCH_MAXNREG
#define PIKO_BATCH_MAXNREG 64
#endif
#ifndef PIKO_BATCH_THREADS
#define PIKO_BATCH_THREADS 128
#endif
constexpr int BATCH_THREADS = PIKO_BATCH_THREADS;  // CTA size of the batch's scan and Process phases, and of its persistent kernel

struct BatchSmem {
  ProcessShared ps;
  unsigned nbig;
};
__device__ __forceinline__ TileSmem batch_tile_smem(const BatchParams& b, unsigned long long* smem, BatchSmem& bs) {
  TileSmem sm;
  sm.skey = smem;
  sm.sbig = reinterpret_cast<int*>(smem + b.max_bin_px);
  sm.sfrag = sm.sbig + blockDim.x;
  sm.s_nbig = &bs.nbig;
  return sm;
}

// All phases in one cooperative launch.  PERSP: perspective-correct attributes;
// one instance per setting
template <bool PERSP>
__global__ void __maxnreg__(PIKO_BATCH_MAXNREG) k_batch_forward(BatchParams b) {
  extern __shared__ __align__(16) unsigned long long smem[];
  __shared__ ScanSmem scan_sm;
  __shared__ BatchSmem bsm;
  const TileSmem sm = batch_tile_smem(b, smem, bsm);
  if (cta_should_stop(b.st)) return;
  phase_vertex<PERSP>(b);
  const bool skip = (b.withhold & TEST_WITHHOLD_BARRIER) && blockIdx.x == 0;
  if (!grid_barrier(b.sync, b.st, b.wait_budget, skip)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) prepare_scan(b);  // the scan runs after a barrier
  phase_count(b);
  if (!grid_barrier(b.sync, b.st, b.wait_budget)) return;
  phase_scan(b, scan_sm);
  if (!grid_barrier(b.sync, b.st, b.wait_budget)) return;
  if (cta_should_stop(b.st)) return;
  phase_scatter(b);
  if (!grid_barrier(b.sync, b.st, b.wait_budget)) return;
  if (cta_should_stop(b.st)) return;
  phase_process<PERSP>(b, bsm.ps, sm);
}

// One launch per phase (the default), each with the registers and threads that suit it: in
// the persistent kernel every phase runs at the Process stage's 64 registers,
// with half the warps that the gathers of the first ones want in flight.
template <bool PERSP>
__global__ void __launch_bounds__(256, 8) k_batch_vertex(BatchParams b) {
  pdl_launch_dependents();
  if (!cta_should_stop(b.st)) phase_vertex<PERSP>(b);
}
__global__ void __launch_bounds__(256, 4) k_batch_count(BatchParams b) {
  pdl_wait();
  pdl_launch_dependents();
  if (cta_should_stop(b.st)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) prepare_scan(b);  // the scan runs after this kernel
  phase_count(b);
}
__global__ void __launch_bounds__(BATCH_THREADS) k_batch_scan(BatchParams b) {
  __shared__ ScanSmem scan_sm;
  pdl_wait();
  pdl_launch_dependents();
  if (!cta_should_stop(b.st)) phase_scan(b, scan_sm);
}
__global__ void __launch_bounds__(256, 6) k_batch_scatter(BatchParams b) {
  pdl_wait();
  pdl_launch_dependents();
  if (!cta_should_stop(b.st)) phase_scatter(b);
}
template <bool PERSP>
__global__ void __maxnreg__(PIKO_BATCH_MAXNREG) k_batch_process(BatchParams b) {
  extern __shared__ __align__(16) unsigned long long smem[];
  __shared__ BatchSmem bsm;
  const TileSmem sm = batch_tile_smem(b, smem, bsm);
  pdl_wait();
  if (!cta_should_stop(b.st)) phase_process<PERSP>(b, bsm.ps, sm);
}

// ------------------------------------------------------------------ backward
// 16 x 2 blocks of pixels of every scene; the gradients are accumulated as in
// the single-scene backward.
struct BatchBwdParams {
  int n;
  const BatchScene* sc;
  const int* pblock_prefix;  // [n+1] 16 x 2 pixel blocks per scene
  int total_pblocks;
  const int4* vtx;
  const float* invw;  // as in BatchParams
  // accumulators (GradAcc) of the finishing pass and the prefix of their chunks
  int ngroups, total_chunks;
  const GradAcc* groups;
  const int* chunk_prefix;
};

__device__ __forceinline__ void fill_bwd_scene(const BatchBwdParams& b, const BatchScene& d, BwdScene& c) {
  c.W = d.g.W; c.H = d.g.H; c.mode = d.mode; c.unclamped = d.unclamped; c.T = d.T; c.V = d.V;
  c.tris = d.tris; c.vtx = b.vtx + d.vtx_base; c.color = d.color;
  c.invw = b.invw ? b.invw + d.vtx_base : nullptr;
  c.pos = nullptr;  // batches do not clip
  c.mvp = nullptr;
  c.key = d.key_out; c.dl = d.dl; c.acc = d.acc; c.copies = d.copies;
}

// Colour and n . L of the vertices of each group of Lambert scenes: the
// attributes may have changed since the forward pass.  One 16-byte gather per
// vertex then serves a pixel in place of six words (the pixel kernel was at 82%
// of the L1's throughput with those).
__global__ void __launch_bounds__(GRAD_CHUNK) k_batch_attributes(BatchBwdParams b) {
  // chunks in a row per CTA, so that it looks its group up once
  const int per = (b.total_chunks + (int)gridDim.x - 1) / (int)gridDim.x, first = (int)blockIdx.x * per;
  if (first >= b.total_chunks) return;
  int g = find_scene(b.chunk_prefix, b.ngroups, first);
  for (int i = first; i < min(first + per, b.total_chunks); ++i) {
    while (__ldg(b.chunk_prefix + g + 1) <= i) ++g;
    const GradAcc& f = b.groups[g];
    const int v = (i - __ldg(b.chunk_prefix + g)) * GRAD_CHUNK + (int)threadIdx.x;
    if (!f.normal || v >= f.V) continue;
    const float *n = f.normal + 3 * (size_t)v, *c = f.color + 3 * (size_t)v;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (f.color) a = make_float4(__ldg(c), __ldg(c + 1), __ldg(c + 2), 0.f);
    a.w = __ldg(n) * __ldg(f.light) + __ldg(n + 1) * __ldg(f.light + 1) + __ldg(n + 2) * __ldg(f.light + 2);
    f.attr[v] = a;
  }
}

// A warp takes BATCH_PIX_RUN blocks of 16 x 2 pixels in a row, so
// that it looks its scene up once for most of them.
constexpr int BATCH_PIX_RUN = 8;
template <bool PERSP>
__global__ void __launch_bounds__(PIX_THREADS, 4) k_batch_backward_pixel(BatchBwdParams b) {
  __shared__ BwdScene ssc[PIX_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int first = (blockIdx.x * (PIX_THREADS / 32) + warp) * BATCH_PIX_RUN;
  if (first >= b.total_pblocks) return;  // the same for the whole warp
  BwdScene& c = ssc[warp];
  int s = find_scene(b.pblock_prefix, b.n, first), held = -1;
  for (int i = first; i < min(first + BATCH_PIX_RUN, b.total_pblocks); ++i) {
    while (s + 1 < b.n && __ldg(b.pblock_prefix + s + 1) <= i) ++s;
    const BatchScene& d = b.sc[s];
    if (d.acc == nullptr) continue;
    if (s != held) {
      __syncwarp();  // the previous scene's reads of c are done
      if (lane == 0) fill_bwd_scene(b, d, c);
      __syncwarp();
      held = s;
    }
    const int lt = i - __ldg(b.pblock_prefix + s);
    const int ntx = (c.W + PIX_W - 1) / PIX_W;
    const int ty = lt / ntx, tx = lt - ty * ntx;
    backward_warp_pixels<PERSP>(c, nullptr, d.attr, tx * PIX_W + (lane & (PIX_W - 1)), ty * PIX_H + lane / PIX_W,
                                tx + ty);
  }
}

// Sums of all vertices into the gradient arrays, a chunk of one group per CTA step.
__global__ void __launch_bounds__(GRAD_CHUNK, 8) k_batch_finish(BatchBwdParams b) {
  __shared__ GradFinishSmem sm;
  cluster_arrive();
  pdl_wait();  // the accumulators
  const int per = (b.total_chunks + (int)gridDim.x - 1) / (int)gridDim.x;
  auto end_of = [&](int cta) { return min((cta + 1) * per, b.total_chunks); };  // one past a CTA's last chunk
  const int first = (int)blockIdx.x * per, end = end_of(blockIdx.x);
  const bool any = first < end;
  int g = any ? find_scene(b.chunk_prefix, b.ngroups, first) : 0;
  double lacc = 0.0;
  for (int i = first; i < end; ++i) {
    if (__ldg(b.chunk_prefix + g + 1) <= i) {  // (every group has a chunk)
      grad_add_light(b.groups[g], lacc);
      lacc = 0.0;
      ++g;
    }
    grad_finish_chunk<4>(b.groups[g], i - __ldg(b.chunk_prefix + g), sm, lacc);
  }
  // whether the last group reaches back to the last chunk of the cluster's first CTA
  const int head_end = end_of((int)blockIdx.x / FINISH_CLUSTER * FINISH_CLUSTER);
  grad_add_light_cluster(any ? b.groups + g : nullptr, lacc, any && __ldg(b.chunk_prefix + g) < head_end);
}

}  // namespace piko

// =====================================================================
// Host side: layout, scratch, launches (called from the C ABI in piko_api.cu)
// =====================================================================

using namespace piko;

namespace {

int ilog2i(int v) {
  int s = 0;
  while ((1 << s) < v) ++s;
  return s;
}

}  // namespace

// Gradient accumulators beyond one per vertex, 16 MB of them at most: copies for
// scenes of few vertices and many pixels (grad_copies), which take fewer than one
// per BATCH_COPY_PX pixels.
constexpr long long BATCH_GACC_EXTRA = 1 << 20;

// Everything the batch keeps between calls; owned by the handle.
struct BatchState {
  // device scratch
  void* desc = nullptr;  // scenes + prefix arrays
  size_t desc_cap = 0;
  int4* vtx = nullptr;
  long long vcap = 0;
  float4* vattr = nullptr;
  long long dcap = 0;
  float* invw = nullptr;
  long long icap = 0;
  BinRect* rect = nullptr;
  long long tcap = 0;
  unsigned* cnt = nullptr;
  unsigned* bin_off = nullptr;
  unsigned* cursor = nullptr;
  unsigned long long* chunk_state = nullptr;
  long long bcap = 0;  // bins
  unsigned* bin_tris = nullptr;
  long long ecap = 0;
  unsigned char* marks = nullptr;
  long long mcap = 0;
  unsigned long long* dkeys = nullptr;  // keys of direct rasterization
  long long dkcap = 0;
  float4* gacc = nullptr;  // gradient sums, zero between calls
  long long gcap = 0;
  bool gacc_dirty = false;  // gacc is not zero: new, or a backward launch failed
  BatchSync* sync = nullptr;
  // host staging (pinned) and the last layout
  void* staging = nullptr;
  size_t staging_cap = 0;
  size_t desc_bytes = 0;   // of the last layout: scenes, 6 prefix arrays, gradient groups and their prefix
  size_t group_off = 0;    // where the gradient groups start
  cudaEvent_t uploaded = nullptr;
  BatchParams params;
  std::vector<BatchScene> host_desc;  // the uploaded descriptors
  size_t smem = 0;
  int grid = 0;
  size_t grid_smem = 0;  // the shared memory that grid was sized for
  int num_sms = 0;
  int n = 0;
  int persp = 0;               // the layout's attribute interpolation (perspective-correct or not)
};

namespace {

template <typename T>
int grow_dev(T** p, long long* cap, long long need, bool zero, std::string& err) {
  if (need <= *cap) return PIKO_OK;
  const long long n = need + need / 4 + 1024;
  if (*p) {
    if (cudaDeviceSynchronize() != cudaSuccess) { err = "synchronize before growing batch scratch"; return PIKO_ERR_CUDA; }
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
  }
  if (cudaMalloc(reinterpret_cast<void**>(p), (size_t)n * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    err = "cudaMalloc of batch scratch failed";
    return PIKO_ERR_OOM;
  }
  if (zero && (cudaMemset(*p, 0, (size_t)n * sizeof(T)) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)) {
    err = "cudaMemset of batch scratch failed";
    return PIKO_ERR_CUDA;
  }
  *cap = n;
  return PIKO_OK;
}

bool valid_bin(int b) { return b == 8 || b == 16 || b == 32 || b == 64; }
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

void batch_state_free(BatchState* bs) {
  if (!bs) return;
  cudaFree(bs->desc);
  cudaFree(bs->vtx);
  cudaFree(bs->vattr);
  cudaFree(bs->invw);
  cudaFree(bs->rect);
  cudaFree(bs->cnt);
  cudaFree(bs->bin_off);
  cudaFree(bs->cursor);
  cudaFree(bs->chunk_state);
  cudaFree(bs->bin_tris);
  cudaFree(bs->gacc);
  cudaFree(bs->dkeys);
  cudaFree(bs->marks);
  cudaFree(bs->sync);
  if (bs->staging) cudaFreeHost(bs->staging);
  if (bs->uploaded) cudaEventDestroy(bs->uploaded);
  cudaGetLastError();
  delete bs;
}

// Builds the descriptors, sizes the scratch and uploads the layout.
// Returns a PIKO_* code; err describes a failure.
int batch_prepare(BatchState*& bs, int num_sms, const piko_scene* scenes, int n, piko_framebuffer* fbs,
                  const int32_t* bin_sizes, const int32_t* schedules, int default_bin_w, int default_bin_h,
                  int default_schedule, int unclamped, int persp, cudaStream_t stream, std::string& err) {
  if (!bs) bs = new BatchState();
  if (n < 1 || !scenes || !fbs) { err = "batch needs n >= 1 scenes and framebuffers"; return PIKO_ERR_INVALID_ARG; }
  std::vector<BatchScene> d(n);
  std::vector<int> pv(n + 1), pt(n + 1), pb(n + 1), ps(n + 1), pd(n + 1), pq(n + 1);
  long long tv = 0, tt = 0, tb = 0, tsd = 0, tdy = 0, tq = 0, tk = 0, px_total = 0;
  int max_bin_px = 64;
  for (int i = 0; i < n; ++i) {
    const piko_scene& s = scenes[i];
    const piko_framebuffer& f = fbs[i];
    const int bw = bin_sizes ? bin_sizes[2 * i] : default_bin_w, bh = bin_sizes ? bin_sizes[2 * i + 1] : default_bin_h;
    int sched = schedules ? schedules[i] : default_schedule;
    if (s.width < 1 || s.height < 1 || s.width > 32767 || s.height > 32767 || !valid_bin(bw) || !valid_bin(bh) ||
        s.num_vertices < 0 || s.num_triangles < 0 || s.reserved != 0 || sched < PIKO_SCHED_STATIC ||
        sched > PIKO_SCHED_HARDWARE || s.shade_mode < PIKO_SHADE_GOURAUD || s.shade_mode > PIKO_SHADE_GBUFFER ||
        !f.key || (s.num_vertices > 0 && (!s.pos || !aligned16(s.pos))) || (s.num_triangles > 0 && !s.tris) ||
        (s.num_triangles > 0 && s.shade_mode == PIKO_SHADE_GOURAUD && !s.color) ||
        (s.num_triangles > 0 && s.shade_mode != PIKO_SHADE_GOURAUD && !s.normal) ||
        (s.shade_mode == PIKO_SHADE_LAMBERT && !s.light_dir) ||
        (s.shade_mode == PIKO_SHADE_GBUFFER && (!f.gbuf_normal || !f.gbuf_albedo))) {
      err = "invalid scene " + std::to_string(i) + " in batch";
      return PIKO_ERR_INVALID_ARG;
    }
    if (sched == PIKO_SCHED_HARDWARE) sched = PIKO_SCHED_DYNAMIC;
    BatchScene& x = d[i];
    std::memset(&x, 0, sizeof(x));
    x.g.W = s.width; x.g.H = s.height;
    x.g.bshift_x = ilog2i(bw); x.g.bshift_y = ilog2i(bh);
    x.g.nbx = (s.width + bw - 1) / bw; x.g.nby = (s.height + bh - 1) / bh;
    x.V = s.num_vertices; x.T = s.num_triangles; x.mode = s.shade_mode; x.schedule = sched;
    x.vtx_base = (int)tv; x.tri_base = (int)tt; x.bin_base = (int)tb;
    // key indices are 32-bit; scenes past that, or without the memory below, bin every triangle
    const long long px = (long long)s.width * s.height;
    px_total += px;
    if (direct_scene(x.T, x.V, px, true) && tk + px < (1LL << 32)) {
      x.direct = 1;
      x.key_base = (unsigned)tk;
      tk += px;
    }
    x.unclamped = unclamped;
    x.pos = reinterpret_cast<const float4*>(s.pos);
    x.tris = s.tris; x.mvp = s.mvp; x.color = s.color; x.normal = s.normal; x.light = s.light_dir;
    x.key_out = reinterpret_cast<unsigned long long*>(f.key);
    x.rgba_out = reinterpret_cast<float4*>(f.rgba);
    x.gnorm_out = reinterpret_cast<uint2*>(f.gbuf_normal);
    x.galb_out = reinterpret_cast<uint2*>(f.gbuf_albedo);
    const int ntiles = x.g.nbx * x.g.nby;
    pv[i] = (int)tv; pt[i] = (int)tt; pb[i] = (int)tb; ps[i] = (int)tsd; pd[i] = (int)tdy; pq[i] = (int)tq;
    tv += x.V; tt += x.T; tb += ntiles;
    tq += (long long)((s.width + PIX_W - 1) / PIX_W) * ((s.height + PIX_H - 1) / PIX_H);
    if (sched == PIKO_SCHED_STATIC) tsd += ntiles;
    else tdy += ntiles;
    if (bw * bh > max_bin_px) max_bin_px = bw * bh;
  }
  pv[n] = (int)tv; pt[n] = (int)tt; pb[n] = (int)tb; ps[n] = (int)tsd; pd[n] = (int)tdy; pq[n] = (int)tq;
  if (tv >= (1LL << 31) || tt >= (1LL << 31) || tb >= (1LL << 31) || tq >= (1LL << 31)) {
    err = "batch too large (a total reaches 2^31)";
    return PIKO_ERR_INVALID_ARG;
  }
  // device scratch
  int r;
  if ((r = grow_dev(&bs->vtx, &bs->vcap, tv, false, err)) != PIKO_OK) return r;
  if ((r = grow_dev(&bs->vattr, &bs->dcap, tv, false, err)) != PIKO_OK) return r;
  if (persp && (r = grow_dev(&bs->invw, &bs->icap, tv, false, err)) != PIKO_OK) return r;
  if ((r = grow_dev(&bs->rect, &bs->tcap, tt, false, err)) != PIKO_OK) return r;
  if ((r = grow_dev(&bs->marks, &bs->mcap, (tt + 31) / 32, false, err)) != PIKO_OK) return r;
  // here and not in the backward call, which may be recorded into a graph
  const long long copies = std::min(std::min(px_total / BATCH_COPY_PX, (BATCH_MAX_COPIES - 1) * tv), BATCH_GACC_EXTRA);
  if (tv + copies > bs->gcap) bs->gacc_dirty = true;
  if ((r = grow_dev(&bs->gacc, &bs->gcap, tv + copies, false, err)) != PIKO_OK) return r;
  if (tb > bs->bcap) {
    // counts must start at zero; offsets/cursors/chunk states are rewritten
    cudaFree(bs->cnt); cudaFree(bs->bin_off); cudaFree(bs->cursor); cudaFree(bs->chunk_state);
    bs->cnt = nullptr; bs->bin_off = nullptr; bs->cursor = nullptr; bs->chunk_state = nullptr;
    const long long cap = tb + tb / 4 + 1024;
    const long long chunks = cap / (BATCH_THREADS * SCAN_PER) + 2;
    if (cudaMalloc(&bs->cnt, sizeof(unsigned) * 2 * (size_t)cap) != cudaSuccess ||
        cudaMalloc(&bs->bin_off, sizeof(unsigned) * (size_t)(cap + 1)) != cudaSuccess ||
        cudaMalloc(&bs->cursor, sizeof(unsigned) * (size_t)cap) != cudaSuccess ||
        cudaMalloc(&bs->chunk_state, sizeof(unsigned long long) * (size_t)chunks) != cudaSuccess ||
        cudaMemset(bs->cnt, 0, sizeof(unsigned) * 2 * (size_t)cap) != cudaSuccess ||
        cudaMemset(bs->chunk_state, 0, sizeof(unsigned long long) * (size_t)chunks) != cudaSuccess) {
      cudaGetLastError();
      err = "cudaMalloc of batch bins failed";
      return PIKO_ERR_OOM;
    }
    bs->bcap = cap;
  }
  cudaStreamCaptureStatus cap_status = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(stream, &cap_status);
  if (tk > bs->dkcap && (cap_status != cudaStreamCaptureStatusNone ||
                         grow_dev(&bs->dkeys, &bs->dkcap, tk, false, err) != PIKO_OK)) {
    err.clear();
    tk = 0;
    for (BatchScene& x : d) x.direct = 0;
  }
  if (bs->ecap == 0 && (r = grow_dev(&bs->bin_tris, &bs->ecap, 2 * tt + 4096, false, err)) != PIKO_OK) return r;
  if (!bs->sync) {
    if (cudaMalloc(&bs->sync, sizeof(BatchSync)) != cudaSuccess || cudaMemset(bs->sync, 0, sizeof(BatchSync)) != cudaSuccess) {
      err = "cudaMalloc of batch barrier failed";
      return PIKO_ERR_OOM;
    }
  }
  // descriptors + 6 prefix arrays, uploaded from pinned memory; room after
  // them for the backward's gradient groups and their prefix
  const size_t dbytes = sizeof(BatchScene) * n;
  const size_t pbytes = sizeof(int) * (n + 1);
  const size_t group_off = (dbytes + 6 * pbytes + 15) / 16 * 16;
  const size_t total = group_off + sizeof(GradAcc) * n + pbytes;
  if (!bs->uploaded && cudaEventCreateWithFlags(&bs->uploaded, cudaEventDisableTiming) != cudaSuccess) {
    err = "cudaEventCreate failed";
    return PIKO_ERR_CUDA;
  }
  if (cap_status == cudaStreamCaptureStatusNone && bs->staging) cudaEventSynchronize(bs->uploaded);
  if (total > bs->staging_cap) {
    if (cap_status != cudaStreamCaptureStatusNone) {
      err = "batch layout grew during stream capture: call once before capturing";
      return PIKO_ERR_INVALID_ARG;
    }
    if (bs->staging) cudaFreeHost(bs->staging);
    cudaFree(bs->desc);
    bs->staging = nullptr; bs->desc = nullptr; bs->staging_cap = 0;
    const size_t cap = total + total / 2 + 4096;
    if (cudaMallocHost(&bs->staging, cap) != cudaSuccess || cudaMalloc(&bs->desc, cap) != cudaSuccess) {
      err = "allocation of batch descriptors failed";
      return PIKO_ERR_OOM;
    }
    bs->staging_cap = cap;
    bs->desc_cap = cap;
  }
  char* h = static_cast<char*>(bs->staging);
  std::memcpy(h, d.data(), dbytes);
  const std::vector<int>* arrays[6] = {&pv, &pt, &pb, &ps, &pd, &pq};
  for (int a = 0; a < 6; ++a) std::memcpy(h + dbytes + a * pbytes, arrays[a]->data(), pbytes);
  if (cudaMemcpyAsync(bs->desc, bs->staging, group_off, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
      cudaEventRecord(bs->uploaded, stream) != cudaSuccess) {
    err = "upload of batch descriptors failed";
    return PIKO_ERR_CUDA;
  }
  char* dd = static_cast<char*>(bs->desc);
  BatchParams& b = bs->params;
  std::memset(&b, 0, sizeof(b));
  b.n = n;
  b.sc = reinterpret_cast<const BatchScene*>(dd);
  b.vtx_prefix = reinterpret_cast<const int*>(dd + dbytes);
  b.tri_prefix = reinterpret_cast<const int*>(dd + dbytes + pbytes);
  b.bin_prefix = reinterpret_cast<const int*>(dd + dbytes + 2 * pbytes);
  b.stat_prefix = reinterpret_cast<const int*>(dd + dbytes + 3 * pbytes);
  b.dyn_prefix = reinterpret_cast<const int*>(dd + dbytes + 4 * pbytes);
  b.pblock_prefix = reinterpret_cast<const int*>(dd + dbytes + 5 * pbytes);
  b.total_pblocks = (int)tq;
  b.total_v = (int)tv; b.total_t = (int)tt; b.total_bins = (int)tb; b.total_static = (int)tsd;
  b.total_dyn = (int)tdy;
  b.vtx = bs->vtx; b.vattr = bs->vattr; b.invw = persp ? bs->invw : nullptr; b.rect = bs->rect; b.marks = bs->marks; b.cnt = bs->cnt; b.bin_off = bs->bin_off;
  b.dkeys = bs->dkeys; b.total_dkeys = (unsigned)tk;
  b.cursor = bs->cursor; b.chunk_state = bs->chunk_state; b.bin_tris = bs->bin_tris;
  b.capacity = (unsigned long long)bs->ecap; b.sync = bs->sync;
  b.max_bin_px = max_bin_px;
  bs->smem = tile_smem_bytes(max_bin_px, BATCH_THREADS);
  const auto kf = persp ? k_batch_forward<true> : k_batch_forward<false>;
  const auto kp = persp ? k_batch_process<true> : k_batch_process<false>;
  if (bs->smem > 48 * 1024 &&
      (cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bs->smem) != cudaSuccess ||
       cudaFuncSetAttribute(kp, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bs->smem) != cudaSuccess)) {
    err = "batch shared memory request refused";
    return PIKO_ERR_CUDA;
  }
  // (the two kernels share their register cap; the query is repeated only for another layout)
  if (bs->grid == 0 || bs->grid_smem != bs->smem || bs->persp != (persp ? 1 : 0)) {
    int per_sm = 0, per_sm_p = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kf, BATCH_THREADS, bs->smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_p, kp, BATCH_THREADS, bs->smem) != cudaSuccess ||
        per_sm < 1 || per_sm_p < 1) {
      cudaGetLastError();
      err = "batch kernel does not fit on an SM";
      return PIKO_ERR_CUDA;
    }
    bs->grid = (per_sm < per_sm_p ? per_sm : per_sm_p) * num_sms;
    bs->grid_smem = bs->smem;
  }
  bs->num_sms = num_sms;
  bs->desc_bytes = total;
  bs->group_off = group_off;
  bs->n = n;
  bs->persp = persp ? 1 : 0;
  bs->host_desc = d;
  return PIKO_OK;
}

// Launches the forward phases, a launch each; persistent: all in one
// cooperative launch (PIKO_OPT_BATCH_LAUNCH 0).  (The
// separate launches are faster at every size: 49 against 62 us for three scenes
// of 5,000 triangles at most, 407 against 455 for 32 of up to 100,000.)
int batch_launch_forward(BatchState* bs, DevStatus* st, bool persistent, cudaStream_t stream, std::string& err,
                         long long wait_budget, int withhold) {
  BatchParams b = bs->params;
  b.st = st;
  b.wait_budget = wait_budget;
  b.withhold = withhold;
  b.capacity = (unsigned long long)bs->ecap;
  b.bin_tris = bs->bin_tris;
  // (the separate launches use only its queue head, which the scan resets)
  if (persistent && cudaMemsetAsync(bs->sync, 0, offsetof(BatchSync, epoch), stream) != cudaSuccess) {
    err = "batch barrier reset failed";
    return PIKO_ERR_CUDA;
  }
  if (persistent) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(bs->grid);
    cfg.blockDim = dim3(BATCH_THREADS);
    cfg.dynamicSmemBytes = bs->smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, bs->persp ? k_batch_forward<true> : k_batch_forward<false>, b);
    if (e != cudaSuccess) {
      err = std::string("cooperative batch launch: ") + cudaGetErrorString(e);
      return PIKO_ERR_CUDA;
    }
    return PIKO_OK;
  }
  auto blocks_of = [&](long long items, int per_sm) {
    const long long need = (items + 255) / 256, wave = (long long)per_sm * bs->num_sms;
    return (int)(need < 1 ? 1 : (need < wave ? need : wave));
  };
  const long long clear = (long long)b.total_dkeys / 4;
  const int vblocks = blocks_of(b.total_v > clear ? b.total_v : clear, 8);
  cudaError_t e = cudaSuccess;
  if (bs->persp)
    k_batch_vertex<true><<<vblocks, 256, 0, stream>>>(b);
  else
    k_batch_vertex<false><<<vblocks, 256, 0, stream>>>(b);
  if ((e = cudaGetLastError()) == cudaSuccess)
    e = launch_pdl(k_batch_count, blocks_of(b.total_t, 4), 256, 0, stream, b);
  const int chunks = (b.total_bins + BATCH_THREADS * SCAN_PER - 1) / (BATCH_THREADS * SCAN_PER);
  if (e == cudaSuccess)
    e = launch_pdl(k_batch_scan, chunks < bs->grid ? (chunks < 1 ? 1 : chunks) : bs->grid, BATCH_THREADS, 0, stream, b);
  if (e == cudaSuccess) e = launch_pdl(k_batch_scatter, blocks_of(b.total_t, 6), 256, 0, stream, b);
  if (e == cudaSuccess)
    e = launch_pdl(bs->persp ? k_batch_process<true> : k_batch_process<false>, bs->grid, BATCH_THREADS, bs->smem, stream, b);
  if (e != cudaSuccess) {
    err = std::string("batch launch: ") + cudaGetErrorString(e);
    return PIKO_ERR_CUDA;
  }
  return PIKO_OK;
}

long long batch_capacity(const BatchState* bs) { return bs ? bs->ecap : 0; }

int batch_grow_entries(BatchState* bs, long long need, std::string& err) {
  return grow_dev(&bs->bin_tris, &bs->ecap, need, false, err);
}

int batch_launch_backward(BatchState* bs, const piko_scene* scenes, int n, const piko_framebuffer* fbs,
                          const float* const* dl, float* const* dc, float* const* dn, float* const* dlt, int num_sms,
                          cudaStream_t stream, std::string& err) {
  if (!bs || bs->n != n) {
    err = "backward_batch needs a forward_batch of the same scenes first";
    return PIKO_ERR_INVALID_ARG;
  }
  // per-scene accumulators go into the descriptors (same layout); scenes in a
  // row with the same attributes and gradient arrays (views of one mesh) share
  // one group of accumulators, which is finished once
  std::vector<BatchScene> d = bs->host_desc;
  std::vector<GradAcc> groups;
  std::vector<int> chunk_prefix(1, 0);
  std::vector<long long> group_px;
  for (int i = 0; i < n; ++i) {
    if (scenes[i].num_triangles != d[i].T || scenes[i].num_vertices != d[i].V ||
        reinterpret_cast<unsigned long long*>(fbs[i].key) != d[i].key_out) {
      err = "backward_batch scenes differ from the last forward_batch";
      return PIKO_ERR_INVALID_ARG;
    }
    if (dl && dl[i] && !aligned16(dl[i])) {
      err = "dl_drgba must be 16-byte aligned";
      return PIKO_ERR_INVALID_ARG;
    }
    d[i].dl = dl ? reinterpret_cast<const float4*>(dl[i]) : nullptr;
    d[i].color = scenes[i].color;
    d[i].normal = scenes[i].normal;
    d[i].light = scenes[i].light_dir;
    const bool lambert = d[i].mode == PIKO_SHADE_LAMBERT;
    GradAcc g;
    g.V = d[i].V;
    g.set = 0;
    g.normal = lambert ? d[i].normal : nullptr;
    g.light = lambert ? d[i].light : nullptr;
    g.color = lambert ? d[i].color : nullptr;
    g.attr = bs->vattr + d[i].vtx_base;
    g.dcolor = dc && (!lambert || d[i].color) ? dc[i] : nullptr;
    g.dnormal = dn && lambert ? dn[i] : nullptr;
    g.dlight = dlt && lambert ? dlt[i] : nullptr;
    d[i].acc = nullptr;
    d[i].copies = 0;
    d[i].attr = nullptr;
    if (!d[i].dl || d[i].mode == PIKO_SHADE_GBUFFER || g.V == 0 || (!g.dcolor && !g.dnormal && !g.dlight)) continue;
    if (!groups.empty()) {
      const GradAcc& q = groups.back();
      if (q.V == g.V && q.normal == g.normal && q.light == g.light && q.color == g.color && q.dcolor == g.dcolor &&
          q.dnormal == g.dnormal && q.dlight == g.dlight) {
        d[i].attr = q.attr;
        d[i].copies = (int)groups.size();  // (the group, until its accumulators are dealt below)
        group_px.back() += (long long)d[i].g.W * d[i].g.H;
        continue;
      }
    }
    d[i].attr = g.attr;
    groups.push_back(g);
    d[i].copies = (int)groups.size();
    group_px.push_back((long long)d[i].g.W * d[i].g.H);
    chunk_prefix.push_back(chunk_prefix.back() + (g.V + GRAD_CHUNK - 1) / GRAD_CHUNK);
  }
  if (groups.empty()) return PIKO_OK;  // nothing to add
  // accumulators: one per vertex of each group (at most the batch's vertices),
  // and copies from what is left
  long long used = 0, spare = bs->gcap;
  for (const GradAcc& g : groups) spare -= g.V;
  for (size_t k = 0; k < groups.size(); ++k) {
    GradAcc& g = groups[k];
    g.copies = grad_copies(group_px[k], g.V, g.V + spare, BATCH_COPY_PX, BATCH_MAX_COPIES);
    g.acc = bs->gacc + used;
    used += (long long)g.copies * g.V;
    spare -= (long long)(g.copies - 1) * g.V;
  }
  for (BatchScene& x : d) {
    if (x.copies == 0) continue;
    const GradAcc& g = groups[x.copies - 1];
    x.acc = g.acc;
    x.copies = g.copies;
  }
  if (bs->gacc_dirty) {
    if (cudaMemsetAsync(bs->gacc, 0, (size_t)bs->gcap * sizeof(float4), stream) != cudaSuccess) {
      err = "gradient sums reset failed";
      return PIKO_ERR_CUDA;
    }
    // a captured clear has not run
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    bs->gacc_dirty = cudaStreamIsCapturing(stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
  }
  cudaStreamCaptureStatus cap_status = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(stream, &cap_status);
  if (cap_status == cudaStreamCaptureStatusNone) cudaEventSynchronize(bs->uploaded);
  char* h = static_cast<char*>(bs->staging);
  const size_t prefix_off = bs->group_off + sizeof(GradAcc) * n;
  std::memcpy(h, d.data(), sizeof(BatchScene) * n);
  std::memcpy(h + bs->group_off, groups.data(), sizeof(GradAcc) * groups.size());
  std::memcpy(h + prefix_off, chunk_prefix.data(), sizeof(int) * chunk_prefix.size());
  // the prefix arrays of the layout are still in the staging block
  if (cudaMemcpyAsync(bs->desc, bs->staging, bs->desc_bytes, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
      cudaEventRecord(bs->uploaded, stream) != cudaSuccess) {
    err = "upload of backward descriptors failed";
    return PIKO_ERR_CUDA;
  }
  BatchBwdParams p;
  p.n = n;
  p.sc = bs->params.sc;
  p.pblock_prefix = bs->params.pblock_prefix;
  p.total_pblocks = bs->params.total_pblocks;
  p.vtx = bs->vtx;
  p.invw = bs->params.invw;  // the interpolation of the last forward_batch
  p.ngroups = (int)groups.size();
  p.total_chunks = chunk_prefix.back();
  p.groups = reinterpret_cast<const GradAcc*>(static_cast<const char*>(bs->desc) + bs->group_off);
  p.chunk_prefix = reinterpret_cast<const int*>(static_cast<const char*>(bs->desc) + prefix_off);
  const int chunk_blocks = p.total_chunks < 8 * num_sms ? p.total_chunks : 8 * num_sms;
  k_batch_attributes<<<chunk_blocks, GRAD_CHUNK, 0, stream>>>(p);
  const int per_cta = PIX_THREADS / 32 * BATCH_PIX_RUN;
  const int pblocks = (p.total_pblocks + per_cta - 1) / per_cta;
  if (bs->persp)
    k_batch_backward_pixel<true><<<pblocks, PIX_THREADS, 0, stream>>>(p);
  else
    k_batch_backward_pixel<false><<<pblocks, PIX_THREADS, 0, stream>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = launch_pdl_cluster(FINISH_CLUSTER, k_batch_finish, (chunk_blocks + FINISH_CLUSTER - 1) / FINISH_CLUSTER * FINISH_CLUSTER,
                           GRAD_CHUNK, 0, stream, p);
  if (e != cudaSuccess) {
    bs->gacc_dirty = true;
    err = std::string("batch backward launch: ") + cudaGetErrorString(e);
    return PIKO_ERR_CUDA;
  }
  return PIKO_OK;
}
