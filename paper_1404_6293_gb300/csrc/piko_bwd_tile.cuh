// piko_bwd_tile.cuh -- gradients of the shading, accumulated per screen tile;
// shared by the single-scene and the batch backward kernels.
//
// Visibility is held fixed by the forward key buffer, so coverage stays exact
// integer arithmetic and only the fragment shader is differentiated: for the
// Lambert shader of Listing 1 (rgb = albedo * s, s = max(0, n . L),
// n = sum b_i n_i, albedo = sum b_i c_i) and for Gouraud (rgb = sum b_i c_i).
// Per pixel, with g = dLoss/drgb:
//   dL/dc_i += s * b_i * g        (Gouraud: b_i * g)
//   dL/dn_i += (g . albedo) b_i L   when s > 0 (or unclamped)
//   dL/dL   += (g . albedo) n
//
// The normal and light gradients are linear in the sums of G b_i, G = g .
// albedo, so a vertex needs four sums only: three of the colour and one of G.
// They live in an accumulator of one float4 per vertex (GradAcc below), which
// a pass over the vertices (grad_finish_chunk) turns into the three gradient
// arrays and leaves zero for the next call.
//
// A warp takes a 16 x 2 block of pixels.  Lanes next to each other in a row
// whose pixels share a winning triangle (a run) are summed by shuffles, in as
// many steps as the longest run of the warp needs, and the first lane of a run
// adds its sums to the accumulators of the triangle's three vertices.
// (Following columns of a 16 x 32 tile down with the sums in registers, flushed
// when the winner changes, executed twice the instructions on scenes of
// 100-pixel triangles: some lane of the warp flushes in nearly every row.
// Groups of any lanes with one triangle, through shared memory or a reduction
// over the warp per group, took 755 us of a batch of 64 uneven scenes against
// 614 for the runs.)
#pragma once

#include <cooperative_groups.h>

#include "piko_internal.cuh"

namespace piko {

// Terms per pixel: q = 3 c + j (c < 3) is g_c s b_j, the colour gradient of
// vertex j (g_c b_j for Gouraud); q = 9 + j is G b_j with G = g . albedo
// (0 where the clamp is inactive).  The normal and light gradients are
// linear in the G b_j sums: dL/dn_j = L sum(G b_j) and dL/dL = sum_j n_j
// sum(G b_j), so they are formed once per vertex from the sums.
constexpr int BWD_VALS = 12;
constexpr unsigned BWD_NONE = 0xFFFFFFFFu;

struct BwdScene {
  int W, H, mode, unclamped, T, V;
  const int* tris;
  const int4* vtx;
  const float* color;
  const float* invw;  // 1 / clip w per vertex: perspective-correct attributes (NULL: screen-space)
  const float4* pos;  // near/far clipping: positions and matrix of clipped winners (NULL: off)
  const float* mvp;
  const unsigned long long* key;
  const float4* dl;
  float4* acc;  // per vertex: sums of g s b (colour) and of G b (zero between calls)
  int copies;   // of acc, V apart
};

// ------------------------------------------------------------ accumulators
// One 16-byte vector reduction per vertex and flushed run.  The L2 takes a
// reduction per sector and instruction, whatever its width: adding the 18
// scalars of a run (9 colour, 9 normal) one by one kept it at its limit, and
// three vector reductions carry the same sums.
__device__ __forceinline__ void grad_add(float4* acc, float c0, float c1, float c2, float G) {
  if (c0 != 0.f || c1 != 0.f || c2 != 0.f || G != 0.f)
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(acc), "f"(c0), "f"(c1), "f"(c2), "f"(G)
                 : "memory");
}

// A group of vertices with one accumulator: the vertices of a scene, or of
// several scenes of a batch that share their attributes and gradient arrays.
struct GradAcc {
  int V;
  int copies;  // of the accumulators, V apart (grad_copies)
  float4* acc;
  const float* normal;  // Lambert (NULL for Gouraud: no normal or light gradients)
  const float* light;
  const float* color;  // with attr: what a batch's backward packs per vertex (Lambert)
  float4* attr;
  float* dcolor;   // NULL: not wanted
  float* dnormal;
  float* dlight;
  int set;  // 1: dcolor and dnormal are stored, not added to (dlight is zero before the call)
};

// Copies of a group's accumulators: neighbouring blocks of pixels add to
// different ones, and the finishing pass adds the copies up.  A vertex of
// triangles of hundreds of pixels takes hundreds of sums one after the other
// into one float; with several copies the rounding error falls with their
// number, as does the queue at one address of the L2.  px: pixels of the
// group's framebuffers; room: accumulators that may be used.
//
// A copy per GRAD_COPY_PX pixels a vertex makes a single scene's sums as exact as
// sums over tiles of 16 x 16 pixels (relative error of dL/dcolour at 46 pixels a
// vertex: 1.2e-7, with a copy per 64 pixels 1.7e-7, by tiles 1.4e-7; at 1,180
// pixels a vertex 1.9, 2.7 and 2.4e-7).  Batches are there with a copy per 64
// (1.9e-7 against 2.0e-7 by tiles on 12 uneven scenes); with one per 16, up to 32,
// their finishing pass took 163 us instead of 89 (64 scenes).
constexpr int GRAD_MAX_COPIES = 16, GRAD_COPY_PX = 8;
constexpr int BATCH_MAX_COPIES = 8, BATCH_COPY_PX = 64;
// (A soup's vertices belong to one triangle each and take few sums: with copies
// by the pixels per triangle a batch of 64 uneven scenes took 1684 us, by the
// pixels per vertex, or without, 1624.)
inline int grad_copies(long long px, long long V, long long room, int per_px, int most) {
  int k = 1;
  while (k < most && px >= per_px * k * V && 2 * k * V <= room) k *= 2;
  return k;
}

constexpr int GRAD_CHUNK = 256;  // vertices per CTA step of the finishing pass, one per thread

struct GradFinishSmem {
  float4 a[GRAD_CHUNK];
  float light[GRAD_CHUNK / 32][3];
};

// Vertices [GRAD_CHUNK chunk, + GRAD_CHUNK) of a group; called by a CTA of
// GRAD_CHUNK threads.  The sums go through shared memory so that the
// gradient arrays (three floats a vertex) are added to in whole sectors.
// Atomic, as several calls on different streams may share the arrays.
// lacc: the light gradient's component tid of the CTA's chunks (threads 0 to 2).
// FLIGHT: copies loaded at a time (1: there is only one).
template <int FLIGHT>
__device__ __forceinline__ void grad_finish_chunk(const GradAcc& f, int chunk, GradFinishSmem& sm, double& lacc) {
  const int tid = threadIdx.x, lane = tid & 31, base = chunk * GRAD_CHUNK, v = base + tid;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  bool hit = false;
  auto take = [&](float4* at, const float4& c) {
    if (c.x == 0.f && c.y == 0.f && c.z == 0.f && c.w == 0.f) return;
    hit = true;
    *at = make_float4(0.f, 0.f, 0.f, 0.f);
    a.x += c.x; a.y += c.y; a.z += c.z; a.w += c.w;
  };
  if (v < f.V) {
    float4* at = f.acc + v;
    if (FLIGHT == 1 || f.copies == 1) {
      take(at, __ldcg(at));
    } else if (f.copies < FLIGHT) {  // (a power of two)
      for (int k = 0; k < f.copies; k += 2, at += 2 * (size_t)f.V) {
        const float4 c0 = __ldcg(at), c1 = __ldcg(at + f.V);
        take(at, c0);
        take(at + f.V, c1);
      }
    } else {
      for (int k0 = 0; k0 < f.copies; k0 += FLIGHT, at += FLIGHT * (size_t)f.V) {
        float4 c[FLIGHT];
#pragma unroll
        for (int k = 0; k < FLIGHT; ++k) c[k] = __ldcg(at + (size_t)k * f.V);
#pragma unroll
        for (int k = 0; k < FLIGHT; ++k) take(at + (size_t)k * f.V, c[k]);
      }
    }
  }
  if (!__syncthreads_or(hit) && !f.set) return;  // (the barrier also ends the last chunk's reads of sm)
  sm.a[tid] = a;
  if (f.normal && f.dlight) {
    float g[3] = {0.f, 0.f, 0.f};
    if (a.w != 0.f) {
#pragma unroll
      for (int k = 0; k < 3; ++k) g[k] = a.w * __ldg(f.normal + 3 * (size_t)v + k);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      for (int o = 16; o > 0; o >>= 1) g[k] += __shfl_xor_sync(FULL_MASK, g[k], o);
      if (lane == 0) sm.light[tid >> 5][k] = g[k];
    }
  }
  __syncthreads();
  if (f.normal && f.dlight && tid < 3) {
    for (int w = 0; w < GRAD_CHUNK / 32; ++w) lacc += (double)sm.light[w][tid];
  }
  const float* s = reinterpret_cast<const float*>(sm.a);
  const int n = 3 * min(GRAD_CHUNK, f.V - base);
  for (int i = tid; i < n; i += GRAD_CHUNK) {
    const int q = i / 3, c = i - 3 * q;
    if (f.set) {
      if (f.dcolor) f.dcolor[3 * (size_t)base + i] = s[4 * q + c];
      if (f.normal && f.dnormal) f.dnormal[3 * (size_t)base + i] = s[4 * q + 3] * __ldg(f.light + c);
      continue;
    }
    if (f.dcolor && s[4 * q + c] != 0.f) atomicAdd(f.dcolor + 3 * (size_t)base + i, s[4 * q + c]);
    if (f.normal && f.dnormal && s[4 * q + 3] != 0.f)
      atomicAdd(f.dnormal + 3 * (size_t)base + i, s[4 * q + 3] * __ldg(f.light + c));
  }
}

// Adds the light sums of a CTA's chunks of a group to its gradient (threads 0 to 2).
__device__ __forceinline__ void grad_add_light(const GradAcc& f, double lacc) {
  if (f.normal && f.dlight && threadIdx.x < 3 && lacc != 0.0) atomicAdd(f.dlight + threadIdx.x, (float)lacc);
}

// The finishing kernels run in clusters, whose first CTA adds the light sums of all
// that end in its group (joins: this CTA does).  They go into three floats one after
// the other; a fine mesh lost precision with an addition per chunk of vertices (500,000
// vertices, 1920x1080: median error of 30 scenes 6.0e-7 of the gradient, 2.4e-7 with
// one per cluster of four, 4.1e-7 summed over pixels).  Clusters of four only where
// chunks are many: 600,000 vertices take the finishing pass 15 us with them, 12 in
// pairs, 11 without.  cluster_arrive at the kernel's start, this at its end, by every
// thread; f: the CTA's last group (NULL: no chunks).
constexpr int FINISH_CLUSTER = 2, FINISH_CLUSTER_MAX = 4;
__device__ __forceinline__ void cluster_arrive() { cooperative_groups::this_cluster().barrier_arrive(); }
__device__ __forceinline__ void grad_add_light_cluster(const GradAcc* f, double lacc, bool joins) {
  __shared__ double part[FINISH_CLUSTER_MAX - 1][3];  // of the other CTAs, with the first
  const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int rank = (int)cluster.block_rank();
  cluster.barrier_wait();  // the first CTA runs: its shared memory can be written
  if (rank != 0 && threadIdx.x < 3)
    cluster.map_shared_rank(&part[0][0], 0)[3 * (rank - 1) + threadIdx.x] = joins ? lacc : 0.0;
  cluster.sync();
  if (rank == 0) {
    if (threadIdx.x < 3)
      for (int k = 1; k < (int)cluster.num_blocks(); ++k) lacc += part[k - 1][threadIdx.x];
  } else if (joins) {
    return;
  }
  if (f) grad_add_light(*f, lacc);
}

// ---------------------------------------------------------------- pixels
constexpr int PIX_THREADS = 256;     // CTA size of the backward kernels: 8 warps, a block of pixels each
constexpr int PIX_W = 16, PIX_H = 2;  // pixels of a warp

// Pixel (x, y) of each lane (lane mod PIX_W along x).  vattr: colour and n . L
// per vertex; without it vdot: n . L (Lambert).  block: the warp's block of
// pixels, which picks the copy of the accumulators.
template <bool PERSP>
__device__ __forceinline__ void backward_warp_pixels(const BwdScene& sc, const float* __restrict__ vdot,
                                                     const float4* __restrict__ vattr, int x, int y,
                                                     int block) {
  const int lane = threadIdx.x & 31;
  // the key and dL/drgba do not come from the vertex stage before this kernel
  const size_t o = (size_t)y * sc.W + x;
  unsigned t = BWD_NONE;
  float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
  if (x < sc.W && y < sc.H) {
    t = __ldg(reinterpret_cast<const unsigned*>(sc.key) + 2 * o);  // the key's triangle word
    g = __ldg(sc.dl + o);
  }
  // a key naming a triangle outside this scene, or one the vertex stage
  // culls, contributes nothing (it cannot come from this scene's forward)
  bool hit = t < (unsigned)sc.T;
  int ia = 0, ib = 0, ic = 0;
  if (hit) {
    ia = __ldg(sc.tris + 3 * (size_t)t); ib = __ldg(sc.tris + 3 * (size_t)t + 1); ic = __ldg(sc.tris + 3 * (size_t)t + 2);
  }
  pdl_wait();  // snapped vertices and light terms
  pdl_launch_dependents();
  if (hit)
    hit = (unsigned)ia < (unsigned)sc.V && (unsigned)ib < (unsigned)sc.V && (unsigned)ic < (unsigned)sc.V;
  int4 p0 = make_int4(0, 0, 0, 0), p1 = p0, p2 = p0;
  long long A = 0;
  bool clipped = false;
  if (hit) {
    p0 = __ldg(sc.vtx + ia); p1 = __ldg(sc.vtx + ib); p2 = __ldg(sc.vtx + ic);
    // twice the area: negative, like the edge functions below, for a triangle
    // wound the other way
    A = (long long)(p1.x - p0.x) * (p2.y - p0.y) - (long long)(p2.x - p0.x) * (p1.y - p0.y);
    if (A == 0 || !(p0.w & p1.w & p2.w)) {  // a winner the vertex stage rejected was clipped
      clipped = sc.pos != nullptr;
      hit = clipped;
    }
  }
  if (!__any_sync(FULL_MASK, hit)) return;
  if (!hit) t = BWD_NONE;
  float v[BWD_VALS];
#pragma unroll
  for (int q = 0; q < BWD_VALS; ++q) v[q] = 0.f;
  if (hit) {
    const int vid[3] = {ia, ib, ic};
    float b[3];
    if (clipped) {
      clip_ray_weights(sc.pos, sc.mvp, sc.W, sc.H, vid, x, y, b[0], b[1], b[2]);
    } else {
      const int dx1 = p0.x - p2.x, dy1 = p0.y - p2.y, dx2 = p1.x - p0.x, dy2 = p1.y - p0.y;
      const int ux = 256 * x + 128 - p0.x, uy = 256 * y + 128 - p0.y;
      if (A == (long long)(int)A) {  // the covered pixel's edge functions lie in [0, A]: exact in 32 bits
        const float fA = (float)(int)A;
        const int w1 = (int)((unsigned)dx1 * (unsigned)uy - (unsigned)dy1 * (unsigned)ux);
        const int w2 = (int)((unsigned)dx2 * (unsigned)uy - (unsigned)dy2 * (unsigned)ux);
        b[0] = __fdiv_rn((float)((int)A - w1 - w2), fA);
        b[1] = __fdiv_rn((float)w1, fA);
        b[2] = __fdiv_rn((float)w2, fA);
      } else {
        const float fA = f32_from_i64(A);
        const long long w1 = (long long)dx1 * uy - (long long)dy1 * ux, w2 = (long long)dx2 * uy - (long long)dy2 * ux;
        b[0] = __fdiv_rn(f32_from_i64(A - w1 - w2), fA);
        b[1] = __fdiv_rn(f32_from_i64(w1), fA);
        b[2] = __fdiv_rn(f32_from_i64(w2), fA);
      }
      if (PERSP)
        perspective_bary(b[0], b[1], b[2], __ldg(sc.invw + vid[0]), __ldg(sc.invw + vid[1]), __ldg(sc.invw + vid[2]));
    }
    if (sc.mode == PIKO_SHADE_GOURAUD) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        v[j] = g.x * b[j]; v[3 + j] = g.y * b[j]; v[6 + j] = g.z * b[j];
      }
    } else {
      float a0 = 0.80f, a1 = 0.75f, a2 = 0.65f;  // material of Listing 1 without colours
      float d = 0.f;                             // n . L = sum_j b_j (n_j . L), by linearity
      if (sc.color) a0 = a1 = a2 = 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (vattr) {
          const float4 q = __ldg(vattr + vid[j]);
          if (sc.color) {
            a0 += b[j] * q.x; a1 += b[j] * q.y; a2 += b[j] * q.z;
          }
          d += b[j] * q.w;
          continue;
        }
        if (sc.color) {
          const float* c = sc.color + 3 * (size_t)vid[j];
          a0 += b[j] * __ldg(c); a1 += b[j] * __ldg(c + 1); a2 += b[j] * __ldg(c + 2);
        }
        d += b[j] * __ldg(vdot + vid[j]);
      }
      const bool active = sc.unclamped || d > 0.f;
      const float sh = sc.unclamped ? d : fmaxf(d, 0.f);
      const float G = active ? (g.x * a0 + g.y * a1 + g.z * a2) : 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (sc.color) {
          v[j] = g.x * sh * b[j]; v[3 + j] = g.y * sh * b[j]; v[6 + j] = g.z * sh * b[j];
        }
        v[9 + j] = G * b[j];
      }
    }
  }
  const unsigned before = __shfl_up_sync(FULL_MASK, t, 1);
  const unsigned heads = __ballot_sync(FULL_MASK, (lane & (PIX_W - 1)) == 0 || before != t);
  const unsigned after = heads & ~((2u << lane) - 1u);  // runs that start behind this lane
  const int end = after ? __ffs(after) - 1 : 32;        // one past this lane's run
#pragma unroll
  for (int o = 1; o < PIX_W; o <<= 1) {
    const bool add = hit && lane + o < end;
    if (!__any_sync(FULL_MASK, add)) break;
#pragma unroll
    for (int q = 0; q < BWD_VALS; ++q) {
      const float u = __shfl_down_sync(FULL_MASK, v[q], o);
      if (add) v[q] += u;
    }
  }
  if (hit && ((heads >> lane) & 1u)) {
    float4* acc = sc.acc + (size_t)(block & (sc.copies - 1)) * sc.V;
    grad_add(acc + ia, v[0], v[3], v[6], v[9]);
    grad_add(acc + ib, v[1], v[4], v[7], v[10]);
    grad_add(acc + ic, v[2], v[5], v[8], v[11]);
  }
}

}  // namespace piko
