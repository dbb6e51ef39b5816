// piko_backward.cu -- attribute gradients of one scene through the shading of
// the forward pass: the tile form (a warp per 16 x 16 tile, piko_bwd_tile.cuh)
// and a per-pixel form for scenes of tiny triangles.
#include "piko_bwd_tile.cuh"

namespace piko {

struct BackwardParams {
  BwdScene sc;
  int ntx, ntiles;
  const float* vdot;  // n . L per vertex (Lambert); per-pixel form only
};

// Warp form (backward_warp_tile): each warp takes whole tiles, grid-stride.
constexpr int BACKWARD_WARPS = BWD_THREADS / 32;
struct BackwardSmem {
  float stage[BACKWARD_WARPS][BWD_VALS][33];
};
#ifndef PIKO_BWD_MINB
#define PIKO_BWD_MINB 3
#endif
template <bool PERSP, bool CLIP>
__global__ void __launch_bounds__(BWD_THREADS, PIKO_BWD_MINB) k_backward(const __grid_constant__ BackwardParams p) {
  extern __shared__ __align__(16) unsigned char bwd_smem_raw[];
  BackwardSmem& sm = *reinterpret_cast<BackwardSmem*>(bwd_smem_raw);
  const int warp = threadIdx.x >> 5;
  pdl_wait();  // snapped vertices
  pdl_launch_dependents();
  float L0 = 0.f, L1 = 0.f, L2 = 0.f;
  if (p.sc.mode == PIKO_SHADE_LAMBERT) {
    L0 = __ldg(p.sc.light); L1 = __ldg(p.sc.light + 1); L2 = __ldg(p.sc.light + 2);
  }
  const int nwarps = gridDim.x * BACKWARD_WARPS;
  for (int tile = blockIdx.x * BACKWARD_WARPS + warp; tile < p.ntiles; tile += nwarps) {
    const int ty = tile / p.ntx, tx = tile - ty * p.ntx;
    backward_warp_tile<PERSP, CLIP>(p.sc, tx * BWD_TILE_W, ty * BWD_TILE_H, sm.stage[warp], L0, L1, L2);
  }
}
constexpr size_t BACKWARD_SMEM = sizeof(BackwardSmem);

// Per-pixel form, for scenes of tiny triangles (a tile would hold nearly as
// many triangles as pixels, so the tile form's runs are a pixel or two long):
// each warp takes an 8 x 4 block of pixels, which shares more winners than a
// row of 32; lanes whose pixels share a winning triangle are summed in shared
// memory and one lane adds the sums to the three vertices' accumulators.
// Bound by the latency of its gathers (key, indices, vertices) and by the L2's
// reductions, so every block is its own warp and CTAs are many.
constexpr int PIX_THREADS = 256;
constexpr int PIX_W = 8, PIX_H = 4;  // pixels of a warp

template <bool PERSP>
__global__ void __launch_bounds__(PIX_THREADS, 4) k_backward_pixel(const __grid_constant__ BackwardParams p) {
  __shared__ float sval[PIX_THREADS / 32][BWD_VALS][32];
  const BwdScene& sc = p.sc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int tile = blockIdx.x * (PIX_THREADS / 32) + warp;
  if (tile >= p.ntiles) return;  // the same for the whole warp
  const int ty = tile / p.ntx, tx = tile - ty * p.ntx;
  const int x = tx * PIX_W + (lane & (PIX_W - 1)), y = ty * PIX_H + lane / PIX_W;
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
  TriSetup s;
  s.v0 = s.v1 = s.v2 = 0;
  bool clipped = false;
  if (hit) {
    const bool in_range = ia >= 0 && ia < sc.V && ib >= 0 && ib < sc.V && ic >= 0 && ic < sc.V;
    hit = in_range && setup_triangle(ia, ib, ic, sc.vtx, s);
    if (!hit && in_range && sc.pos) {  // a winner the vertex stage rejected was clipped
      clipped = hit = true;
      s.v0 = ia; s.v1 = ib; s.v2 = ic;
    }
  }
  if (!hit) t = BWD_NONE;
  float v[BWD_VALS];
#pragma unroll
  for (int q = 0; q < BWD_VALS; ++q) v[q] = 0.f;
  if (hit) {
    const int vid[3] = {s.v0, s.v1, s.v2};
    float b[3];
    if (clipped) {
      clip_ray_weights(sc.pos, sc.mvp, sc.W, sc.H, vid, x, y, b[0], b[1], b[2]);
    } else {
      const float fA = f32_from_i64(s.A);
      if (s.A < (1LL << 31)) {  // the covered pixel's edge functions lie in [0, A]: exact in 32 bits
        const int Px = 256 * x + 128, Py = 256 * y + 128;
        const int w1 = edge_fn_wrap32(s.X2, s.Y2, s.X0, s.Y0, Px, Py), w2 = edge_fn_wrap32(s.X0, s.Y0, s.X1, s.Y1, Px, Py);
        b[0] = __fdiv_rn((float)((int)s.A - w1 - w2), fA);
        b[1] = __fdiv_rn((float)w1, fA);
        b[2] = __fdiv_rn((float)w2, fA);
      } else {
        const long long Px = 256LL * x + 128, Py = 256LL * y + 128;
        const long long w1 = (long long)(s.X0 - s.X2) * (Py - s.Y2) - (long long)(s.Y0 - s.Y2) * (Px - s.X2);
        const long long w2 = (long long)(s.X1 - s.X0) * (Py - s.Y0) - (long long)(s.Y1 - s.Y0) * (Px - s.X0);
        b[0] = __fdiv_rn(f32_from_i64(s.A - w1 - w2), fA);
        b[1] = __fdiv_rn(f32_from_i64(w1), fA);
        b[2] = __fdiv_rn(f32_from_i64(w2), fA);
      }
      if (PERSP)
        perspective_bary(b[0], b[1], b[2], __ldg(sc.invw + vid[0]), __ldg(sc.invw + vid[1]), __ldg(sc.invw + vid[2]));
    }
    if (sc.mode == PIKO_SHADE_GOURAUD) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        v[3 * j] = g.x * b[j]; v[3 * j + 1] = g.y * b[j]; v[3 * j + 2] = g.z * b[j];
      }
    } else {
      float a0 = 0.80f, a1 = 0.75f, a2 = 0.65f;  // material of Listing 1 without colours
      if (sc.color) {
        a0 = a1 = a2 = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const float* c = sc.color + 3 * (size_t)vid[j];
          a0 += b[j] * __ldg(c); a1 += b[j] * __ldg(c + 1); a2 += b[j] * __ldg(c + 2);
        }
      }
      // n . L = sum_j b_j (n_j . L), by linearity
      const float d = b[0] * __ldg(p.vdot + vid[0]) + b[1] * __ldg(p.vdot + vid[1]) + b[2] * __ldg(p.vdot + vid[2]);
      const bool active = sc.unclamped || d > 0.f;
      const float sh = sc.unclamped ? d : fmaxf(d, 0.f);
      const float G = active ? (g.x * a0 + g.y * a1 + g.z * a2) : 0.f;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (sc.color) {
          v[3 * j] = g.x * sh * b[j]; v[3 * j + 1] = g.y * sh * b[j]; v[3 * j + 2] = g.z * sh * b[j];
        }
        v[9 + j] = G * b[j];
      }
    }
  }
  // group lanes by winning triangle; the lowest lane of each group sums
  // the group's contributions and adds them to the vertices
  const unsigned grp = __match_any_sync(FULL_MASK, t);
  const bool leader = hit && (grp & lt_mask) == 0u;
  const bool alone = __popc(grp) == 1;
  if (!alone) {
#pragma unroll
    for (int q = 0; q < BWD_VALS; ++q) sval[warp][q][lane] = v[q];
  }
  __syncwarp();
  if (leader) {
    for (unsigned rest = grp & ~(1u << lane); rest; rest &= rest - 1) {
      const int src = __ffs(rest) - 1;
#pragma unroll
      for (int q = 0; q < BWD_VALS; ++q) v[q] += sval[warp][q][src];
    }
    grad_add(sc.acc + s.v0, v[0], v[1], v[2], v[9]);
    grad_add(sc.acc + s.v1, v[3], v[4], v[5], v[10]);
    grad_add(sc.acc + s.v2, v[6], v[7], v[8], v[11]);
  }
}

// Sums of all vertices into the gradient arrays (grad_finish_chunk).
__global__ void __launch_bounds__(GRAD_CHUNK) k_backward_finish(const __grid_constant__ GradAcc f) {
  __shared__ GradFinishSmem sm;
  pdl_wait();  // the accumulators
  const int chunks = (f.V + GRAD_CHUNK - 1) / GRAD_CHUNK;
  for (int c = blockIdx.x; c < chunks; c += gridDim.x) grad_finish_chunk(f, c, sm);
}

using BackwardKernel = void (*)(BackwardParams);

BackwardKernel backward_kernel(bool persp, bool clip) {
  if (persp) return clip ? k_backward<true, true> : k_backward<true, false>;
  return clip ? k_backward<false, true> : k_backward<false, false>;
}

// Blocks of the single-scene backward kernel: as many as fit on the device
// at once, a tile per warp (the shared-memory opt-in is per device, so it is
// cached per device).
int backward_grid(int tiles, int num_sms) {
  static int per_sm_of[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  int& per_sm = per_sm_of[dev & 63];
  if (per_sm == 0) {
    int v = 0;
    bool ok = true;
    // the instances share the launch bounds and the shared-memory size
    for (int k = 0; k < 4; ++k)
      ok = ok && cudaFuncSetAttribute(backward_kernel(k & 1, k & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)BACKWARD_SMEM) == cudaSuccess;
    if (!ok ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, backward_kernel(false, false), BWD_THREADS,
                                                      BACKWARD_SMEM) != cudaSuccess ||
        v < 1)
      v = 1;
    per_sm = v;
  }
  long long blocks = (long long)per_sm * num_sms;
  const long long need = (tiles + BACKWARD_WARPS - 1) / BACKWARD_WARPS;
  if (blocks > need) blocks = need;
  return blocks < 1 ? 1 : (int)blocks;
}

}  // namespace piko

using namespace piko;

// acc: V accumulators, zero before and after the call; vdot: n . L per vertex
// of the vertex stage launched just before (Lambert).
int piko_backward_launch(int W, int H, int mode, int unclamped, int T, int V, const int* tris, const int4* vtx,
                         const float* vdot, const float* color, const float* normal, const float* light,
                         const float* invw, const float* pos, const float* mvp, const unsigned long long* key,
                         const float* dl_drgba, float4* acc, float* dcolor, float* dnormal, float* dlight, int num_sms,
                         cudaStream_t s) {
  const long long npix = (long long)W * H;
#ifndef PIKO_BWD_PIXEL_FORM  // 0: every scene takes the tile form (for comparisons)
#define PIKO_BWD_PIXEL_FORM 1
#endif
  const bool lambert = mode == PIKO_SHADE_LAMBERT;
  GradAcc f;
  f.V = V; f.acc = acc;
  f.normal = lambert ? normal : nullptr;
  f.light = light;
  f.dcolor = !lambert || color ? dcolor : nullptr;
  f.dnormal = lambert ? dnormal : nullptr;
  f.dlight = lambert ? dlight : nullptr;
  if (V <= 0 || T <= 0 || (!f.dcolor && !f.dnormal && !f.dlight)) return 0;  // nothing to add
  BackwardParams p;
  BwdScene& c = p.sc;
  c.W = W; c.H = H; c.mode = mode; c.unclamped = unclamped; c.T = T; c.V = V;
  c.tris = tris; c.vtx = vtx; c.color = color; c.normal = normal; c.light = light; c.invw = invw;
  c.pos = reinterpret_cast<const float4*>(pos); c.mvp = mvp;
  c.key = key; c.dl = reinterpret_cast<const float4*>(dl_drgba);
  c.acc = acc;
  p.vdot = vdot;
  cudaError_t e;
  if (PIKO_BWD_PIXEL_FORM && 4LL * T > npix) {
    // more than one triangle per four pixels: triangles of a few pixels
    p.ntx = (W + PIX_W - 1) / PIX_W;
    p.ntiles = p.ntx * ((H + PIX_H - 1) / PIX_H);
    const int blocks = (p.ntiles + PIX_THREADS / 32 - 1) / (PIX_THREADS / 32);
    e = launch_pdl(invw ? k_backward_pixel<true> : k_backward_pixel<false>, blocks, PIX_THREADS, 0, s, p);
  } else {
    p.ntx = (W + BWD_TILE_W - 1) / BWD_TILE_W;
    p.ntiles = p.ntx * ((H + BWD_TILE_H - 1) / BWD_TILE_H);
    const int blocks = backward_grid(p.ntiles, num_sms);
    e = launch_pdl(backward_kernel(invw != nullptr, pos != nullptr), blocks, BWD_THREADS, BACKWARD_SMEM, s, p);
  }
  if (e != cudaSuccess) return 1;
  const int chunks = (V + GRAD_CHUNK - 1) / GRAD_CHUNK;
  return launch_pdl(k_backward_finish, chunks < 8 * num_sms ? chunks : 8 * num_sms, GRAD_CHUNK, 0, s, f) == cudaSuccess
             ? 0
             : 1;
}
