// piko_backward.cu -- attribute gradients of one scene through the shading of
// the forward pass: the tile form (a warp per 16 x 16 tile, piko_bwd_tile.cuh)
// and a per-pixel form for scenes of tiny triangles.
#include "piko_bwd_tile.cuh"

namespace piko {

struct BackwardParams {
  BwdScene sc;
  int ntx, ntiles;
  // per vertex, of the vertex stage (Lambert); pixel form only
  const float* vdot;    // n . L
  const float4* vattr;  // colour and n . L (NULL: color and vdot)
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

// Pixel form (backward_warp_pixels): a warp per 8 x 4 pixels.
template <bool PERSP>
__global__ void __launch_bounds__(PIX_THREADS, 4) k_backward_pixel(const __grid_constant__ BackwardParams p) {
  __shared__ float sval[PIX_THREADS / 32][BWD_VALS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x * (PIX_THREADS / 32) + warp;
  if (tile >= p.ntiles) return;  // the same for the whole warp
  const int ty = tile / p.ntx, tx = tile - ty * p.ntx;
  backward_warp_pixels<PERSP>(p.sc, p.vdot, p.vattr, tx * PIX_W + (lane & (PIX_W - 1)), ty * PIX_H + lane / PIX_W, sval[warp], 0.f,
                              0.f, 0.f);
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
// of the vertex stage launched just before (Lambert), vattr (or NULL): colour
// and n . L in its place.
int piko_backward_launch(int W, int H, int mode, int unclamped, int T, int V, const int* tris, const int4* vtx,
                         const float* vdot, const float4* vattr, const float* color, const float* normal,
                         const float* light,
                         const float* invw, const float* pos, const float* mvp, const unsigned long long* key,
                         const float* dl_drgba, float4* acc, float* dcolor, float* dnormal, float* dlight, int num_sms,
                         cudaStream_t s) {
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
  p.vattr = vattr;
  cudaError_t e;
  if (PIKO_BWD_PIXEL_FORM && bwd_pixel_form(T, W, H)) {
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
