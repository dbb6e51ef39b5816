// piko_backward.cu -- attribute gradients of one scene through the shading of
// the forward pass (piko_bwd_tile.cuh).
#include "piko_bwd_tile.cuh"

namespace piko {

struct BackwardParams {
  BwdScene sc;
  int ntx, ntiles;
  // per vertex, of the vertex stage (Lambert)
  const float* vdot;    // n . L
  const float4* vattr;  // colour and n . L (NULL: color and vdot)
};

// A warp per 16 x 2 pixels.
template <bool PERSP>
__global__ void __launch_bounds__(PIX_THREADS, 5) k_backward_pixel(const __grid_constant__ BackwardParams p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x * (PIX_THREADS / 32) + warp;
  if (tile >= p.ntiles) return;  // the same for the whole warp
  const int ty = tile / p.ntx, tx = tile - ty * p.ntx;
  backward_warp_pixels<PERSP>(p.sc, p.vdot, p.vattr, tx * PIX_W + (lane & (PIX_W - 1)), ty * PIX_H + lane / PIX_W,
                              tx + ty);
}

// Sums of all vertices into the gradient arrays (grad_finish_chunk).  Copies come
// with few vertices, where the time is that of a chain of loads: eight at a time
// there (16 copies of 3,721 vertices: 6.2 us, 10.7 two at a time), and few enough
// registers for every warp of the SM without copies.
template <bool COPIES>
__global__ void __launch_bounds__(GRAD_CHUNK, COPIES ? 4 : 8)
    k_backward_finish(const __grid_constant__ GradAcc f) {
  __shared__ GradFinishSmem sm;
  cluster_arrive();
  pdl_wait();  // the accumulators
  const int chunks = (f.V + GRAD_CHUNK - 1) / GRAD_CHUNK;
  double lacc = 0.0;
  for (int c = blockIdx.x; c < chunks; c += gridDim.x) grad_finish_chunk<COPIES ? 8 : 1>(f, c, sm, lacc);
  grad_add_light_cluster(&f, lacc, true);
}

}  // namespace piko

using namespace piko;

// acc: acc_room >= V accumulators, zero before and after the call; vdot: n . L per vertex
// of the vertex stage launched just before (Lambert), vattr (or NULL): colour
// and n . L in its place.  set: the gradients are stored (a dlight that is
// wanted being zero already); needs V > 0, T > 0 and a gradient to write.
int piko_backward_launch(int W, int H, int mode, int unclamped, int T, int V, const int* tris, const int4* vtx,
                         const float* vdot, const float4* vattr, const float* color, const float* normal,
                         const float* light,
                         const float* invw, const float* pos, const float* mvp, const unsigned long long* key,
                         const float* dl_drgba, float4* acc, long long acc_room, float* dcolor, float* dnormal,
                         float* dlight, int set, int num_sms, cudaStream_t s) {
  const bool lambert = mode == PIKO_SHADE_LAMBERT;
  GradAcc f;
  f.V = V; f.acc = acc; f.set = set;
  f.copies = grad_copies((long long)W * H, V, acc_room, GRAD_COPY_PX, GRAD_MAX_COPIES);
  f.normal = lambert ? normal : nullptr;
  f.light = light;
  f.color = nullptr;
  f.attr = nullptr;
  f.dcolor = !lambert || color ? dcolor : nullptr;
  f.dnormal = lambert ? dnormal : nullptr;
  f.dlight = lambert ? dlight : nullptr;
  if (V <= 0 || T <= 0 || (!f.dcolor && !f.dnormal && !f.dlight)) return 0;  // nothing to add
  BackwardParams p;
  BwdScene& c = p.sc;
  c.W = W; c.H = H; c.mode = mode; c.unclamped = unclamped; c.T = T; c.V = V;
  c.tris = tris; c.vtx = vtx; c.color = color; c.invw = invw;
  c.pos = reinterpret_cast<const float4*>(pos); c.mvp = mvp;
  c.key = key; c.dl = reinterpret_cast<const float4*>(dl_drgba);
  c.acc = acc; c.copies = f.copies;
  p.vdot = vdot;
  p.vattr = vattr;
  p.ntx = (W + PIX_W - 1) / PIX_W;
  p.ntiles = p.ntx * ((H + PIX_H - 1) / PIX_H);
  const int blocks = (p.ntiles + PIX_THREADS / 32 - 1) / (PIX_THREADS / 32);
  const cudaError_t e =
      launch_pdl(invw ? k_backward_pixel<true> : k_backward_pixel<false>, blocks, PIX_THREADS, 0, s, p);
  if (e != cudaSuccess) return 1;
  const int chunks = (V + GRAD_CHUNK - 1) / GRAD_CHUNK;
  // all CTAs take as many chunks as the fullest: no fewer steps in a row, and fewer
  // additions to the light gradient
  const int steps = (chunks + 8 * num_sms - 1) / (8 * num_sms), ctas = (chunks + steps - 1) / steps;
  const int cluster = chunks > 1024 ? FINISH_CLUSTER_MAX : FINISH_CLUSTER;
  return launch_pdl_cluster(cluster, f.copies > 1 ? k_backward_finish<true> : k_backward_finish<false>,
                            (ctas + cluster - 1) / cluster * cluster, GRAD_CHUNK, 0, s, f) == cudaSuccess
             ? 0
             : 1;
}
