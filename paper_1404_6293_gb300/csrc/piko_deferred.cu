// piko_deferred.cu -- per-pixel light pass over a G-buffer (deferred shading).
//
// Shader complexity measured in number of lights is the axis of the
// paper's Fig. (a) in Sec. 7.2; the supplementary deferred-shading raster
// pipeline the paper mentions in Sec. 7.1 is not printed, so the light model
// is this library's:
//   S = (x + 0.5, y + 0.5, depth / (2^24 - 1) * D),  D = max(W, H),  r = D / 4
//   rgb = albedo * sum_l I_l * max(0, n . (P_l - S) / |P_l - S|) / (1 + |P_l - S|^2 / r^2)
// with n and albedo read from the binary16 G-buffer.  The pass is bound by
// instruction issue (about 20 operations per pixel and light against 24 bytes
// per pixel): lights live in shared memory, two to a record, and a thread
// evaluates two lights of its pixel at a time with packed float32 arithmetic
// (f32x2 instructions: one issue, two results).
#include <cuda_fp16.h>

#include "piko_internal.cuh"

namespace piko {

__device__ __forceinline__ float4 unpack_half4(uint2 v) {
  const __half2 lo = *reinterpret_cast<const __half2*>(&v.x);
  const __half2 hi = *reinterpret_cast<const __half2*>(&v.y);
  const float2 a = __half22float2(lo), b = __half22float2(hi);
  return make_float4(a.x, a.y, b.x, b.y);
}

// Two float32 lanes in one 64-bit register (lo first).
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack(F2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ float rsqrt_normal(float x) {  // x is a normal number
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Two lights: x0 x1 y0 y1 z0 z1 I0 I1.
struct alignas(16) LightPair {
  F2 x, y, z, w;
};

// A light whose terms stay far from float32's ends in light_pairs: position
// within 64 D, not a denormal-sized distance from the plane of depth 0, and a
// finite intensity of ordinary size.  D >= 1 is the larger framebuffer side.
__device__ __forceinline__ bool ordinary_light(float4 p, float D) {
  const float m = 64.0f * D;
  return fabsf(p.x) <= m && fabsf(p.y) <= m && fabsf(p.z) <= m && (p.z == 0.0f || fabsf(p.z) >= 1e-15f) &&
         fabsf(p.w) <= 1e30f;
}

// sum_l I_l max(0, n . d) / (|d| (1 + |d|^2 / r^2)) over pairs of ordinary
// lights.  The two roots and divisions of a term become one reciprocal square
// root: 1 / (|d| t) = rsqrt(|d|^2 t^2), at most 3e24 for ordinary lights; the
// lower clamp only meets d = 0, whose n . d is 0.
__device__ __forceinline__ float light_pairs(const LightPair* lights, int npairs, float4 n, float sx, float sy,
                                             float sz, float inv_r2) {
  const F2 mx = f2(-sx, -sx), my = f2(-sy, -sy), mz = f2(-sz, -sz);
  const F2 nx = f2(n.x, n.x), ny = f2(n.y, n.y), nz = f2(n.z, n.z);
  const F2 ir = f2(inv_r2, inv_r2), one = f2(1.0f, 1.0f);
  F2 acc = f2(0.f, 0.f);
#pragma unroll 4
  for (int l = 0; l < npairs; ++l) {
    const LightPair p = lights[l];
    const F2 dx = add2(p.x, mx), dy = add2(p.y, my), dz = add2(p.z, mz);
    const F2 d2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    const F2 nd = fma2(nz, dz, fma2(ny, dy, mul2(nx, dx)));
    const F2 t = fma2(d2, ir, one);
    float q0, q1, c0, c1;
    unpack(mul2(mul2(d2, t), t), q0, q1);
    unpack(nd, c0, c1);
    const F2 rs = f2(rsqrt_normal(fmaxf(q0, 1.17549435e-38f)), rsqrt_normal(fmaxf(q1, 1.17549435e-38f)));
    acc = fma2(mul2(p.w, f2(fmaxf(c0, 0.f), fmaxf(c1, 0.f))), rs, acc);
  }
  float a0, a1;
  unpack(acc, a0, a1);
  return a0 + a1;
}

// The term of one ordinary light, the first of a record: the last of an odd number.
// (A pair padded with a light of intensity 0 would add 0 * inf = NaN where a
// binary16 normal is infinite.)
__device__ __forceinline__ float light_last(const float* s, float4 n, float sx, float sy, float sz, float inv_r2) {
  const float dx = s[0] - sx, dy = s[2] - sy, dz = s[4] - sz;
  const float d2 = dx * dx + dy * dy + dz * dz;
  const float nd = n.x * dx + n.y * dy + n.z * dz;
  const float t = __fmaf_rn(d2, inv_r2, 1.0f);
  return s[6] * fmaxf(nd, 0.f) * rsqrt_normal(fmaxf(d2 * t * t, 1.17549435e-38f));
}

// The same sum for any lights, one by one.
__device__ __forceinline__ float light_singles(const float4* __restrict__ lights, int n_lights, float4 n, float sx,
                                               float sy, float sz, float inv_r2) {
  float acc = 0.f;
  for (int l = 0; l < n_lights; ++l) {
    const float4 p = __ldg(lights + l);
    const float dx = p.x - sx, dy = p.y - sy, dz = p.z - sz;
    const float d2 = dx * dx + dy * dy + dz * dz;
    const float nd = n.x * dx + n.y * dy + n.z * dz;
    if (d2 > 0.f && nd > 0.f) acc += __fdividef(p.w * nd * rsqrtf(d2), 1.0f + d2 * inv_r2);
  }
  return acc;
}

// One pixel per thread; the CTAs' lights are loaded once per 256 pixels.
__global__ void __launch_bounds__(256) k_deferred_light(int W, int H, const unsigned long long* __restrict__ key,
                                                        const uint2* __restrict__ gnorm,
                                                        const uint2* __restrict__ galb,
                                                        const float4* __restrict__ lights, int n_lights,
                                                        float4* __restrict__ rgba) {
  extern __shared__ __align__(16) float slights[];
  const float D = (float)max(W, H);
  const int npairs = n_lights / 2;
  bool odd_light = false;
  for (int i = threadIdx.x; i < n_lights; i += blockDim.x) {
    const float4 p = lights[i];
    odd_light |= !ordinary_light(p, D);
    float* s = slights + 8 * (i >> 1) + (i & 1);
    s[0] = p.x; s[2] = p.y; s[4] = p.z; s[6] = p.w;
  }
  const bool singles = __syncthreads_or(odd_light);
  const float inv_r2 = 1.0f / ((0.25f * D) * (0.25f * D));
  const float zscale = D / 16777215.0f;
  const int npix = W * H;  // W, H <= 32767
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= npix) return;
  const unsigned long long k = __ldg(key + i);
  if (k == KEY_EMPTY) {
    rgba[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const int y = i / W, x = i - y * W;
  const float4 n = unpack_half4(__ldg(gnorm + i));
  const float4 a = unpack_half4(__ldg(galb + i));
  const float sx = (float)x + 0.5f, sy = (float)y + 0.5f;
  const float sz = (float)(unsigned)(k >> 32) * zscale;
  float acc = 0.f;
  if (singles) {
    acc = light_singles(lights, n_lights, n, sx, sy, sz, inv_r2);
  } else {
    if (n_lights & 1) acc = light_last(slights + 8 * npairs, n, sx, sy, sz, inv_r2);
    acc += light_pairs(reinterpret_cast<const LightPair*>(slights), npairs, n, sx, sy, sz, inv_r2);
  }
  rgba[i] = make_float4(a.x * acc, a.y * acc, a.z * acc, 1.0f);
}

void launch_deferred_light(int W, int H, const unsigned long long* key, const uint2* gnorm, const uint2* galb,
                           const float4* lights, int n_lights, float4* rgba, int num_sms, cudaStream_t s) {
  (void)num_sms;
  const long long npix = (long long)W * H;
  const int blocks = (int)((npix + 255) / 256);
  k_deferred_light<<<blocks, 256, (size_t)((n_lights + 1) / 2) * sizeof(LightPair), s>>>(W, H, key, gnorm, galb, lights,
                                                                                         n_lights, rgba);
}

}  // namespace piko
