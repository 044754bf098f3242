// FP32 CUDA-core fV-SRN kernels: ray-marching render (all shading modes)
// and point evaluation (density, adjoint input gradient).
//
// A warp evaluates the network (Section 3 layer equation, Eq. 1-2 Fourier
// features, Section 4.2 latent grid) for its 32 rays / points as one tile
// (srn_tile32.cuh); rays, features, gathers and compositing are one lane per
// ray / point.  The parameters are staged once per CTA in shared memory, and
// no intermediate state touches global memory (the fused-network idea of
// Section 4).
#pragma once
#include "srn_df.cuh"
#include "srn_fp32.h"
#include "srn_tile32.cuh"

namespace srn {
namespace fp32 {

using namespace net32;

// Rows of 32 floats a warp's tile needs: the inputs and activations share
// one block, unless the backward needs the inputs again.
inline int tile_rows(const tile32::Net& t, int C, bool adjoint, bool dout) {
  return (adjoint ? t.rows + C : (t.rows > C ? t.rows : C)) + (dout ? 4 : 0);
}

// Density (and gradient for shading) at the lanes' positions p + pl (pairs)
// for shading mode SH; the finite-difference neighbours are offset as pairs.
// All lanes of the warp take part.
template <int C, int SH, bool WIDE>
__device__ __forceinline__ float sample_field(const tile32::Ctx& c, float* rows, const Latent& lat, float3 p,
                                              float3 pl, float fd_h, float3& g) {
  constexpr int S = tile32::kPts;
  const tile32::Net& t = *c.t;
  if constexpr (SH == SRN_SHADE_ADJOINT) {
    float* x = rows + t.rows * S;
    tile32::Acc<C> df[kMaxL - 1], a;
    tile32::forward<C, true, WIDE>(c, rows, x, lat, p, pl, df);
    const float rho = tile32::last_layer<C, S>(x, c.sm, t, 0);
    tile32::seed<C>(a, c.sm, t, nullptr);
    g = tile32::input_gradient<C, WIDE>(c, rows, x, lat, p, a, df);
    return rho;
  } else {
    tile32::forward<C, false, WIDE>(c, rows, rows, lat, p, pl, nullptr);
    const float rho = tile32::last_layer<C, S>(rows, c.sm, t, 0);
    if constexpr (SH == SRN_SHADE_HEAD)
      g = make_float3(tile32::last_layer<C, S>(rows, c.sm, t, 1), tile32::last_layer<C, S>(rows, c.sm, t, 2),
                      tile32::last_layer<C, S>(rows, c.sm, t, 3));
    __syncwarp();
    if constexpr (SH == SRN_SHADE_FD) {
      float o[6];
#pragma unroll 1
      for (int k = 0; k < 6; ++k) {
        float3 qh = p, ql = pl;
        df::offset_axis(qh, ql, k >> 1, (k & 1) ? -fd_h : fd_h);
        tile32::forward<C, false, WIDE>(c, rows, rows, lat, qh, ql, nullptr);
        const float v = tile32::last_layer<C, S>(rows, c.sm, t, 0);
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 6; ++e)
          if (e == k) o[e] = v;
      }
      g = make_float3((o[0] - o[1]) / (2.0f * fd_h), (o[2] - o[3]) / (2.0f * fd_h), (o[4] - o[5]) / (2.0f * fd_h));
    }
    return rho;
  }
}

// Render: a warp takes 32 / K rays, K consecutive samples of each at a time
// (K = 1, 2, 4, 8; K lanes per ray, pixel tiles of 8 x 4, 4 x 4, 4 x 2,
// 2 x 2).  The samples of a ray only meet in the compositing, which runs in
// order over the K lanes; samples past the one that ends the ray are dropped
// (at most K - 1 a ray).  Large images take K = 1; small ones have too few
// rays to fill the chip, and their time is a ray's chain of samples.
template <int C, int SH, bool WIDE>
__global__ void __launch_bounds__(32 * tile32::max_warps(C), 1)
    render_fp32_kernel(const NetDev net, const BatchDev b, const tile32::Net t, int rows, int log2k) {
  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  __shared__ TFDev tf;
  load_tf(tf, b.tf);
  tile32::load_net<C>(sm, t, net);
  const tile32::Ctx ctx{sm, &t, net.act, tile32::nerf_rows(sm + t.oF, t.m)};
  float* mine = sm + t.total + (threadIdx.x >> 5) * rows * tile32::kPts;

  const int lane = threadIdx.x & 31, K = 1 << log2k;
  const int lw = log2k == 0 ? 3 : (log2k == 3 ? 1 : 2), lh = 5 - log2k - lw;  // log2 of the pixel tile's sides
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int tiles_x = (b.W + (1 << lw) - 1) >> lw, tiles_y = (b.H + (1 << lh) - 1) >> lh;
  const long long tpf = (long long)tiles_x * tiles_y;
  const long long frame = warp / tpf;
  if (frame >= (long long)b.n_times * b.n_views) return;
  const int tt = (int)(warp - frame * tpf), ray_id = lane >> log2k, off = lane & (K - 1);
  const int px = ((tt % tiles_x) << lw) + (ray_id & ((1 << lw) - 1)), py = ((tt / tiles_x) << lh) + (ray_id >> lw);
  const int view = (int)(frame % b.n_views), ti = (int)(frame / b.n_views);
  const bool inside = px < b.W && py < b.H;

  const Latent lat = make_latent(net, b.times[ti]);
  // ray geometry in double-float arithmetic (srn_df.cuh): direction, box
  // entry / exit and sample positions carry ~44 bits, so the network sees
  // positions rounded once
  df::Ray ray;
  float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
  unsigned int ns = 0;
  bool live = inside && df::ray_setup(b.cams[view], b.W, b.H, px, py, ray);  // the same in a ray's K lanes
  const float3 d = live ? make_float3(ray.d[0].h, ray.d[1].h, ray.d[2].h) : make_float3(0.f, 0.f, 0.f);
  float3 p = make_float3(0.5f, 0.5f, 0.5f), pl = make_float3(0.f, 0.f, 0.f);
  for (int k = off;; k += K) {
    float len = 0.f;
    const bool have = live && df::segment(ray, k, b.step, len, p, pl);
    if (!__any_sync(0xffffffffu, have)) break;
    // lanes without a sample evaluate their last position (or the centre); nothing reads the result
    float3 g = make_float3(0.f, 0.f, 0.f);
    const float rho = sample_field<C, SH, WIDE>(ctx, mine, lat, p, pl, b.fd_h, g);
    __syncwarp();
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (have) {
      c = tf_eval(tf, rho);
      c.w = -expm1f(-c.w * tf.opacity_scale * len);
      if (SH != SRN_SHADE_NONE) shade(c, g, d);
    }
    for (int i = 0; i < K; ++i) {
      const int src = (lane & ~(K - 1)) + i;
      float4 v = c;
      bool any = have;
      if (K > 1) {
        v.x = __shfl_sync(0xffffffffu, c.x, src);
        v.y = __shfl_sync(0xffffffffu, c.y, src);
        v.z = __shfl_sync(0xffffffffu, c.z, src);
        v.w = __shfl_sync(0xffffffffu, c.w, src);
        any = __shfl_sync(0xffffffffu, (int)have, src) != 0;
      }
      live = live && any;  // the ray's last segment is behind it
      if (live) {
        ns += off == 0;
        const float w = (1.0f - A) * v.w;
        C0 = fmaf(w, v.x, C0);
        C1 = fmaf(w, v.y, C1);
        C2 = fmaf(w, v.z, C2);
        A += w;
        live = !(A >= b.et);
      }
    }
  }
  if (inside && off == 0) {
    size_t idx = ((size_t)frame * b.H + py) * b.W + px;
    reinterpret_cast<float4*>(b.out)[idx] = make_float4(C0, C1, C2, A);
  }
  add_samples(b.samples, ns);
}

// Point evaluation: mode 0 writes out[n][D]; mode 1 writes rho[n] and the
// adjoint gradient grad[n][3] (when grad is not null); mode 2 writes the
// input vector-Jacobian product grad[n][3] = sum_d dout[n][d] d out_d / d p.
template <int C, int MODE, bool WIDE>
__global__ void __launch_bounds__(32 * tile32::max_warps(C), 1)
    eval_fp32_kernel(const NetDev net, const float* __restrict__ pts, int n, float time, float* __restrict__ out,
                     float* __restrict__ grad, const float* __restrict__ dout, const tile32::Net t, int rows) {
  constexpr int S = tile32::kPts;
  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  tile32::load_net<C>(sm, t, net);
  const tile32::Ctx ctx{sm, &t, net.act, tile32::nerf_rows(sm + t.oF, t.m)};
  float* mine = sm + t.total + (threadIdx.x >> 5) * rows * S;
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const Latent lat = make_latent(net, time);
  const float3 zero = make_float3(0.f, 0.f, 0.f);
  for (long long tile = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); tile * 32 < n;
       tile += (long long)gridDim.x * wpb) {
    const long long j = tile * 32 + lane;
    const bool valid = j < n;
    const float3 p = valid ? clamp_p(make_float3(pts[3 * j], pts[3 * j + 1], pts[3 * j + 2]))
                           : make_float3(0.5f, 0.5f, 0.5f);
    if constexpr (MODE == 0) {
      tile32::forward<C, false, WIDE>(ctx, mine, mine, lat, p, zero, nullptr);
      for (int d = 0; d < t.D; ++d) {
        const float v = tile32::last_layer<C, S>(mine, sm, t, d);
        if (valid) out[(size_t)j * t.D + d] = v;
      }
    } else {
      float* x = mine + t.rows * S;
      float* seeds = x + C * S;
      tile32::Acc<C> df[kMaxL - 1], a;
      tile32::forward<C, true, WIDE>(ctx, mine, x, lat, p, zero, df);
      if constexpr (MODE == 1) {
        const float v = tile32::last_layer<C, S>(x, sm, t, 0);
        if (valid) out[j] = v;
        if (grad) tile32::seed<C>(a, sm, t, nullptr);
      } else {
        for (int d = 0; d < t.D; ++d) seeds[d * S + lane] = valid ? dout[(size_t)j * t.D + d] : 0.f;
        __syncwarp();
        tile32::seed<C>(a, sm, t, seeds);
      }
      if (grad) {
        const float3 g = tile32::input_gradient<C, WIDE>(ctx, mine, x, lat, p, a, df);
        if (valid) {
          grad[3 * j] = g.x;
          grad[3 * j + 1] = g.y;
          grad[3 * j + 2] = g.z;
        }
      }
    }
    __syncwarp();
  }
}

template <int C, int SH>
cudaError_t launch_render_t(const NetDev& net, const BatchDev& b, cudaStream_t s) {
  const tile32::Net t = tile32::make_net(net, SH == SRN_SHADE_ADJOINT);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // samples of a ray per warp: double while that leaves at most the warps the
  // SMs hold at once (16 each; beyond, the dropped samples only cost)
  int log2k = 0;
  long long tiles = 0;
  for (;; ++log2k) {
    const int lw = log2k == 0 ? 3 : (log2k == 3 ? 1 : 2), lh = 5 - log2k - lw;
    tiles = (long long)((b.W + (1 << lw) - 1) >> lw) * ((b.H + (1 << lh) - 1) >> lh) * b.n_views * b.n_times;
    if (log2k == 3 || 2 * tiles > 16ll * sms) break;
  }
  const int rows = tile_rows(t, C, SH == SRN_SHADE_ADJOINT, false);
  const int warps = tile32::warps_for(t, C, rows, 0, sms, (int)sizeof(TFDev));
  const size_t smem = sizeof(float) * ((size_t)t.total + (size_t)warps * rows * tile32::kPts);
  auto k = t.wide ? render_fp32_kernel<C, SH, true> : render_fp32_kernel<C, SH, false>;
  e = tile32::allow_dynamic(k, (int)sizeof(TFDev));
  if (e != cudaSuccess) return e;
  const long long blocks = (tiles + warps - 1) / warps;
  k<<<(unsigned)blocks, 32 * warps, smem, s>>>(net, b, t, rows, log2k);
  return cudaGetLastError();
}

template <int C, int MODE>
cudaError_t launch_eval_t(const NetDev& net, const float* pts, int n, float time, float* out, float* grad,
                          const float* dout, cudaStream_t s) {
  const tile32::Net t = tile32::make_net(net, MODE != 0);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const long long tiles = ((long long)n + 31) / 32;
  const int rows = tile_rows(t, C, MODE != 0, MODE == 2);
  int warps = tile32::warps_for(t, C, rows, tiles, sms);
  // A gradient gathers each point's corners twice; from 32 channels on the
  // second time finds them in an L1 that fewer tiles leave larger (300,000
  // points, two layers: 32 channels 295 -> 260 us, 64 channels 504 -> 389).
  // Not where that would take a second wave for a few tiles.
  if (MODE != 0 && t.F >= 32 && warps > 8 && tiles >= 16ll * sms) warps = 8;
  const size_t smem = sizeof(float) * ((size_t)t.total + (size_t)warps * rows * tile32::kPts);
  auto k = t.wide ? eval_fp32_kernel<C, MODE, true> : eval_fp32_kernel<C, MODE, false>;
  e = tile32::allow_dynamic(k);
  if (e != cudaSuccess) return e;
  // CTAs stage the parameters once and walk the tiles: one per SM, by which warps were counted
  const long long blocks = (tiles + warps - 1) / warps;
  k<<<(unsigned)(blocks < sms ? blocks : sms), 32 * warps, smem, s>>>(net, pts, n, time, out, grad, dout, t, rows);
  return cudaGetLastError();
}

// Explicit instantiation of one width's render (all shading modes) or point
// evaluation (both modes).
#define SRN_FP32_RENDER(C, SH)                                                                  \
  template cudaError_t launch_render_t<C, SH>(const NetDev&, const BatchDev&, cudaStream_t);
#define SRN_FP32_EVAL(C, MODE)                                                                  \
  template cudaError_t launch_eval_t<C, MODE>(const NetDev&, const float*, int, float, float*, float*, \
                                              const float*, cudaStream_t);

}  // namespace fp32
}  // namespace srn
