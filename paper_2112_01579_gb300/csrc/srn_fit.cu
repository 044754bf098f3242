// World-space fit (Section 5 training setup: uniformly drawn positions, L1
// loss against the trilinear density of the volume, Adam) and the parameter
// backward of the network, FP32 throughout.
//
// Pipeline of one step (all on the caller's stream, no host sync):
//   1. point kernel: Philox4x32-10 sample (counter = point, step; uniform or
//      the Section 6.2 error-proportional distribution), ground
//      truth, forward with stashed pre-activations, loss, backward through
//      the layers.  Weight gradients: each CTA stages delta_i and v_i of its
//      128 points in shared memory and accumulates dW_i = sum_p delta v^T for
//      the entries it owns (fixed order); one partial row per CTA.  Latent
//      adjoints dz and the cell of every point go to scratch.
//      (Two-layer width-32 density networks take the tensor-core point
//      kernel of srn_fit_mma.cu instead; other networks of up to four layers
//      and 48 inputs the tiled kernel, fit_tile_kernel.)
//   2. stable radix sort of (cell, point) pairs: up to 512 cells one 9-bit
//      pass; up to 2^18 cells a pass over the leading eight bits, then each
//      leading digit by itself (a block, or several where points crowd);
//      else 8-bit digits from the lowest.  A pass is
//      per-block per-warp digit counts, a scan per digit over the blocks and a
//      stable scatter (which adds the digits' prefix and, for one pass, writes
//      the cell offsets).
//   3. latent-grid gradient without floating-point atomics: sums of
//      w_corner(p) * dz per (cell, corner), a block per dense cell or a warp
//      per sparse one, then each vertex adds its <= 8 partials.  Fixed orders
//      and butterflies throughout, so the gradient is bit-reproducible.
//   4. fixed-order reduction of the CTA partials (weights, biases, loss), in
//      the same launch as the vertex gather.
//   5. Adam over grid, weights and biases (skipped if anything is not
//      finite), refreshing the FP16 copies.
#include <limits.h>

#include <algorithm>
#include <utility>

#include "srn_fit.h"
#include "srn_net32.cuh"
#include "srn_sample.cuh"
#include "srn_tile32.cuh"

namespace srn {
namespace {

using namespace net32;

constexpr int kFitThreads = 128;
constexpr int kSortThreads = 256;
// Keys per sort block: 8 warps x 4 or 8 rounds x 32.  Blocks of 1024 fill the
// SMs from 2^18 points; larger sets and the static area (whose histogram
// bounds its batch) take 2048.
constexpr int kSortItems = 2048, kSortItemsSmall = 1024;

__device__ __forceinline__ float sgnf(float x) { return x > 0.f ? 1.f : (x < 0.f ? -1.f : 0.f); }

struct PointArgs {
  int n;
  int mode;  // 0: fit (sample, loss); 1: backward of given points / adjoints
  const float* pts_in;
  const float* dout_in;
  unsigned long long seed;
  int step;
  float time;
  VolDev vol;
  float gw, gs;
  const unsigned long long* cdf;  // Section 6.2 adaptive distribution (null: uniform)
  int cdf_res;
  const int* step_ptr;            // step index in device memory (graph replay), else `step`
  float* pts;   // scratch out
  float* dz;
  unsigned int* key;
  unsigned int* idx;
  float* part;
  int n_entries;
  int dstride;  // stride of the staged input rows
  int stall_test;  // timeout-path test (tensor-core point kernel only)
};

// Adds the contribution of the CTA's points to the gradient entries of one
// layer: W block (dout x din at woff) and bias block (dout at boff).  Each
// sum over the CTA's points runs as four interleaved partial sums (points
// p = 4q + r) combined at the end, a fixed order.
__device__ __forceinline__ void accumulate_layer(float* sacc, const float* sdelta, int dstr_d, const float* svin,
                                                 int dstr_v, int dout, int din, int woff, int boff) {
  const int tid = threadIdx.x;
  for (int e = tid; e < dout * din; e += kFitThreads) {
    const int o = e / din, j = e - o * din;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
    for (int p = 0; p < kFitThreads; p += 4) {
      s0 = fmaf(sdelta[p * dstr_d + o], svin[p * dstr_v + j], s0);
      s1 = fmaf(sdelta[(p + 1) * dstr_d + o], svin[(p + 1) * dstr_v + j], s1);
      s2 = fmaf(sdelta[(p + 2) * dstr_d + o], svin[(p + 2) * dstr_v + j], s2);
      s3 = fmaf(sdelta[(p + 3) * dstr_d + o], svin[(p + 3) * dstr_v + j], s3);
    }
    sacc[woff + e] += (s0 + s1) + (s2 + s3);
  }
  for (int e = tid; e < dout; e += kFitThreads) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
    for (int p = 0; p < kFitThreads; p += 4) {
      s0 += sdelta[p * dstr_d + e];
      s1 += sdelta[(p + 1) * dstr_d + e];
      s2 += sdelta[(p + 2) * dstr_d + e];
      s3 += sdelta[(p + 3) * dstr_d + e];
    }
    sacc[boff + e] += (s0 + s1) + (s2 + s3);
  }
}

template <int C>
__global__ void __launch_bounds__(kFitThreads, 4) fit_point_kernel(const NetDev net, const PointArgs a, const Layout L) {
  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  const int dstr_d = C + 1, dstr_v = a.dstride;
  float* sdelta = sm + L.total;
  float* svin = sdelta + kFitThreads * dstr_d;
  float* sacc = svin + kFitThreads * dstr_v;
  float* sred = sacc + ((a.n_entries + 3) & ~3);
  load_net<C>(sm, L, net);
  const int tid = threadIdx.x;
  const int step = a.step_ptr ? *a.step_ptr : a.step;
  for (int e = tid; e < a.n_entries; e += kFitThreads) sacc[e] = 0.f;

  // packed offsets of each layer's weights / biases in [W | b]
  const int d0 = L.d0, l = L.l, D = L.D;
  const int nW = C * d0 + (l - 2) * C * C + D * C;
  const Latent lat = make_latent(net, a.time);
  const float inv_n = 1.0f / (float)a.n;
  float loss_acc = 0.f;
  const int nchunks = (a.n + kFitThreads - 1) / kFitThreads;

  for (int chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    const int j = chunk * kFitThreads + tid;
    const bool valid = j < a.n;
    float3 p = make_float3(0.5f, 0.5f, 0.5f);
    float out[4] = {0.f, 0.f, 0.f, 0.f}, dout[4] = {0.f, 0.f, 0.f, 0.f};
    float hs[kMaxL][C];
    if (valid) {
      if (a.mode == 0) p = sample::fit_point(a.cdf, a.cdf_res, a.seed, step, j, a.n);
      else p = clamp_p(make_float3(a.pts_in[3 * j], a.pts_in[3 * j + 1], a.pts_in[3 * j + 2]));
      forward<C>(sm, L, net.act, lat, p, out, hs);
      if (a.mode == 0) {
        const float r = out[0] - vol_sample(a.vol, p);
        loss_acc += fabsf(r);
        dout[0] = sgnf(r) * inv_n;
        if (D == 4) {
          const float hh[3] = {1.0f / (float)(a.vol.nx - 1), 1.0f / (float)(a.vol.ny - 1),
                               1.0f / (float)(a.vol.nz - 1)};
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            float3 pp = p, pm = p;
            if (ax == 0) { pp.x = clamp01f(p.x + hh[0]); pm.x = clamp01f(p.x - hh[0]); }
            if (ax == 1) { pp.y = clamp01f(p.y + hh[1]); pm.y = clamp01f(p.y - hh[1]); }
            if (ax == 2) { pp.z = clamp01f(p.z + hh[2]); pm.z = clamp01f(p.z - hh[2]); }
            const float g = (vol_sample(a.vol, pp) - vol_sample(a.vol, pm)) / (2.0f * hh[ax]);
            const float ra = out[1 + ax] - a.gs * g;
            loss_acc += a.gw * fabsf(ra);
            dout[1 + ax] = a.gw * sgnf(ra) * inv_n;
          }
        }
      } else {
        for (int dd = 0; dd < D; ++dd) dout[dd] = a.dout_in[(size_t)j * D + dd];
      }
    }
    // ---- last layer (C -> D): delta = dout, input = act(h_{l-2}); the
    // activation and its derivative come from one sin/cos evaluation
    float dact[C];
#pragma unroll
    for (int o = 0; o < C; ++o) {
      float av = 0.f, dv = 0.f;
      if (valid) act_and_df(net.act, hs[l - 2][o], av, dv);
      svin[tid * dstr_v + o] = av;
      dact[o] = dv;
    }
#pragma unroll
    for (int dd = 0; dd < 4; ++dd)
      if (dd < D) sdelta[tid * dstr_d + dd] = dout[dd];
    __syncthreads();
    accumulate_layer(sacc, sdelta, dstr_d, svin, dstr_v, D, C, nW - D * C, nW + (l - 1) * C);
    __syncthreads();
    float delta[C];
#pragma unroll
    for (int jj = 0; jj < C; ++jj) {
      float g = 0.f;
      for (int dd = 0; dd < D; ++dd) g = fmaf(sm[L.oWl + dd * C + jj], dout[dd], g);
      delta[jj] = g * dact[jj];
    }
    // ---- hidden layers i = l-2 .. 1 (C -> C)
    for (int i = l - 2; i >= 1; --i) {
#pragma unroll
      for (int o = 0; o < C; ++o) {
        float av = 0.f, dv = 0.f;
        if (valid) act_and_df(net.act, hs[i - 1][o], av, dv);
        sdelta[tid * dstr_d + o] = delta[o];
        svin[tid * dstr_v + o] = av;
        dact[o] = dv;
      }
      __syncthreads();
      accumulate_layer(sacc, sdelta, dstr_d, svin, dstr_v, C, C, C * d0 + (i - 1) * C * C, nW + i * C);
      __syncthreads();
      const float* Wrm = sm + L.oHid + (i - 1) * L.hidStride + C * C + C;
      float g[C];
#pragma unroll
      for (int jj = 0; jj < C; ++jj) g[jj] = 0.f;
#pragma unroll
      for (int o = 0; o < C; ++o) axpy<C>(g, Wrm + o * C, delta[o]);
#pragma unroll
      for (int jj = 0; jj < C; ++jj) delta[jj] = g[jj] * dact[jj];
    }
    // ---- layer 0 (d0 -> C): input [p, sin(Fp), cos(Fp), z]
#pragma unroll
    for (int o = 0; o < C; ++o) sdelta[tid * dstr_d + o] = delta[o];
    {
      float* v = svin + tid * dstr_v;
      v[0] = p.x; v[1] = p.y; v[2] = p.z;
      const float* Fm = sm + L.oF;
      for (int k = 0; k < L.m; ++k) {
        const float e = Fm[3 * k] * p.x + Fm[3 * k + 1] * p.y + Fm[3 * k + 2] * p.z;
        float s, c;
        sincosf(e, &s, &c);
        v[3 + k] = s;
        v[3 + L.m + k] = c;
      }
      const Cell cell = make_cell(lat, p);
      for (int f = 0; f < L.F; f += 4) {
        const float4 z = latent4(lat, cell, f);
        v[3 + 2 * L.m + f] = z.x;
        v[3 + 2 * L.m + f + 1] = z.y;
        v[3 + 2 * L.m + f + 2] = z.z;
        v[3 + 2 * L.m + f + 3] = z.w;
      }
      if (L.ti) v[3 + 2 * L.m + L.F] = lat.tin;
      if (!valid)
        for (int q = 0; q < d0; ++q) v[q] = 0.f;
    }
    __syncthreads();
    accumulate_layer(sacc, sdelta, dstr_d, svin, dstr_v, C, d0, 0, nW);
    __syncthreads();
    if (valid) {
      const float* W0T = sm + L.oW0T;
      float4* dzj = reinterpret_cast<float4*>(a.dz + (size_t)j * L.F);
      for (int f = 0; f < L.F; f += 4) {
        const float* r = W0T + (3 + 2 * L.m + f) * C;
        dzj[f >> 2] = make_float4(dotrow<C>(r, delta), dotrow<C>(r + C, delta), dotrow<C>(r + 2 * C, delta),
                                  dotrow<C>(r + 3 * C, delta));
      }
      a.pts[3 * j] = p.x;
      a.pts[3 * j + 1] = p.y;
      a.pts[3 * j + 2] = p.z;
      int ix, iy, iz;
      float fx, fy, fz;
      cell_coord(p.x, lat.R, ix, fx);
      cell_coord(p.y, lat.R, iy, fy);
      cell_coord(p.z, lat.R, iz, fz);
      a.key[j] = (unsigned)((iz * (lat.R - 1) + iy) * (lat.R - 1) + ix);
      a.idx[j] = (unsigned)j;
    }
  }
  // ---- per-CTA partials: gradient entries, then the loss sum (fixed tree)
  float* row = a.part + (size_t)blockIdx.x * (a.n_entries + 1);
  for (int e = tid; e < a.n_entries; e += kFitThreads) row[e] = sacc[e];
  sred[tid] = loss_acc;
  __syncthreads();
  for (int w = kFitThreads / 2; w > 0; w >>= 1) {
    if (tid < w) sred[tid] += sred[tid + w];
    __syncthreads();
  }
  if (tid == 0) row[a.n_entries] = sred[0];
}

// ---------------------------------------------------------------- tiled point kernel
// The point kernel for networks of two to four layers with at most 48 inputs
// (every shape of the plain and main workloads): the same step as
// fit_point_kernel, each warp running its 32 points as a tile (srn_tile32.cuh).
//
// What bounds it: FP32 FMAs (forward, backward and weight gradient, about
// 3 x sum d_in d_out per point) and the shared-memory loads that feed them.
// The weight gradient dW_i = sum_p delta v^T takes a 4 x 3 (layer 0) or 4 x 2
// block of entries per thread over the CTA's 128 points, four points per
// 16-byte load: 7 loads for 48 FMAs, where one entry at a time takes two
// loads per FMA.  A thread keeps its entries in registers over all its
// chunks; sums of 32 points are formed first and then added, so the rounding
// error does not grow with the number of points a CTA takes.  The vectors of
// every layer stay in shared memory from the forward to the backward (a
// layer's adjoint rows take the place of its activations once the gradient
// that needs them is done), the activation derivatives in registers, so
// neither sines nor Fourier features are evaluated twice.  Fit step of the
// main configuration (32^3 x 16, four layers) at 2^18 points: 876 -> 305 us
// (with the sort and gather below); 65,537 points of the same network through
// autograd 434 -> 250 us.
constexpr int kTileStride = 36;  // floats per adjoint row: eight rows' 16-byte loads hit distinct banks
constexpr int kTileMaxIn = 48;   // inputs of layer 0: 16 threads x 3 entries
// Points with a residual below this are decided by the accurate functions.  It
// holds what inline and library sines move an output by on trained networks of
// the workloads' shapes (4e-7 at most of 2^18 points, densities and gradient
// outputs) and at Xavier's weights (1e-6).  With larger weights the two differ
// by more (twice Xavier's, four layers: 1e-5), and both are as far from 64 bits
// (1.3e-5 and 1.1e-5 at most, 1.8e-6 rms each): which sign is right is then not
// decided by either, and a wider band would only cost.  A converged fit
// (residuals around 0.01) has a few hundred points of 2^18 in it.
constexpr float kSignBand = 4.0e-6f;

// acc[i][j] += sum over the CTA's points of d[o_i][p] v[r_j][p], o_i = tid % 8
// + 8 i, r_j = tid / 8 + 16 j (rows past `rows` repeat the last one; their
// sums are never stored).  d and v are the first warp's rows, `wstride`
// floats apart per warp.
// VS: floats per row of v (rows a quarter-warp reads together are one row, so
// v needs no padding).
template <int NJ, int VS>
__device__ __forceinline__ void outer_sum(float (&acc)[4][NJ], const float* d, const float* v, int wstride, int rows) {
  const int og = threadIdx.x & 7, jg = threadIdx.x >> 3;
  int vr[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) vr[j] = min(jg + 16 * j, rows - 1) * VS;
#pragma unroll 1
  for (int w = 0; w < kFitThreads / 32; ++w) {
    const float* dw = d + w * wstride + og * kTileStride;
    const float* vw = v + w * wstride;
    float2 s[4][NJ];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) s[i][j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < 32; p += 4) {
      float4 dd[4], vv[NJ];
#pragma unroll
      for (int i = 0; i < 4; ++i) dd[i] = *reinterpret_cast<const float4*>(dw + 8 * i * kTileStride + p);
#pragma unroll
      for (int j = 0; j < NJ; ++j) vv[j] = *reinterpret_cast<const float4*>(vw + vr[j] + p);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          s[i][j] = __ffma2_rn(make_float2(dd[i].x, dd[i].y), make_float2(vv[j].x, vv[j].y), s[i][j]);
          s[i][j] = __ffma2_rn(make_float2(dd[i].z, dd[i].w), make_float2(vv[j].z, vv[j].w), s[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] += s[i][j].x + s[i][j].y;
  }
}

// Sum of one row's 32 values, and of two rows' products, in four interleaved sums.
__device__ __forceinline__ float row_sum(const float* r) {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int p = 0; p < 32; p += 4) {
    const float4 x = *reinterpret_cast<const float4*>(r + p);
    s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
  }
  return (s.x + s.y) + (s.z + s.w);
}
__device__ __forceinline__ float row_dot(const float* r, const float* w) {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int p = 0; p < 32; p += 4) {
    const float4 x = *reinterpret_cast<const float4*>(r + p), y = *reinterpret_cast<const float4*>(w + p);
    s.x = fmaf(x.x, y.x, s.x); s.y = fmaf(x.y, y.y, s.y); s.z = fmaf(x.z, y.z, s.z); s.w = fmaf(x.w, y.w, s.w);
  }
  return (s.x + s.y) + (s.z + s.w);
}

// dz[j][f] for the lane's four points and F / 4 channels from the adjoint rows d.
template <int F>
__device__ __forceinline__ void store_dz(const float* d, const float* Wz, float* dz, int j0, int n) {
  const int pg = tile32::point_group(), og = tile32::out_group();
  float2 acc[2][F / 4];
  tile32::back<32, kTileStride, F / 4, 4>(acc, d, Wz, [&](int f) { return og * (F / 4) + f; });
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int j = j0 + 4 * pg + i;
    if (j < n) {
      float* out = dz + (size_t)j * F + og * (F / 4);
#pragma unroll
      for (int f = 0; f < F / 4; ++f) out[f] = (i & 1) ? acc[i >> 1][f].y : acc[i >> 1][f].x;
    }
  }
}

template <int NL, bool SNAKE>
__global__ void __launch_bounds__(kFitThreads, 2) fit_tile_kernel(const __grid_constant__ NetDev net,
                                                                  const __grid_constant__ PointArgs a,
                                                                  const __grid_constant__ tile32::Net t, int wfloats) {
  constexpr int C = 32, S = kTileStride, NH = NL - 1;  // NH activations per point
  constexpr int VS = 32;  // floats per input row
  // four layers: the first activation's derivatives wait in shared memory (a
  // lane's own 32 values), which leaves registers for loads in flight
  constexpr bool PARK = NL == 4;
  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  tile32::load_net<C>(sm, t, net);
  const bool nerf = tile32::nerf_rows(sm + t.oF, t.m);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* base0 = sm + t.total;                // first warp's rows
  float* v0 = base0 + warp * wfloats;         // layer inputs, then NH blocks of activation rows, then dout
  float* act0 = v0 + t.d0 * VS;
  float* sdout = act0 + NH * C * S;
  float4* parked = reinterpret_cast<float4*>(sdout + 4 * S) + lane;
  const int pg = tile32::point_group(), og = tile32::out_group();
  const int step = a.step_ptr ? *a.step_ptr : a.step;
  const Latent lat = make_latent(net, a.time);
  const float inv_n = 1.0f / (float)a.n;
  const int D = t.D, nchunks = (a.n + kFitThreads - 1) / kFitThreads;

  float g0[4][3], gh[NL > 2 ? NL - 2 : 1][4][2], gb[NH], gl[4], gbl = 0.f, loss_acc = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    gl[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) g0[i][j] = 0.f;
#pragma unroll
    for (int h = 0; h < NL - 2; ++h) gh[h][i][0] = gh[h][i][1] = 0.f;
  }
#pragma unroll
  for (int h = 0; h < NH; ++h) gb[h] = 0.f;

  for (int chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    const int j = chunk * kFitThreads + tid;
    const bool valid = j < a.n;
    float3 p = make_float3(0.5f, 0.5f, 0.5f);
    if (valid) {
      if (a.mode == 0) p = sample::fit_point(a.cdf, a.cdf_res, a.seed, step, j, a.n);
      else p = clamp_p(make_float3(a.pts_in[3 * j], a.pts_in[3 * j + 1], a.pts_in[3 * j + 2]));
    }
    // ---- forward: activations to shared memory, their derivatives kept
    if (valid) {
      tile32::put_inputs<VS>(v0, sm, t, lat, nerf, p);
    } else {
      for (int k = 0; k < t.d0; ++k) v0[k * VS + lane] = 0.f;
    }
    __syncwarp();
    tile32::Acc<C> x, df[NH];
    tile32::set_bias<C>(x, sm + t.ob0);
    tile32::layer<C, VS>(x, v0, sm + t.oW0, t.d0);
    tile32::activate_call<C, SNAKE>(x, df[0]);
    if (PARK) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < C / 8; q += 2)
          parked[(2 * i + q / 2) * 32] =
              make_float4(df[0].v[i][q].x, df[0].v[i][q].y, df[0].v[i][q + 1].x, df[0].v[i][q + 1].y);
    }
    tile32::put<C, S>(x, act0);
    __syncwarp();
#pragma unroll
    for (int h = 1; h < NH; ++h) {
      const float* W = sm + t.oHid + (h - 1) * t.hidStride;
      tile32::set_bias<C>(x, W + C * C);
      tile32::layer<C, S>(x, act0 + (h - 1) * C * S, W, C);
      tile32::activate_call<C, SNAKE>(x, df[h]);
      tile32::put<C, S>(x, act0 + h * C * S);
      __syncwarp();
    }
    const float* alast = act0 + (NH - 1) * C * S;
    float dout[4] = {0.f, 0.f, 0.f, 0.f};
    if (a.mode == 0) {
      float out[4], want[4] = {0.f, 0.f, 0.f, 0.f};
      if (valid) {
        want[0] = vol_sample(a.vol, p);
        if (D == 4) {
          const float hh[3] = {1.0f / (float)(a.vol.nx - 1), 1.0f / (float)(a.vol.ny - 1),
                               1.0f / (float)(a.vol.nz - 1)};
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            float3 pp = p, pm = p;
            if (ax == 0) { pp.x = clamp01f(p.x + hh[0]); pm.x = clamp01f(p.x - hh[0]); }
            if (ax == 1) { pp.y = clamp01f(p.y + hh[1]); pm.y = clamp01f(p.y - hh[1]); }
            if (ax == 2) { pp.z = clamp01f(p.z + hh[2]); pm.z = clamp01f(p.z - hh[2]); }
            want[1 + ax] = a.gs * ((vol_sample(a.vol, pp) - vol_sample(a.vol, pm)) / (2.0f * hh[ax]));
          }
        }
      }
#pragma unroll
      for (int dd = 0; dd < 4; ++dd) out[dd] = dd < D ? tile32::last_layer<C, S>(alast, sm, t, dd) : 0.f;
      // the sign of a residual decides a point's whole gradient: a point with
      // one within kSignBand of zero takes its outputs from the accurate
      // functions
      bool close = false;
#pragma unroll
      for (int dd = 0; dd < 4; ++dd) close |= valid && dd < D && fabsf(out[dd] - want[dd]) < kSignBand;
      for (unsigned int m = __ballot_sync(0xffffffffu, close); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const float3 q = make_float3(__shfl_sync(0xffffffffu, p.x, src), __shfl_sync(0xffffffffu, p.y, src),
                                     __shfl_sync(0xffffffffu, p.z, src));
        const float4 o = tile32::accurate_point(sm, t, net.act, lat, q, sdout);
        if (lane == src) out[0] = o.x, out[1] = o.y, out[2] = o.z, out[3] = o.w;
      }
      if (valid) {
        const float r = out[0] - want[0];
        loss_acc += fabsf(r);
        dout[0] = sgnf(r) * inv_n;
        if (D == 4) {
#pragma unroll
          for (int dd = 1; dd < 4; ++dd) {
            const float ra = out[dd] - want[dd];
            loss_acc += a.gw * fabsf(ra);
            dout[dd] = a.gw * sgnf(ra) * inv_n;
          }
        }
      }
    } else if (valid) {
#pragma unroll
      for (int dd = 0; dd < 4; ++dd)
        if (dd < D) dout[dd] = a.dout_in[(size_t)j * D + dd];
    }
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) sdout[dd * S + lane] = dout[dd];
    __syncwarp();
    // ---- last layer: gradients over the warp's own points (lane = input), then delta
#pragma unroll
    for (int dd = 0; dd < 4; ++dd)
      if (dd < D) gl[dd] += row_dot(alast + lane * S, sdout + dd * S);
    if (lane < D) gbl += row_sum(sdout + lane * S);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < C / 8; ++q) x.v[i][q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) {
      if (dd < D) {
        const float4 dv = *reinterpret_cast<const float4*>(sdout + dd * S + 4 * pg);
        const float ds[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
        for (int q = 0; q < C / 8; ++q) {
          const float2 w = *reinterpret_cast<const float2*>(sm + t.oWl + dd * C + og * (C / 4) + 2 * q);
#pragma unroll
          for (int i = 0; i < 4; ++i) x.v[i][q] = __ffma2_rn(w, make_float2(ds[i], ds[i]), x.v[i][q]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < C / 8; ++q) {
        x.v[i][q].x *= df[NH - 1].v[i][q].x;
        x.v[i][q].y *= df[NH - 1].v[i][q].y;
      }
    __syncwarp();  // the last activations are read
    tile32::put<C, S>(x, act0 + (NH - 1) * C * S);
    __syncthreads();
    // ---- hidden layers: adjoint rows of layer h in block h, inputs in block h - 1
#pragma unroll
    for (int h = NH - 1; h >= 1; --h) {
      const float* dh = act0 + h * C * S;
      outer_sum<2, S>(gh[h - 1], base0 + t.d0 * VS + h * C * S, base0 + t.d0 * VS + (h - 1) * C * S, wfloats, C);
      gb[h] += row_sum(dh + lane * S);
      float2 g[2][C / 4];
      tile32::back<C, S, C / 4>(g, dh, sm + t.oHid + (h - 1) * t.hidStride,
                                [&](int q) { return og * (C / 4) + q; });
      if (PARK && h == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < C / 8; q += 2) {
            const float4 v = parked[(2 * i + q / 2) * 32];
            df[0].v[i][q] = make_float2(v.x, v.y);
            df[0].v[i][q + 1] = make_float2(v.z, v.w);
          }
      }
      __syncthreads();  // block h - 1's activations are read
      float* dn = act0 + (h - 1) * C * S + og * (C / 4) * S + 4 * pg;
#pragma unroll
      for (int q = 0; q < C / 4; ++q) {
        auto dfv = [&](int i) { return (q & 1) ? df[h - 1].v[i][q / 2].y : df[h - 1].v[i][q / 2].x; };
        *reinterpret_cast<float4*>(dn + q * S) =
            make_float4(g[0][q].x * dfv(0), g[0][q].y * dfv(1), g[1][q].x * dfv(2), g[1][q].y * dfv(3));
      }
      __syncthreads();
    }
    // ---- layer 0, the latent adjoint and the point's cell
    outer_sum<3, VS>(g0, base0 + t.d0 * VS, base0, wfloats, t.d0);
    gb[0] += row_sum(act0 + lane * S);
    {
      const float* Wz = sm + t.oW0 + (3 + 2 * t.m) * C;
      const int j0 = chunk * kFitThreads + warp * 32;
      switch (t.F) {
        case 4: store_dz<4>(act0, Wz, a.dz, j0, a.n); break;
        case 8: store_dz<8>(act0, Wz, a.dz, j0, a.n); break;
        case 16: store_dz<16>(act0, Wz, a.dz, j0, a.n); break;
        default: store_dz<32>(act0, Wz, a.dz, j0, a.n);
      }
    }
    if (valid) {
      a.pts[3 * j] = p.x;
      a.pts[3 * j + 1] = p.y;
      a.pts[3 * j + 2] = p.z;
      int ix, iy, iz;
      float fx, fy, fz;
      cell_coord(p.x, lat.R, ix, fx);
      cell_coord(p.y, lat.R, iy, fy);
      cell_coord(p.z, lat.R, iz, fz);
      a.key[j] = (unsigned)((iz * (lat.R - 1) + iy) * (lat.R - 1) + ix);
      a.idx[j] = (unsigned)j;
    }
    __syncthreads();
  }

  // ---- the CTA's partial row [W | b | loss]
  const int nW = C * t.d0 + (NL - 2) * C * C + D * C;
  float* row = a.part + (size_t)blockIdx.x * (a.n_entries + 1);
  const int o8 = tid & 7, j16 = tid >> 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (j16 + 16 * q < t.d0) row[(o8 + 8 * i) * t.d0 + tile32::input_column(j16 + 16 * q, t.m)] = g0[i][q];
#pragma unroll
    for (int h = 0; h < NL - 2; ++h)
#pragma unroll
      for (int q = 0; q < 2; ++q) row[C * t.d0 + h * C * C + (o8 + 8 * i) * C + j16 + 16 * q] = gh[h][i][q];
  }
  // entries each warp summed over its own points: the four warps in order
  constexpr int kRows = 4 + NH + 2;  // last-layer weights, biases, last bias, loss
  float* ex = base0;
  __syncthreads();
#pragma unroll
  for (int dd = 0; dd < 4; ++dd) ex[(dd * 4 + warp) * 32 + lane] = gl[dd];
#pragma unroll
  for (int h = 0; h < NH; ++h) ex[((4 + h) * 4 + warp) * 32 + lane] = gb[h];
  ex[((4 + NH) * 4 + warp) * 32 + lane] = gbl;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, w);
  ex[((5 + NH) * 4 + warp) * 32 + lane] = loss_acc;
  __syncthreads();
  for (int e = tid; e < kRows * 32; e += kFitThreads) {
    const int r = e >> 5, o = e & 31;
    const float* q = ex + r * 128 + o;
    const float s = ((q[0] + q[32]) + q[64]) + q[96];
    if (r < 4) {
      if (r < D) row[nW - D * C + r * C + o] = s;
    } else if (r < 4 + NH) {
      row[nW + (r - 4) * C + o] = s;
    } else if (r == 4 + NH) {
      if (o < D) row[nW + NH * C + o] = s;
    } else if (o == 0) {
      row[a.n_entries] = s;
    }
  }
}

// One warp's tile in floats (input rows, activation rows, output adjoints,
// four layers: parked derivatives).
int fit_tile_floats(const NetDev& net) {
  return net_d0(net) * 32 + ((net.l - 1) * 32 + 4) * kTileStride + (net.l == 4 ? 32 * 32 : 0);
}
size_t fit_tile_smem(const NetDev& net) {
  return sizeof(float) * ((size_t)tile32::make_net(net).total + (size_t)(kFitThreads / 32) * fit_tile_floats(net));
}
// Up to four layers: their activation derivatives fit a thread's registers
// (32 a layer), and with at most 48 inputs two CTAs' rows fit an SM's shared
// memory (113 KB a CTA).  Deeper or wider-input networks keep
// fit_point_kernel, which stashes in local memory.
bool fit_tile_supported(const NetDev& net) {
  return net.c == 32 && net.l >= 2 && net.l <= 4 && net_d0(net) <= kTileMaxIn && net.F <= 32;
}

template <int NL>
cudaError_t fit_tile_t(const NetDev& net, const PointArgs& pa, int grid, cudaStream_t st) {
  // an instantiation for each activation: one for both, whose out-of-line
  // activation holds the code of both, took 8 us more of a 300 us step
  auto k = net.act == SRN_ACT_SNAKEALT ? fit_tile_kernel<NL, true> : fit_tile_kernel<NL, false>;
  const size_t smem = fit_tile_smem(net);
  cudaError_t e = tile32::allow_dynamic(k);
  if (e != cudaSuccess) return e;
  k<<<grid, kFitThreads, smem, st>>>(net, pa, tile32::make_net(net), fit_tile_floats(net));
  return cudaGetLastError();
}

cudaError_t launch_fit_tile(const NetDev& net, const PointArgs& pa, int grid, cudaStream_t st) {
  if (net.l == 2) return fit_tile_t<2>(net, pa, grid, st);
  return net.l == 3 ? fit_tile_t<3>(net, pa, grid, st) : fit_tile_t<4>(net, pa, grid, st);
}

// ---------------------------------------------------------------- radix sort
// A warp's keys of one sort block (ROUNDS x 32, all loads in flight at once);
// `end`: first index past the keys.
template <int ROUNDS>
__device__ __forceinline__ void load_keys(const unsigned int* __restrict__ keys, int base, int end,
                                          unsigned int (&k)[ROUNDS]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int i = base + r * 32 + lane;
    k[r] = i < end ? keys[i] : 0u;
  }
}

// Digit counts of the warp's keys: equal digits within a round are grouped
// with __match_any_sync.  NB bins.
template <int NB, int ROUNDS>
__device__ __forceinline__ void warp_digit_counts(const unsigned int (&k)[ROUNDS], int base, int end, int shift,
                                                  unsigned int* cnt) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool valid = base + r * 32 + lane < end;
    const unsigned int d = valid ? (k[r] >> shift) & (unsigned)(NB - 1) : 0xFFFFFFFFu;
    const unsigned int peers = __match_any_sync(0xffffffffu, d);
    if (valid && lane == __ffs(peers) - 1) cnt[d] += __popc(peers);
    __syncwarp();
  }
}

// Stable scatter of the warp's keys and values from cnt[d], the position of
// the warp's next key of digit d.
template <int NB, int ROUNDS>
__device__ __forceinline__ void warp_scatter(const unsigned int (&k)[ROUNDS], const unsigned int (&v)[ROUNDS], int base,
                                             int end, int shift, unsigned int* cnt, unsigned int* __restrict__ kout,
                                             unsigned int* __restrict__ vout) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool valid = base + r * 32 + lane < end;
    const unsigned int d = valid ? (k[r] >> shift) & (unsigned)(NB - 1) : 0xFFFFFFFFu;
    const unsigned int peers = __match_any_sync(0xffffffffu, d);
    const unsigned int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid) {
      const unsigned int pos = cnt[d] + rank;
      if (kout) kout[pos] = k[r];
      vout[pos] = v[r];
    }
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) cnt[d] += __popc(peers);
    __syncwarp();
  }
}

// hist[d * nblocks + block] = count of digit d in the block (digit-major, so
// one exclusive scan gives every (digit, block) its output offset).
template <int NB, int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) sort_hist_kernel(const unsigned int* __restrict__ keys, int n,
                                                                 int shift, unsigned int* __restrict__ hist,
                                                                 int nblocks) {
  __shared__ unsigned int cnt[8][NB];
  const int w = threadIdx.x >> 5, base = blockIdx.x * (ROUNDS * kSortThreads) + w * (ROUNDS * 32);
  unsigned int k[ROUNDS];
  load_keys<ROUNDS>(keys, base, n, k);
  for (int i = threadIdx.x; i < 8 * NB; i += kSortThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  warp_digit_counts<NB, ROUNDS>(k, base, n, shift, cnt[w]);
  __syncthreads();
  for (int d = threadIdx.x; d < NB; d += kSortThreads) {
    unsigned int t = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) t += cnt[q][d];
    hist[(size_t)d * nblocks + blockIdx.x] = t;
  }
}

// Exclusive scan of m counts in place, in segments of `seg` values, one block
// per segment: tiles of 8192 values are staged coalesced in shared memory,
// each thread scans 8 consecutive values, and a block-wide scan of the thread
// sums plus a running carry links the tiles.  Segment b starts from
// carry_in[b] (the exclusive scan of the segment sums; 0 when carry_in is
// null).  Integer sums in a fixed order, so deterministic.
constexpr int kScanThreads = 1024, kScanPer = 8, kScanTile = kScanThreads * kScanPer;

// sums[b] = sum of segment b of a.
__global__ void __launch_bounds__(kScanThreads) seg_sum_kernel(const unsigned int* __restrict__ a, int m, int seg,
                                                               unsigned int* __restrict__ sums) {
  __shared__ unsigned int wsum[32];
  const int b0 = blockIdx.x * seg, b1 = min(m, b0 + seg);
  unsigned int t = 0;
  for (int i = b0 + threadIdx.x; i < b1; i += kScanThreads) t += a[i];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    unsigned int w = wsum[threadIdx.x];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) w += __shfl_xor_sync(0xffffffffu, w, off);
    if (threadIdx.x == 0) sums[blockIdx.x] = w;
  }
}

__global__ void __launch_bounds__(kScanThreads) scan_kernel(unsigned int* __restrict__ a, int m, int seg,
                                                            const unsigned int* __restrict__ carry_in) {
  __shared__ unsigned int tile[kScanTile + kScanTile / 32];  // padded: 8-strided reads stay conflict-free
  __shared__ unsigned int part[32];
  __shared__ unsigned int carry_s;
  const int tid = threadIdx.x;
  const int s0 = blockIdx.x * seg, s1 = min(m, s0 + seg);
  if (tid == 0) carry_s = carry_in ? carry_in[blockIdx.x] : 0u;
  for (int base = s0; base < s1; base += kScanTile) {
    for (int i = tid; i < kScanTile; i += kScanThreads) {
      const int g = base + i;
      tile[i + i / 32] = g < s1 ? a[g] : 0u;
    }
    __syncthreads();
    unsigned int v[kScanPer], s = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int i = tid * kScanPer + k;
      v[k] = tile[i + i / 32];
      s += v[k];
    }
    // block-wide inclusive scan of the thread sums: warp shuffles, then the
    // 32 warp totals by warp 0
    const int lane = tid & 31, warp = tid >> 5;
    unsigned int x = s;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= off) x += y;
    }
    if (lane == 31) part[warp] = x;
    __syncthreads();
    if (warp == 0) {
      unsigned int w = part[lane];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += y;
      }
      part[lane] = w;
    }
    __syncthreads();
    const unsigned int incl = (warp > 0 ? part[warp - 1] : 0u) + x;
    unsigned int run = carry_s + incl - s;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
      const int i = tid * kScanPer + k;
      tile[i + i / 32] = run;
      run += v[k];
    }
    __syncthreads();
    for (int i = tid; i < kScanTile; i += kScanThreads) {
      const int g = base + i;
      if (g < s1) a[g] = tile[i + i / 32];
    }
    if (tid == kScanThreads - 1) carry_s += incl;
    __syncthreads();
  }
}

// Exclusive scan of one digit's counts over the sort blocks (one block per
// digit, up to kDigitThreads * kDigitPer sort blocks), in place; the digit's
// total to totals[digit].  The scatter kernel adds the exclusive scan of the
// totals itself, so one launch replaces the segmented scan of the whole
// histogram.  Integer sums in a fixed order.
constexpr int kDigitThreads = 256, kDigitPer = 4;

__global__ void __launch_bounds__(kDigitThreads) digit_scan_kernel(unsigned int* __restrict__ hist, int nblocks,
                                                                  unsigned int* __restrict__ totals) {
  __shared__ unsigned int part[kDigitThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned int* row = hist + (size_t)blockIdx.x * nblocks;
  unsigned int v[kDigitPer], s = 0;
#pragma unroll
  for (int k = 0; k < kDigitPer; ++k) {
    const int i = tid * kDigitPer + k;
    v[k] = i < nblocks ? row[i] : 0u;
    s += v[k];
  }
  unsigned int x = s;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) part[warp] = x;
  __syncthreads();
  unsigned int before = 0;
  for (int w = 0; w < warp; ++w) before += part[w];
  unsigned int run = before + x - s;
#pragma unroll
  for (int k = 0; k < kDigitPer; ++k) {
    const int i = tid * kDigitPer + k;
    if (i < nblocks) row[i] = run;
    run += v[k];
  }
  if (tid == kDigitThreads - 1) totals[blockIdx.x] = before + x;
}

template <int NB, int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(const unsigned int* __restrict__ kin,
                                                                    const unsigned int* __restrict__ vin,
                                                                    unsigned int* __restrict__ kout,
                                                                    unsigned int* __restrict__ vout, int n, int shift,
                                                                    const unsigned int* __restrict__ scanned,
                                                                    int nblocks, unsigned int* __restrict__ cell_start,
                                                                    int n_cells,
                                                                    const unsigned int* __restrict__ totals) {
  __shared__ unsigned int cnt[8][NB];
  __shared__ unsigned int dbase[NB];  // keys of all smaller digits (0 when `scanned` is already global)
  __shared__ unsigned int wpart[kSortThreads / 32];
  const int w = threadIdx.x >> 5, base = blockIdx.x * (ROUNDS * kSortThreads) + w * (ROUNDS * 32);
  unsigned int key[ROUNDS], val[ROUNDS];
  load_keys<ROUNDS>(kin, base, n, key);
  load_keys<ROUNDS>(vin, base, n, val);
  if (totals) {
    // exclusive scan of the digit totals, NB / kSortThreads consecutive digits per thread
    constexpr int PER = NB / kSortThreads;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int v[PER], t = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      v[k] = totals[threadIdx.x * PER + k];
      t += v[k];
    }
    unsigned int x = t;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= off) x += y;
    }
    if (lane == 31) wpart[warp] = x;
    __syncthreads();
    unsigned int run = x - t;
    for (int w = 0; w < warp; ++w) run += wpart[w];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      dbase[threadIdx.x * PER + k] = run;
      run += v[k];
    }
  } else {
    for (int d = threadIdx.x; d < NB; d += kSortThreads) dbase[d] = 0u;
  }
  for (int i = threadIdx.x; i < 8 * NB; i += kSortThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  // one-pass sort (the digit is the whole cell index): the start of cell c in
  // the sorted order is the exclusive prefix of digit c, block 0's entry
  if (cell_start && blockIdx.x == 0)
    for (int c = threadIdx.x; c <= n_cells; c += kSortThreads)
      cell_start[c] = c < NB ? dbase[c] + scanned[(size_t)c * nblocks] : (unsigned int)n;
  warp_digit_counts<NB, ROUNDS>(key, base, n, shift, cnt[w]);
  __syncthreads();
  for (int d = threadIdx.x; d < NB; d += kSortThreads) {
    unsigned int at = dbase[d] + scanned[(size_t)d * nblocks + blockIdx.x];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const unsigned int c = cnt[q][d];
      cnt[q][d] = at;
      at += c;
    }
  }
  __syncthreads();
  warp_scatter<NB, ROUNDS>(key, val, base, n, shift, cnt[w], kout, vout);
}

// Second half of the sort when the leading eight bits of the cell index are
// in order: the keys of a leading digit (about n / 256, in chunks of 2048) are
// sorted by the remaining LOW bits in shared memory, stable, and the starts of
// the digit's cells written.  In place of a second histogram, scan and scatter
// over all keys and a pass for the cell starts.
//
// One block on a digit's keys is right where points spread.  Where they may
// crowd (points a caller gave, or drawn by the error), one block could be left
// with most of the batch: 2^18 points in one digit took 0.3 ms where the rest
// of the sort takes 0.02.  From kCutFrom points on, digits of more than
// kBucketWhole keys are therefore cut into segments: the blocks behind the
// first 256 count them, bucket_split_kernel scatters each from the counts of
// all.  Both find their segment from the digits' totals; a block without one
// ends at once (4 us a step, which evenly drawn points do not pay).
constexpr int kBucketWhole = 65536, kCutFrom = 2 * kBucketWhole, kSegKeys = 8192, kSegMost = 32;

// Keys of a segment of a digit with `total` keys: 8192 at least, at most 32 segments.
__host__ __device__ inline int seg_len(int total) {
  const int each = (total + kSegMost - 1) / kSegMost;
  return each <= kSegKeys ? kSegKeys : (each + 2047) / 2048 * 2048;
}
// At least the segments of n keys, however they fall (a cut digit with t >
// kBucketWhole keys has at most t / 8192 + 1 <= 9 t / 65536 of them).
inline int seg_count(int n) { return n <= kCutFrom ? 0 : (int)((long long)n * 9 / 65536); }
inline int bucket_low(int bits) { return bits <= 16 ? 8 : 10; }  // log2 of the bins of one digit

struct Segment {
  int digit, first, c0, c1;  // leading digit, its first key, the segment's keys
  int row0, index, rows;     // count rows of the digit's segments: the first, this one, how many
};

// Segment `id` of all cut digits (256 threads; the same answer in all, digit < 0: none).
__device__ __forceinline__ Segment find_segment(const unsigned int* __restrict__ totals, int id) {
  __shared__ int wsum[2][8];
  __shared__ Segment found;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int total = (int)totals[tid], len = seg_len(total);
  const int segs = total > kBucketWhole ? (total + len - 1) / len : 0;
  if (!__syncthreads_or(segs)) return Segment{-1, 0, 0, 0, 0, 0, 0};  // no digit is cut
  int a = total, b = segs;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, a, off), z = __shfl_up_sync(0xffffffffu, b, off);
    if (lane >= off) {
      a += y;
      b += z;
    }
  }
  if (lane == 31) {
    wsum[0][w] = a;
    wsum[1][w] = b;
  }
  if (tid == 0) found.digit = -1;
  __syncthreads();
  for (int q = 0; q < w; ++q) {
    a += wsum[0][q];
    b += wsum[1][q];
  }
  const int first = a - total, row0 = b - segs;
  if (id >= row0 && id < row0 + segs) {
    const int c0 = first + (id - row0) * len;
    found = Segment{tid, first, c0, min(c0 + len, first + total), row0, id - row0, segs};
  }
  __syncthreads();
  return found;
}

// next[low bits] += counts of the keys c0 .. c1 - 1 (one add per value a warp
// meets, so that equal keys do not queue up).
__device__ __forceinline__ void count_low(const unsigned int* __restrict__ kin, int c0, int c1, unsigned int mask,
                                          unsigned int* next) {
  for (int base = c0; base < c1; base += kSortThreads) {
    const int i = base + (int)threadIdx.x;
    const unsigned int d = i < c1 ? kin[i] & mask : 0xFFFFFFFFu;
    const unsigned int peers = __match_any_sync(0xffffffffu, d);
    if (i < c1 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&next[d], (unsigned int)__popc(peers));
  }
}

// next[bin] (counts of a whole digit) -> the position of the bin's first key,
// `first` being the digit's; writes the starts of the digit's cells when asked.
template <int NB>
__device__ __forceinline__ void scan_bins(unsigned int* next, unsigned int first, unsigned int mask, int digit,
                                          int low_bits, long long n_cells, unsigned int* __restrict__ cell_start) {
  constexpr int PER = NB / kSortThreads;  // consecutive bins of a thread
  __shared__ unsigned int wpart[kSortThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  unsigned int v[PER], t = 0u;
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    v[e] = next[tid * PER + e];
    t += v[e];
  }
  unsigned int x = t;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) wpart[w] = x;
  __syncthreads();
  unsigned int run = first + x - t;
  for (int q = 0; q < w; ++q) run += wpart[q];
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    const int bin = tid * PER + e;
    const long long cell = ((long long)digit << low_bits) + bin;
    if (cell_start && bin <= (int)mask && cell < n_cells) cell_start[cell] = run;
    next[bin] = run;
    run += v[e];
  }
}

// Stable scatter of the keys c0 .. c1 - 1 of one digit by their low bits from
// next[bin], the position of the bin's next key.
template <int NB>
__device__ __forceinline__ void scatter_low(const unsigned int* __restrict__ kin, const unsigned int* __restrict__ vin,
                                            unsigned int* __restrict__ vout, int c0, int c1, unsigned int mask,
                                            unsigned int (*cnt)[NB], unsigned int* next) {
  constexpr int ROUNDS = 8;
  const int tid = threadIdx.x, w = tid >> 5;
  for (int c = c0; c < c1; c += ROUNDS * kSortThreads) {
    const int base = c + w * (ROUNDS * 32);
    unsigned int key[ROUNDS], val[ROUNDS];
    load_keys<ROUNDS>(kin, base, c1, key);
    load_keys<ROUNDS>(vin, base, c1, val);
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) key[r] &= mask;
    for (int i = tid; i < 8 * NB; i += kSortThreads) (&cnt[0][0])[i] = 0u;
    __syncthreads();
    warp_digit_counts<NB, ROUNDS>(key, base, c1, 0, cnt[w]);
    __syncthreads();
    for (int d = tid; d < NB; d += kSortThreads) {
      unsigned int at = next[d];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const unsigned int c = cnt[q][d];
        cnt[q][d] = at;
        at += c;
      }
      next[d] = at;
    }
    __syncthreads();
    warp_scatter<NB, ROUNDS>(key, val, base, c1, 0, cnt[w], nullptr, vout);
    __syncthreads();
  }
}

template <int LOW>
__global__ void __launch_bounds__(kSortThreads) bucket_sort_kernel(const unsigned int* __restrict__ kin,
                                                                   const unsigned int* __restrict__ vin,
                                                                   unsigned int* __restrict__ vout, int n,
                                                                   int low_bits, unsigned int* __restrict__ cell_start,
                                                                   long long n_cells,
                                                                   const unsigned int* __restrict__ totals, int whole,
                                                                   unsigned int* __restrict__ seg_counts) {
  constexpr int NB = 1 << LOW;
  __shared__ unsigned int cnt[8][NB];
  __shared__ unsigned int next[NB];
  __shared__ unsigned int wpart[kSortThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const unsigned int mask = (1u << low_bits) - 1u;
  for (int i = tid; i < NB; i += kSortThreads) next[i] = 0u;
  if (blockIdx.x >= 256) {
    const int id = (int)blockIdx.x - 256;
    const Segment s = find_segment(totals, id);
    if (s.digit < 0) return;
    count_low(kin, s.c0, s.c1, mask, next);
    __syncthreads();
    for (int i = tid; i < NB; i += kSortThreads) seg_counts[(size_t)id * NB + i] = next[i];
    return;
  }
  // keys of the smaller leading digits
  unsigned int before = tid < (int)blockIdx.x ? totals[tid] : 0u;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
  if (lane == 0) wpart[w] = before;
  __syncthreads();
  unsigned int first = 0u;
#pragma unroll
  for (int q = 0; q < kSortThreads / 32; ++q) first += wpart[q];
  if (blockIdx.x == 0 && tid == 0) cell_start[n_cells] = (unsigned int)n;
  const int total = (int)totals[blockIdx.x];
  if (total > whole) return;  // bucket_split_kernel's
  const int b0 = (int)first, b1 = b0 + total;
  for (int i = b0 + tid; i < b1; i += kSortThreads) atomicAdd(&next[kin[i] & mask], 1u);
  __syncthreads();
  scan_bins<NB>(next, first, mask, (int)blockIdx.x, low_bits, n_cells, cell_start);
  scatter_low<NB>(kin, vin, vout, b0, b1, mask, cnt, next);
}

template <int LOW>
__global__ void __launch_bounds__(kSortThreads) bucket_split_kernel(const unsigned int* __restrict__ kin,
                                                                    const unsigned int* __restrict__ vin,
                                                                    unsigned int* __restrict__ vout, int low_bits,
                                                                    unsigned int* __restrict__ cell_start,
                                                                    long long n_cells,
                                                                    const unsigned int* __restrict__ totals,
                                                                    const unsigned int* __restrict__ seg_counts) {
  constexpr int NB = 1 << LOW;
  __shared__ unsigned int cnt[8][NB];
  __shared__ unsigned int next[NB], before[NB];
  const int tid = threadIdx.x;
  const Segment s = find_segment(totals, (int)blockIdx.x);
  if (s.digit < 0) return;
  for (int i = tid; i < NB; i += kSortThreads) {
    unsigned int all = 0u, b = 0u;
    const unsigned int* row = seg_counts + (size_t)s.row0 * NB + i;
#pragma unroll 8
    for (int q = 0; q < s.rows; ++q) {
      const unsigned int c = row[(size_t)q * NB];
      all += c;
      b += q < s.index ? c : 0u;
    }
    next[i] = all;
    before[i] = b;
  }
  __syncthreads();
  const unsigned int mask = (1u << low_bits) - 1u;
  scan_bins<NB>(next, (unsigned int)s.first, mask, s.digit, low_bits, n_cells, s.index == 0 ? cell_start : nullptr);
  __syncthreads();
  for (int i = tid; i < NB; i += kSortThreads) next[i] += before[i];
  scatter_low<NB>(kin, vin, vout, s.c0, s.c1, mask, cnt, next);
}

// segs: blocks for the segments of crowded digits (seg_count; 0: no digit is cut).
template <int LOW>
void launch_buckets(const unsigned int* kin, const unsigned int* vin, unsigned int* vout, int n, int bits,
                    unsigned int* cell_start, long long n_cells, const unsigned int* totals, int segs,
                    unsigned int* seg_counts, cudaStream_t st) {
  bucket_sort_kernel<LOW><<<256 + segs, kSortThreads, 0, st>>>(kin, vin, vout, n, bits - 8, cell_start, n_cells,
                                                               totals, segs > 0 ? kBucketWhole : INT_MAX, seg_counts);
  if (segs > 0)
    bucket_split_kernel<LOW><<<segs, kSortThreads, 0, st>>>(kin, vin, vout, bits - 8, cell_start, n_cells, totals,
                                                            seg_counts);
}

// cell_start[c] = first sorted position with key >= c, for c in [0, n_cells].
__global__ void cell_start_kernel(const unsigned int* __restrict__ skeys, int n, unsigned int* __restrict__ start,
                                  int n_cells) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s > n) return;
  const int cur = s < n ? (int)skeys[s] : n_cells;
  const int prev = s > 0 ? (int)skeys[s - 1] : -1;
  for (int c = prev + 1; c <= cur; ++c) start[c] = (unsigned int)s;
}

// One warp per grid vertex: gather w_corner(p_j) * dz_j over the points of the
// vertex's adjacent cells (fixed cell order, sorted point order, lane-strided)
// and reduce across lanes with a fixed butterfly.
struct GradArgs {
  const float* pts;
  const float* dz;
  const unsigned int* sidx;
  const unsigned int* start;
  const float* cell_part;
  int R;
  float w0, w1;
  float* g0;
  float* g1;
};

template <int F>
__device__ __forceinline__ void grid_grad_block(const GradArgs& a, int block, unsigned int* __restrict__ flag) {
  const float* __restrict__ pts = a.pts;
  const float* __restrict__ dz = a.dz;
  const unsigned int* __restrict__ sidx = a.sidx;
  const unsigned int* __restrict__ start = a.start;
  const int R = a.R;
  const float w0 = a.w0, w1 = a.w1;
  float* __restrict__ g0 = a.g0;
  float* __restrict__ g1 = a.g1;
  const long long v = ((long long)block * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (v >= (long long)R * R * R) return;
  const int vx = (int)(v % R), vy = (int)((v / R) % R), vz = (int)(v / ((long long)R * R));
  float acc[F];
#pragma unroll
  for (int f = 0; f < F; ++f) acc[f] = 0.f;
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dzz = c >> 2;
    const int cx = vx - dx, cy = vy - dy, cz = vz - dzz;
    if (cx < 0 || cy < 0 || cz < 0 || cx > R - 2 || cy > R - 2 || cz > R - 2) continue;
    const int cell = (cz * (R - 1) + cy) * (R - 1) + cx;
    const int s0 = (int)start[cell], s1 = (int)start[cell + 1];
    for (int s = s0 + lane; s < s1; s += 32) {
      const int j = (int)sidx[s];
      int ix, iy, iz;
      float fx, fy, fz;
      cell_coord(pts[3 * j], R, ix, fx);
      cell_coord(pts[3 * j + 1], R, iy, fy);
      cell_coord(pts[3 * j + 2], R, iz, fz);
      const float w = (dx ? fx : 1.0f - fx) * (dy ? fy : 1.0f - fy) * (dzz ? fz : 1.0f - fz);
      const float4* zz = reinterpret_cast<const float4*>(dz + (size_t)j * F);
#pragma unroll
      for (int f = 0; f < F; f += 4) {
        const float4 q = zz[f / 4];
        acc[f] = fmaf(w, q.x, acc[f]);
        acc[f + 1] = fmaf(w, q.y, acc[f + 1]);
        acc[f + 2] = fmaf(w, q.z, acc[f + 2]);
        acc[f + 3] = fmaf(w, q.w, acc[f + 3]);
      }
    }
  }
#pragma unroll
  for (int f = 0; f < F; ++f)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], off);
  if (lane == 0) {
    bool bad = false;
#pragma unroll
    for (int f = 0; f < F; ++f) {
      g0[(size_t)v * F + f] = w0 * acc[f];
      if (g1) g1[(size_t)v * F + f] = w1 * acc[f];
      bad |= !isfinite(acc[f]);
    }
    if (bad) atomicOr(flag, 1u);
  }
}

// Dense cells (many points per cell): one block of 8 warps per cell, warp c
// sums w_corner_c(p) * dz over the cell's points (sorted order, lane-strided,
// fixed butterfly) into part[cell][c][F]; vertex_gather_block then adds the
// <= 8 partials of each vertex in a fixed order.  The block stages the cell's
// points (place in the cell, dz) in shared memory 256 at a time, so each point is
// gathered from global memory once instead of once per corner; lane l still
// takes points l, l + 32, ... in order, so the sums are those of a warp
// reading global memory directly.
template <int F>
__global__ void __launch_bounds__(256) cell_corner_kernel(const float* __restrict__ pts,
                                                          const float* __restrict__ dz,
                                                          const unsigned int* __restrict__ sidx,
                                                          const unsigned int* __restrict__ start, int R,
                                                          long long n_cells, float* __restrict__ part) {
  constexpr int kChunk = 256;
  __shared__ float sp[kChunk][3];
  __shared__ float4 sz[kChunk][F / 4];
  const long long cell = blockIdx.x;
  if (cell >= n_cells) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = warp;
  const int dx = c & 1, dy = (c >> 1) & 1, dzz = c >> 2;
  float acc[F];
#pragma unroll
  for (int f = 0; f < F; ++f) acc[f] = 0.f;
  const int s0 = (int)start[cell], s1 = (int)start[cell + 1];
  // a thread's point of the next chunk is loaded while this one is summed
  // (its index one chunk earlier still)
  const int tid = threadIdx.x;
  int j = s0 + tid < s1 ? (int)sidx[s0 + tid] : 0;
  float3 q = make_float3(0.f, 0.f, 0.f);
  float4 z[F / 4];
  auto fetch = [&](bool any) {
    if (!any) return;
    q = make_float3(pts[3 * (size_t)j], pts[3 * (size_t)j + 1], pts[3 * (size_t)j + 2]);
    const float4* zz = reinterpret_cast<const float4*>(dz + (size_t)j * F);
#pragma unroll
    for (int f = 0; f < F / 4; ++f) z[f] = zz[f];
  };
  fetch(s0 + tid < s1);
  j = s0 + kChunk + tid < s1 ? (int)sidx[s0 + kChunk + tid] : 0;
  for (int base = s0; base < s1; base += kChunk) {
    const int cnt = min(kChunk, s1 - base);
    __syncthreads();
    if (tid < cnt) {
      int i;
      cell_coord(q.x, R, i, sp[tid][0]);
      cell_coord(q.y, R, i, sp[tid][1]);
      cell_coord(q.z, R, i, sp[tid][2]);
#pragma unroll
      for (int f = 0; f < F / 4; ++f) sz[tid][f] = z[f];
    }
    __syncthreads();
    fetch(base + kChunk + tid < s1);
    j = base + 2 * kChunk + tid < s1 ? (int)sidx[base + 2 * kChunk + tid] : 0;
    for (int i = lane; i < cnt; i += 32) {
      const float fx = sp[i][0], fy = sp[i][1], fz = sp[i][2];
      const float w = (dx ? fx : 1.0f - fx) * (dy ? fy : 1.0f - fy) * (dzz ? fz : 1.0f - fz);
#pragma unroll
      for (int f = 0; f < F; f += 4) {
        const float4 q = sz[i][f / 4];
        acc[f] = fmaf(w, q.x, acc[f]);
        acc[f + 1] = fmaf(w, q.y, acc[f + 1]);
        acc[f + 2] = fmaf(w, q.z, acc[f + 2]);
        acc[f + 3] = fmaf(w, q.w, acc[f + 3]);
      }
    }
  }
#pragma unroll
  for (int f = 0; f < F; ++f)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], off);
  if (lane == 0) {
#pragma unroll
    for (int f = 0; f < F; ++f) part[((size_t)cell * 8 + c) * F + f] = acc[f];
  }
}

// Sparse cells (few points per cell): one warp per cell.  A lane owns one
// corner and four channels (F = 16: 8 x 4 lanes; narrower vectors leave lane
// groups that take every second or fourth point, wider ones give a lane two
// channel groups), the points' cell coordinates are computed one point per
// lane and handed round, and a point's dz row is read once per warp instead
// of once per vertex.  The corner sums go to part[cell][corner][F], summed per
// vertex by vertex_gather_block as for dense cells.  Bound by the latency of
// three dependent loads per cell (offsets, point index, point); a warp per
// vertex over its eight cells, with its butterfly over 32 mostly idle lanes,
// took 57 us for 32^3 vertices whatever the number of points.
//
// Points may crowd: a cell of more than kLongCell points is left to all eight
// warps of its CTA (one warp on 2^18 points of one cell: 32 ms; so 2.2).
constexpr int kLongCell = 96;

constexpr int kCellPass = 16;  // points a warp brings to shared memory at a time

// Corner sums of a crowded cell's points, the rows of dz through shared memory
// so that a pass has one wait for all of them.
template <int F>
struct CellSum {
  static constexpr int QL = F >= 16 ? 4 : F / 4;  // lanes per corner
  static constexpr int QN = F / (4 * QL);         // channel groups per lane
  static constexpr int G = 32 / (8 * QL);         // points side by side
  static constexpr int LR = F / 4;                // lanes per row of dz
  static constexpr int P = kCellPass, NR = P * LR >= 32 ? P * LR / 32 : 1;  // row loads of a lane
  float4 acc[QN];

  // acc = the corner sums of the points base .. base + P - 1, then `stride`
  // on, up to s1.  Each P are summed first, so that the rounding error does
  // not grow with the length of one chain.  weights (of the eight corners) and
  // rows: the warp's P entries.
  __device__ __forceinline__ void run(const float* __restrict__ pts, const float* __restrict__ dz,
                                      const unsigned int* __restrict__ sidx, int R, int base, int s1, int stride,
                                      float4 (*weights)[2], float4 (*rows)[LR]) {
    const int lane = threadIdx.x & 31, g = lane / (8 * QL), c = (lane / QL) & 7, q = lane % QL;
#pragma unroll
    for (int e = 0; e < QN; ++e) acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    // a pass's points and rows are loaded while the one before is summed,
    // their indices one pass earlier still
    float4 v[NR];
    float3 at = make_float3(0.f, 0.f, 0.f);
    int j = index_at(sidx, base, s1);
    auto fetch = [&](int b) {
#pragma unroll
      for (int e = 0; e < NR; ++e) {
        const int src = e * (32 / LR) + lane / LR, jk = __shfl_sync(0xffffffffu, j, src);
        if (src < P && b + src < s1) v[e] = reinterpret_cast<const float4*>(dz + (size_t)jk * F)[lane % LR];
      }
      if (lane < P && b + lane < s1)
        at = make_float3(pts[3 * (size_t)j], pts[3 * (size_t)j + 1], pts[3 * (size_t)j + 2]);
      j = index_at(sidx, b + stride, s1);
    };
    fetch(base);
#pragma unroll 1
    for (; base < s1; base += stride) {
      const int cnt = min(P, s1 - base);
      if (lane < cnt) {
        int i;
        float x, y, z;
        cell_coord(at.x, R, i, x);
        cell_coord(at.y, R, i, y);
        cell_coord(at.z, R, i, z);
        const float u = 1.0f - z, yz[4] = {(1.0f - y) * u, y * u, (1.0f - y) * z, y * z};
        weights[lane][0] = make_float4((1.0f - x) * yz[0], x * yz[0], (1.0f - x) * yz[1], x * yz[1]);
        weights[lane][1] = make_float4((1.0f - x) * yz[2], x * yz[2], (1.0f - x) * yz[3], x * yz[3]);
      }
#pragma unroll
      for (int e = 0; e < NR; ++e) {
        const int src = e * (32 / LR) + lane / LR;
        if (src < cnt) rows[src][lane % LR] = v[e];
      }
      __syncwarp();
      fetch(base + stride);
      float4 a[QN];
#pragma unroll
      for (int e = 0; e < QN; ++e) a[e] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int k = g; k < cnt; k += G) {
        const float w = reinterpret_cast<const float*>(weights[k])[c];
#pragma unroll
        for (int e = 0; e < QN; ++e) {
          const float4 x = rows[k][q + e * QL];
          a[e].x = fmaf(w, x.x, a[e].x);
          a[e].y = fmaf(w, x.y, a[e].y);
          a[e].z = fmaf(w, x.z, a[e].z);
          a[e].w = fmaf(w, x.w, a[e].w);
        }
      }
      __syncwarp();
#pragma unroll
      for (int e = 0; e < QN; ++e) {
        acc[e].x += a[e].x;
        acc[e].y += a[e].y;
        acc[e].z += a[e].z;
        acc[e].w += a[e].w;
      }
    }
#pragma unroll
    for (int e = 0; e < QN; ++e)
#pragma unroll
      for (int off = 8 * QL; off < 32; off <<= 1) {
        acc[e].x += __shfl_xor_sync(0xffffffffu, acc[e].x, off);
        acc[e].y += __shfl_xor_sync(0xffffffffu, acc[e].y, off);
        acc[e].z += __shfl_xor_sync(0xffffffffu, acc[e].z, off);
        acc[e].w += __shfl_xor_sync(0xffffffffu, acc[e].w, off);
      }
  }
  // The lane's point of the P from b on.
  static __device__ __forceinline__ int index_at(const unsigned int* __restrict__ sidx, int b, int s1) {
    const int i = b + (int)(threadIdx.x & 31);
    return (threadIdx.x & 31) < P && i < s1 ? (int)sidx[i] : 0;
  }
  // The sums as rows [8 corners][F] of out.
  __device__ __forceinline__ void store(float* out) const {
    const int lane = threadIdx.x & 31;
    if (lane >= 8 * QL) return;
    float4* o = reinterpret_cast<float4*>(out + (lane / QL) * F) + lane % QL;
#pragma unroll
    for (int e = 0; e < QN; ++e) o[e * QL] = acc[e];
  }
};

// The crowded cells of a CTA (bits of `crowded`; lane l holds the first point
// of cell l and of the next one), by all its warps.
template <int F>
__device__ __noinline__ void crowded_cells(const float* __restrict__ pts, const float* __restrict__ dz,
                                           const unsigned int* __restrict__ sidx, int R, long long cell0, int at,
                                           int end, unsigned int crowded, float* __restrict__ part) {
  __shared__ float4 weights[8][kCellPass][2], rows[8][kCellPass][F / 4];
  const int warp = threadIdx.x >> 5;
  for (unsigned int left = crowded; left; left &= left - 1) {
    const int w = __ffs(left) - 1;
    const int c0 = __shfl_sync(0xffffffffu, at, w), c1 = __shfl_sync(0xffffffffu, end, w);
    CellSum<F> sum;
    sum.run(pts, dz, sidx, R, c0 + kCellPass * warp, c1, 8 * kCellPass, weights[warp], rows[warp]);
    sum.store(reinterpret_cast<float*>(rows[warp]));  // a warp's rows hold twice its sums
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * F; i += 256) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) t += reinterpret_cast<const float*>(rows[k])[i];
      part[(size_t)(cell0 + w) * 8 * F + i] = t;
    }
    __syncthreads();
  }
}

template <int F>
__global__ void __launch_bounds__(256, 6)
    cell_warp_kernel(const float* __restrict__ pts, const float* __restrict__ dz, const unsigned int* __restrict__ sidx,
                     const unsigned int* __restrict__ start, int R, long long n_cells, float* __restrict__ part) {
  constexpr int QL = F >= 16 ? 4 : F / 4;      // lanes per corner
  constexpr int QN = F / (4 * QL);             // channel groups per lane
  constexpr int G = 32 / (8 * QL);             // points side by side
  const int lane = threadIdx.x & 31, g = lane / (8 * QL), c = (lane / QL) & 7, q = lane % QL;
  const int warp = threadIdx.x >> 5;
  const long long cell0 = (long long)blockIdx.x * 8, cell = cell0 + warp;
  // every warp reads the offsets of the CTA's cells, so that all know without
  // a barrier which ones are crowded
  const int at = lane < 9 ? (int)start[min(cell0 + lane, n_cells)] : 0;
  const int end = __shfl_down_sync(0xffffffffu, at, 1);
  const unsigned int crowded = __ballot_sync(0xffffffffu, lane < 8 && end - at > kLongCell);
  if (crowded) crowded_cells<F>(pts, dz, sidx, R, cell0, at, end, crowded, part);
  if (cell >= n_cells || (crowded >> warp & 1u)) return;
  const int s0 = __shfl_sync(0xffffffffu, at, warp), s1 = __shfl_sync(0xffffffffu, end, warp);
  float4 acc[QN];
#pragma unroll
  for (int e = 0; e < QN; ++e) acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int base = s0; base < s1; base += 32) {
    const int cnt = min(32, s1 - base);
    int j = 0, i;
    float fx = 0.f, fy = 0.f, fz = 0.f;
    if (lane < cnt) {
      j = (int)sidx[base + lane];
      cell_coord(pts[3 * (size_t)j], R, i, fx);
      cell_coord(pts[3 * (size_t)j + 1], R, i, fy);
      cell_coord(pts[3 * (size_t)j + 2], R, i, fz);
    }
#pragma unroll 4
    for (int k = 0; k < cnt; k += G) {
      const int src = k + g;  // lanes past cnt hold zeros; their weight is cleared below
      const int jk = __shfl_sync(0xffffffffu, j, src);
      const float x = __shfl_sync(0xffffffffu, fx, src), y = __shfl_sync(0xffffffffu, fy, src),
                  z = __shfl_sync(0xffffffffu, fz, src);
      if (G == 1 || src < cnt) {
        const float w = ((c & 1) ? x : 1.0f - x) * ((c & 2) ? y : 1.0f - y) * ((c & 4) ? z : 1.0f - z);
        const float4* row = reinterpret_cast<const float4*>(dz + (size_t)jk * F) + q;
#pragma unroll
        for (int e = 0; e < QN; ++e) {
          const float4 v = row[e * QL];
          acc[e].x = fmaf(w, v.x, acc[e].x);
          acc[e].y = fmaf(w, v.y, acc[e].y);
          acc[e].z = fmaf(w, v.z, acc[e].z);
          acc[e].w = fmaf(w, v.w, acc[e].w);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < QN; ++e) {
#pragma unroll
    for (int off = 8 * QL; off < 32; off <<= 1) {
      acc[e].x += __shfl_xor_sync(0xffffffffu, acc[e].x, off);
      acc[e].y += __shfl_xor_sync(0xffffffffu, acc[e].y, off);
      acc[e].z += __shfl_xor_sync(0xffffffffu, acc[e].z, off);
      acc[e].w += __shfl_xor_sync(0xffffffffu, acc[e].w, off);
    }
    if (g == 0) reinterpret_cast<float4*>(part + ((size_t)cell * 8 + c) * F)[q + e * QL] = acc[e];
  }
}

template <int F>
__device__ __forceinline__ void vertex_gather_block(const GradArgs& a, int block, unsigned int* __restrict__ flag) {
  const float* __restrict__ part = a.cell_part;
  const int R = a.R;
  const float w0 = a.w0, w1 = a.w1;
  float* __restrict__ g0 = a.g0;
  float* __restrict__ g1 = a.g1;
  const long long i = (long long)block * blockDim.x + threadIdx.x;
  if (i >= (long long)R * R * R * F) return;
  const long long v = i / F;
  const int f = (int)(i - v * F);
  const int vx = (int)(v % R), vy = (int)((v / R) % R), vz = (int)(v / ((long long)R * R));
  float acc = 0.f;
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dzz = c >> 2;
    const int cx = vx - dx, cy = vy - dy, cz = vz - dzz;
    if (cx < 0 || cy < 0 || cz < 0 || cx > R - 2 || cy > R - 2 || cz > R - 2) continue;
    const long long cell = ((long long)cz * (R - 1) + cy) * (R - 1) + cx;
    acc += part[(cell * 8 + c) * F + f];
  }
  g0[i] = w0 * acc;
  if (g1) g1[i] = w1 * acc;
  if (!isfinite(acc)) atomicOr(flag, 1u);
}

// Fixed-order sum of the CTA partials: weights, biases and the loss.  A
// block covers 32 entries; its 8 warps each sum a contiguous eighth of the
// partial rows in row order, then the 8 sums are added in warp order.
struct ReduceArgs {
  const float* part;
  int n_cta, nW, nb;
  float* outW;
  float* outb;
  float* loss;
  float inv_n;
};

__device__ __forceinline__ void reduce_parts_block(const ReduceArgs& a, int block, unsigned int* __restrict__ flag) {
  __shared__ float acc[8][32];
  const float* __restrict__ part = a.part;
  const int n_cta = a.n_cta, nW = a.nW, nb = a.nb;
  float* __restrict__ outW = a.outW;
  float* __restrict__ outb = a.outb;
  float* __restrict__ loss = a.loss;
  const float inv_n = a.inv_n;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = block * 32 + lane;
  const int ne = nW + nb;
  const int r0 = (int)((long long)n_cta * w / 8), r1 = (int)((long long)n_cta * (w + 1) / 8);
  float s = 0.f;
  if (e <= ne) {
#pragma unroll 16  // the loads in flight together; the sum stays in row order
    for (int c = r0; c < r1; ++c) s += part[(size_t)c * (ne + 1) + e];
  }
  acc[w][lane] = s;
  __syncthreads();
  if (w == 0 && e <= ne) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += acc[k][lane];
    if (e < nW) outW[e] = t;
    else if (e < ne) outb[e - nW] = t;
    else if (loss) {
      t *= inv_n;
      *loss = t;
    }
    if (!isfinite(t) && (e < ne || loss)) atomicOr(flag, 1u);
  }
}

// The latent-grid gradient gather and the fixed-order reduction of the
// weight partials are independent: one launch runs both, blocks
// [0, gather_blocks) gathering, the rest reducing.
template <int F, bool DENSE>
__global__ void __launch_bounds__(256) grad_tail_kernel(const GradArgs g, int gather_blocks, const ReduceArgs r,
                                                        unsigned int* __restrict__ flag) {
  if ((int)blockIdx.x < gather_blocks) {
    if (DENSE) vertex_gather_block<F>(g, blockIdx.x, flag);
    else grid_grad_block<F>(g, blockIdx.x, flag);
  } else {
    reduce_parts_block(r, blockIdx.x - gather_blocks, flag);
  }
}

__device__ __forceinline__ void adam_update(float* __restrict__ grid, float* __restrict__ W, float* __restrict__ b,
                                            const float* __restrict__ g, float* __restrict__ m,
                                            float* __restrict__ v, size_t ng, size_t nW, size_t nb, float lr_grid,
                                            float lr_net, int step, __half* __restrict__ grid_h,
                                            __half* __restrict__ W_h, const int* __restrict__ grid_exp) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const int gk = (grid_h && grid_exp) ? *grid_exp : 0;
  const float t1 = (float)step + 1.0f;  // exact below 2^24; no int overflow at INT_MAX
  const float bc1 = 1.0f - powf(b1, t1), bc2 = 1.0f - powf(b2, t1);
  const size_t n = ng + nW + nb;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float upd = (mi / bc1) / (sqrtf(vi / bc2) + eps);
    if (i < ng) {
      const float t = grid[i] - lr_grid * upd;
      grid[i] = t;
      if (grid_h) grid_h[i] = __float2half_rn(ldexpf(t, -gk));
    } else if (i < ng + nW) {
      const float t = W[i - ng] - lr_net * upd;
      W[i - ng] = t;
      if (W_h) W_h[i - ng] = __float2half_rn(t);
    } else {
      b[i - ng - nW] -= lr_net * upd;
    }
  }
}

// Adam (beta1 0.9, beta2 0.999, eps 1e-8, bias correction at step + 1) over
// [grid | weights | biases]; refreshes the FP16 copies.  Skipped entirely
// when the step produced a non-finite loss or gradient (flag bit 0,
// SRN_ERR_NONFINITE) or a bounded wait of the point kernel gave up (bit 1,
// SRN_ERR_TIMEOUT).  With the step index
// in device memory (step_ptr), the last block to finish advances it by one
// for the next step (flag[1] counts finished blocks and is reset by that block).
__global__ void adam_kernel(float* __restrict__ grid, float* __restrict__ W, float* __restrict__ b,
                            const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v, size_t ng,
                            size_t nW, size_t nb, float lr_grid, float lr_net, int step_arg, int* __restrict__ step_ptr,
                            unsigned int* __restrict__ flag, unsigned int* __restrict__ status,
                            __half* __restrict__ grid_h, __half* __restrict__ W_h,
                            const int* __restrict__ grid_exp) {
  const int step = step_ptr ? *step_ptr : step_arg;
  const unsigned int f = *flag;
  if (f) {
    if (blockIdx.x == 0 && threadIdx.x == 0)
      atomicExch(status, (unsigned int)((f & 2u) ? SRN_ERR_TIMEOUT : SRN_ERR_NONFINITE));
  } else {
    adam_update(grid, W, b, g, m, v, ng, nW, nb, lr_grid, lr_net, step, grid_h, W_h, grid_exp);
  }
  if (step_ptr) {
    __syncthreads();  // every thread of the block has read *step_ptr
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned int done = atomicAdd(flag + 1, 1u);
      if (done == gridDim.x - 1) {
        __threadfence();
        flag[1] = 0u;
        flag[0] = 0u;  // the next replayed step starts with a clear non-finite flag
        *step_ptr = (int)((unsigned int)step + 1u);
      }
    }
  }
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

// Latent-grid gradient and the reduction of the weight partials: per-cell
// corner sums (a block per cell from 32 points a cell on average, where a
// cell's points are worth staging in shared memory, else a warp per cell),
// then the sums of each vertex.  Without the per-cell array (the static
// scratch area, grids whose array would pass kMaxCellPart bytes) a warp per
// vertex gathers from the points.
constexpr size_t kMaxCellPart = (size_t)256 << 20;

template <int F>
void launch_grid_grad(const FitScratch& s, const GradArgs& ga, const ReduceArgs& ra, int rblocks, int n,
                      cudaStream_t st) {
  const long long n_vert = (long long)ga.R * ga.R * ga.R;
  if (!s.cell_part) {
    const int gblocks = (int)((n_vert * 32 + 255) / 256);
    grad_tail_kernel<F, false><<<gblocks + rblocks, 256, 0, st>>>(ga, gblocks, ra, s.flag);
    return;
  }
  const long long cells = (long long)s.n_cells;
  if ((size_t)n >= 32 * s.n_cells)
    cell_corner_kernel<F><<<(unsigned)cells, 256, 0, st>>>(ga.pts, ga.dz, ga.sidx, ga.start, ga.R, cells, s.cell_part);
  else
    cell_warp_kernel<F><<<(unsigned)((cells + 7) / 8), 256, 0, st>>>(ga.pts, ga.dz, ga.sidx, ga.start, ga.R, cells,
                                                                     s.cell_part);
  const int vb = (int)((n_vert * F + 255) / 256);
  grad_tail_kernel<F, true><<<vb + rblocks, 256, 0, st>>>(ga, vb, ra, s.flag);
}

template <int ROUNDS>
void launch_hist(int dbits, int nblocks, const unsigned int* k, int n, int shift, unsigned int* hist, cudaStream_t st) {
  if (dbits == 9) sort_hist_kernel<512, ROUNDS><<<nblocks, kSortThreads, 0, st>>>(k, n, shift, hist, nblocks);
  else sort_hist_kernel<256, ROUNDS><<<nblocks, kSortThreads, 0, st>>>(k, n, shift, hist, nblocks);
}

template <int ROUNDS>
void launch_scatter(int dbits, int nblocks, const unsigned int* k, const unsigned int* v, unsigned int* ko,
                    unsigned int* vo, int n, int shift, const unsigned int* hist, unsigned int* cs, int n_cells,
                    const unsigned int* totals, cudaStream_t st) {
  if (dbits == 9)
    sort_scatter_kernel<512, ROUNDS><<<nblocks, kSortThreads, 0, st>>>(k, v, ko, vo, n, shift, hist, nblocks, cs,
                                                                       n_cells, totals);
  else
    sort_scatter_kernel<256, ROUNDS><<<nblocks, kSortThreads, 0, st>>>(k, v, ko, vo, n, shift, hist, nblocks, cs,
                                                                       n_cells, totals);
}

// Steps 1-4 shared by the fit and the backward.  Writes the grid gradient
// (all keyframes) to dgrid, weights / biases to dW / db, the loss (fit) to
// loss.
cudaError_t run_backward(FitScratch& s, const NetDev& net, PointArgs pa, float* dgrid, float* dW, float* db,
                         float* loss, cudaStream_t st, unsigned int* mma_status = nullptr) {
  const int n = pa.n;
  const int nW = (int)(net_weight_count(net)), nb = (int)net_bias_count(net);
  Layout L = make_layout(net);
  // odd row stride: per-thread rows written at the same column hit distinct banks
  const int dstride = ((net_d0(net) > net.c ? net_d0(net) : net.c) + 1) | 1;
  pa.dstride = dstride;
  pa.n_entries = nW + nb;
  pa.pts = s.pts;
  pa.dz = s.dz;
  pa.key = s.key;
  pa.idx = s.idx;
  pa.part = s.part;
  int n_cta = std::min(s.max_cta, (n + kFitThreads - 1) / kFitThreads);
  size_t smem = sizeof(float) * ((size_t)L.total + kFitThreads * (net.c + 1) + (size_t)kFitThreads * dstride +
                                 ((pa.n_entries + 3) & ~3) + kFitThreads);
  // graph-replayed fit steps (step index in device memory) find the flag
  // cleared by the previous step's Adam kernel or by the replay set-up
  cudaError_t e = pa.step_ptr ? cudaSuccess : cudaMemsetAsync(s.flag, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  if (pa.mode == 0 && n > 0 && mma_status && fit_mma_supported(net) && s.max_cta >= fit_mma_rows_per_cta()) {
    // tensor-core point kernel: one partial row per warpgroup
    const int rows = fit_mma_rows_per_cta();
    const int grid = std::max(1, std::min({sm_count(), s.max_cta / rows, (n + 128 * rows - 1) / (128 * rows)}));
    PointArgsMma ma{n,           pa.seed, pa.step, pa.time, pa.vol, pa.cdf, pa.cdf_res, pa.step_ptr,
                    s.pts,       s.dz,    s.key,   s.idx,  s.part, s.flag, pa.stall_test};
    e = launch_fit_mma(net, ma, grid, mma_status, st);
    if (e != cudaSuccess) return e;
    n_cta = grid * rows;
  } else if (n_cta > 0 && fit_tile_supported(net)) {
    // two CTAs of 128 points per SM
    n_cta = std::min(n_cta, 2 * sm_count());
    if ((e = launch_fit_tile(net, pa, n_cta, st)) != cudaSuccess) return e;
  } else if (n_cta > 0) {
    auto k = fit_point_kernel<32>;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<n_cta, kFitThreads, smem, st>>>(net, pa, L);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // sort (cell, point) by cell
  unsigned int *k_in = s.key, *v_in = s.idx, *k_out = s.key_alt, *v_out = s.idx_alt;
  int bits = 1;
  while (((size_t)1 << bits) < s.n_cells) ++bits;
  const bool small_blocks = s.sort_items == kSortItemsSmall;
  const int nblocks = (n + s.sort_items - 1) / s.sort_items;
  // up to 512 cells: one pass with 9-bit digits; up to 2^18 cells: the leading
  // eight bits, then each leading digit's keys by themselves (18 bits leave
  // ten, 32 KB of counters) where the counts of crowded digits find room (not
  // in the static area past 2^16 cells); else 8-bit digits from the lowest
  const bool one_pass = s.radix_bins == 512 && bits <= 9;
  const int segs = pa.mode == 0 && !pa.cdf ? 0 : seg_count(n);  // evenly drawn points do not crowd
  const bool buckets = !one_pass && bits > 9 && bits <= 18 && nblocks <= kDigitThreads * kDigitPer &&
                       ((size_t)segs << bucket_low(bits)) <= s.hist_len;
  const int dbits = one_pass ? 9 : 8;
  const int hist_m = (1 << dbits) * nblocks;
  const int nseg = (hist_m + kScanTile - 1) / kScanTile;  // one 8192-value tile per scan block
  unsigned int* seg_sums = s.hist + s.hist_len;
  bool starts_done = false;
  for (int shift = buckets ? bits - 8 : 0; shift < bits && n > 0; shift += dbits) {
    // a single pass leaves the cell starts to the scatter kernel
    unsigned int* cs = one_pass ? s.cell_start : nullptr;
    starts_done = one_pass || buckets;
    if (small_blocks) launch_hist<4>(dbits, nblocks, k_in, n, shift, s.hist, st);
    else launch_hist<8>(dbits, nblocks, k_in, n, shift, s.hist, st);
    const unsigned int* totals = nullptr;
    if (nblocks <= kDigitThreads * kDigitPer) {
      // one block per digit; the scatter kernel adds the digits' prefix
      digit_scan_kernel<<<1 << dbits, kDigitThreads, 0, st>>>(s.hist, nblocks, s.digit_totals);
      totals = s.digit_totals;
    } else if (nseg > 1) {
      seg_sum_kernel<<<nseg, kScanThreads, 0, st>>>(s.hist, hist_m, kScanTile, seg_sums);
      scan_kernel<<<1, kScanThreads, 0, st>>>(seg_sums, nseg, nseg, nullptr);
      scan_kernel<<<nseg, kScanThreads, 0, st>>>(s.hist, hist_m, kScanTile, seg_sums);
    } else {
      scan_kernel<<<1, kScanThreads, 0, st>>>(s.hist, hist_m, hist_m, nullptr);
    }
    if (small_blocks)
      launch_scatter<4>(dbits, nblocks, k_in, v_in, k_out, v_out, n, shift, s.hist, cs, (int)s.n_cells, totals, st);
    else
      launch_scatter<8>(dbits, nblocks, k_in, v_in, k_out, v_out, n, shift, s.hist, cs, (int)s.n_cells, totals, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    std::swap(k_in, k_out);
    std::swap(v_in, v_out);
    if (buckets) {
      // the histogram's space is free again: the counts of the segments
      if (bucket_low(bits) == 8)
        launch_buckets<8>(k_in, v_in, v_out, n, bits, s.cell_start, (long long)s.n_cells, totals, segs, s.hist, st);
      else
        launch_buckets<10>(k_in, v_in, v_out, n, bits, s.cell_start, (long long)s.n_cells, totals, segs, s.hist, st);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      std::swap(v_in, v_out);
    }
  }
  if (!starts_done) cell_start_kernel<<<(n + 1 + 255) / 256, 256, 0, st>>>(k_in, n, s.cell_start, (int)s.n_cells);
  // grid gradient: the gathers below write every vertex of the two bracketing
  // keyframes; other keyframes (and everything when there are no points) are zeroed
  const size_t gsz = (size_t)net.R * net.R * net.R * net.F;
  if (net.nkey > 2 || n == 0) {
    e = cudaMemsetAsync(dgrid, 0, sizeof(float) * gsz * net.nkey, st);
    if (e != cudaSuccess) return e;
  }
  int k0 = 0;
  float f = 0.f;
  {
    // keyframe bracket of the step's time (same rule as the kernels' time_weights)
    if (net.nkey > 1) {
      const float t = pa.time;
      if (t <= net.key_times[0]) { k0 = 0; f = 0.f; }
      else if (t >= net.key_times[net.nkey - 1]) { k0 = net.nkey - 2; f = 1.f; }
      else {
        while (k0 < net.nkey - 2 && t >= net.key_times[k0 + 1]) ++k0;
        f = (t - net.key_times[k0]) / (net.key_times[k0 + 1] - net.key_times[k0]);
      }
    }
  }
  const float w0 = net.nkey > 1 ? 1.0f - f : 1.0f, w1 = f;
  float* g0 = dgrid + (size_t)k0 * gsz;
  float* g1 = net.nkey > 1 ? g0 + gsz : nullptr;
  const int ne = nW + nb;
  const ReduceArgs ra{s.part, n_cta, nW, nb, dW, db, loss, 1.0f / (float)n};
  const int rblocks = (ne + 1 + 31) / 32;
  if (n > 0) {
    const GradArgs ga{s.pts, s.dz, v_in, s.cell_start, s.cell_part, net.R, w0, w1, g0, g1};
    switch (net.F) {
      case 4: launch_grid_grad<4>(s, ga, ra, rblocks, n, st); break;
      case 8: launch_grid_grad<8>(s, ga, ra, rblocks, n, st); break;
      case 16: launch_grid_grad<16>(s, ga, ra, rblocks, n, st); break;
      default: launch_grid_grad<32>(s, ga, ra, rblocks, n, st);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else {
    e = cudaMemsetAsync(dW, 0, sizeof(float) * nW, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(db, 0, sizeof(float) * nb, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t fit_scratch_alloc(FitScratch& s, const NetDev& net, int max_points) {
  memset(&s, 0, sizeof(s));
  s.max_points = max_points;
  if (max_points <= 0) return cudaSuccess;
  s.n_cells = (size_t)(net.R - 1) * (net.R - 1) * (net.R - 1);
  s.n_entries = net_weight_count(net) + net_bias_count(net);
  s.n_grid = net_grid_count(net);
  s.max_cta = std::min(4 * sm_count(), (max_points + kFitThreads - 1) / kFitThreads);
  const size_t n = (size_t)max_points;
  s.sort_items = max_points <= kSortItemsSmall * kDigitThreads * kDigitPer ? kSortItemsSmall : kSortItems;
  const size_t nsb = (n + s.sort_items - 1) / s.sort_items;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void** p, size_t bytes) {
    if (e == cudaSuccess) e = cudaMalloc(p, bytes < 16 ? 16 : bytes);
  };
  alloc((void**)&s.pts, sizeof(float) * 3 * n);
  alloc((void**)&s.dz, sizeof(float) * net.F * n);
  alloc((void**)&s.key, sizeof(unsigned int) * n);
  alloc((void**)&s.key_alt, sizeof(unsigned int) * n);
  alloc((void**)&s.idx, sizeof(unsigned int) * n);
  alloc((void**)&s.idx_alt, sizeof(unsigned int) * n);
  s.radix_bins = sort_bins(s.n_cells);
  // radix histograms, which also hold the counts of crowded digits (of 2^10
  // bins past 2^16 cells), then the per-segment sums of their scan
  s.hist_len = s.radix_bins * nsb;
  if (s.n_cells > 65536) s.hist_len = std::max(s.hist_len, (size_t)seg_count(max_points) << 10);
  alloc((void**)&s.hist, sizeof(unsigned int) * (s.hist_len + (s.radix_bins * nsb) / 8192 + 1));
  alloc((void**)&s.digit_totals, sizeof(unsigned int) * s.radix_bins);
  alloc((void**)&s.cell_start, sizeof(unsigned int) * (s.n_cells + 1));
  alloc((void**)&s.part, sizeof(float) * (size_t)s.max_cta * (s.n_entries + 1));
  alloc((void**)&s.grads, sizeof(float) * (s.n_grid + s.n_entries));
  alloc((void**)&s.flag, sizeof(unsigned int) * 4);
  if (e == cudaSuccess) e = cudaMemset(s.flag, 0, sizeof(unsigned int) * 4);  // flag[1]: Adam's block counter
  // cell keys and point indices start valid (cell 0, point 0) and are only ever
  // overwritten with valid ones, so a step whose point kernel gave up (bounded
  // wait, SRN_ERR_TIMEOUT) still sorts and gathers inside the buffers
  for (unsigned int* q : {s.key, s.key_alt, s.idx, s.idx_alt})
    if (e == cudaSuccess) e = cudaMemset(q, 0, sizeof(unsigned int) * n);
  const size_t part_bytes = sizeof(float) * s.n_cells * 8 * net.F;
  if ((size_t)max_points >= 32 * s.n_cells) {
    alloc((void**)&s.cell_part, part_bytes);
  } else if (e == cudaSuccess && part_bytes <= kMaxCellPart && cudaMalloc((void**)&s.cell_part, part_bytes) != cudaSuccess) {
    s.cell_part = nullptr;  // no room: the gradient is gathered per vertex, as for larger grids
    cudaGetLastError();
  }
  return e;
}

void fit_scratch_free(FitScratch& s) {
  void* ps[] = {s.pts, s.dz, s.key, s.key_alt, s.idx, s.idx_alt, s.hist, s.digit_totals, s.cell_start, s.part,
                s.grads, s.flag,
                s.cell_part};
  for (void* p : ps)
    if (p) cudaFree(p);
  memset(&s, 0, sizeof(s));
}

int static_sort_items() { return kSortItems; }

int sort_bins(size_t n_cells) { return n_cells <= 512 ? 512 : 256; }

bool fit_supported(const NetDev& net) {
  return net.c == 32 && (net.F == 4 || net.F == 8 || net.F == 16 || net.F == 32) && net.l <= kMaxL;
}

cudaError_t launch_backward(FitScratch& s, const NetDev& net, const float* pts, int n, float time, const float* dout,
                            float* dgrid, float* dW, float* db, cudaStream_t st) {
  if (!fit_supported(net)) return cudaErrorNotSupported;
  PointArgs pa{};
  pa.n = n;
  pa.mode = 1;
  pa.pts_in = pts;
  pa.dout_in = dout;
  pa.time = time;
  return run_backward(s, net, pa, dgrid, dW, db, nullptr, st);
}

cudaError_t launch_fit_step(FitScratch& s, const NetDev& net, const FitArgs& a, cudaStream_t st) {
  if (!fit_supported(net)) return cudaErrorNotSupported;
  PointArgs pa{};
  pa.n = a.n;
  pa.mode = 0;
  pa.seed = a.seed;
  pa.step = a.step;
  pa.time = a.time;
  pa.vol = a.vol;
  pa.gw = a.grad_weight;
  pa.gs = a.grad_scale;
  pa.cdf = a.cdf;
  pa.cdf_res = a.cdf_res;
  pa.step_ptr = a.step_ptr;
  pa.stall_test = a.stall_test;
  const size_t ng = s.n_grid, nW = net_weight_count(net), nb = net_bias_count(net);
  cudaError_t e = run_backward(s, net, pa, s.grads, s.grads + ng, s.grads + ng + nW, a.loss, st, a.status);
  if (e != cudaSuccess) return e;
  const size_t n = ng + nW + nb;
  unsigned int blocks = (unsigned int)std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 8);
  adam_kernel<<<blocks, 256, 0, st>>>(a.grid, a.weights, a.biases, s.grads, a.adam_m, a.adam_v, ng, nW, nb, a.lr_grid,
                                      a.lr_net, a.step, a.step_ptr, s.flag, a.status, a.grid_h, a.weights_h,
                                      a.grid_exp);
  return cudaGetLastError();
}

namespace {
__global__ void step_counter_kernel(int* step, int value, unsigned int* flag) {
  *step = value;
  *flag = 0u;
}
}  // namespace

cudaError_t launch_step_counter(int* step, int value, unsigned int* flag, cudaStream_t st) {
  step_counter_kernel<<<1, 1, 0, st>>>(step, value, flag);
  return cudaGetLastError();
}

}  // namespace srn
