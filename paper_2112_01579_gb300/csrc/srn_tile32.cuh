// FP32 network on tiles of 32 points per warp: the layer products as small
// register-tiled matrix products out of shared memory.
//
// A warp keeps the vectors of its 32 points in shared memory, one row of 32
// floats per vector entry (row k = input k of all points).  Work that belongs
// to a point (sampling, Fourier features, latent gather, transfer function)
// runs one lane per point; a layer runs with each lane holding 4 points x C/4
// outputs, so one input step costs 1 + C/16 16-byte shared loads for C FMAs,
// where a thread that owns a whole point (its C outputs against broadcast
// weights) needs C / 4 loads for the same C FMAs.  Activations are applied in
// the 4 x C/4 layout, so their values never need a lane of their own.  Every
// output is the bias plus its products in input order, one FMA each: the same
// bits as a thread walking the inputs alone.
#pragma once

#include "srn_net32.cuh"

namespace srn {
namespace tile32 {

using net32::Cell;
using net32::Latent;

constexpr int kPts = 32;  // points of a warp's tile

// Shared-memory image of the parameters, offsets in floats (multiples of 4).
// Layer 0's rows are in the order the inputs are produced: p, then sin and
// cos of each Fourier row, the latent vector, the time input.
struct Net {
  int d0, l, D, m, F, ti;
  int oF, oW0, ob0, oHid, hidStride, oWl, obl, total;
};

inline Net make_net(const NetDev& n) {
  Net t;
  const int C = n.c;
  t.d0 = net_d0(n); t.l = n.l; t.D = n.D; t.m = n.m; t.F = n.F; t.ti = n.ti;
  int o = 0;
  t.oF = o; o += ((3 * n.m + 3) / 4) * 4;
  t.oW0 = o; o += t.d0 * C;
  t.ob0 = o; o += C;
  t.oHid = o; t.hidStride = C * C + C;
  o += (n.l - 2) * t.hidStride;
  t.oWl = o; o += n.D * C;
  t.obl = o; o += 4;
  t.total = o;
  return t;
}

// Column of the weight matrix W_0 (inputs [p, sin, cos, z, t]) at row k of the tile.
__device__ __forceinline__ int input_column(int k, int m) {
  if (k < 3 || k >= 3 + 2 * m) return k;
  const int q = k - 3;
  return (q & 1) ? 3 + m + (q >> 1) : 3 + (q >> 1);
}

// Stages the parameters: every layer transposed to [in][out].
template <int C>
__device__ void load_net(float* sm, const Net& t, const NetDev& n) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < 3 * t.m; i += nt) sm[t.oF + i] = n.fourier[i];
  const float* W = n.W;
  for (int i = tid; i < t.d0 * C; i += nt) {
    const int k = i / C, o = i - k * C;
    sm[t.oW0 + i] = W[(size_t)o * t.d0 + input_column(k, t.m)];
  }
  for (int i = tid; i < C; i += nt) sm[t.ob0 + i] = n.b[i];
  W += (size_t)t.d0 * C;
  const float* bb = n.b + C;
  for (int h = 0; h < t.l - 2; ++h) {
    float* base = sm + t.oHid + h * t.hidStride;
    for (int i = tid; i < C * C; i += nt) {
      const int j = i / C, o = i - j * C;
      base[i] = W[o * C + j];
    }
    for (int i = tid; i < C; i += nt) base[C * C + i] = bb[i];
    W += C * C;
    bb += C;
  }
  for (int i = tid; i < t.D * C; i += nt) sm[t.oWl + i] = W[i];
  for (int i = tid; i < t.D; i += nt) sm[t.obl + i] = bb[i];
  __syncthreads();
}

// The lane's place in the 4 x C/4 layout: points 4 pg .. 4 pg + 3, outputs
// og C/4 .. (eight consecutive lanes share one output group, so their weight
// loads are one broadcast and their point loads one 128-byte row).
__device__ __forceinline__ int point_group() { return threadIdx.x & 7; }
__device__ __forceinline__ int out_group() { return (threadIdx.x >> 3) & 3; }

// acc[i][q] holds outputs (2q, 2q + 1) of the lane's output group for point i.
template <int C>
struct Acc {
  float2 v[4][C / 8];
};

template <int C>
__device__ __forceinline__ void set_bias(Acc<C>& a, const float* bias) {
  const float* b = bias + out_group() * (C / 4);
#pragma unroll
  for (int q = 0; q < C / 8; ++q) {
    const float2 bb = *reinterpret_cast<const float2*>(b + 2 * q);
#pragma unroll
    for (int i = 0; i < 4; ++i) a.v[i][q] = bb;
  }
}

// a += x W over the K rows of x (row stride S floats), W [K][C], rows ascending.
template <int C, int S>
__device__ __forceinline__ void layer(Acc<C>& a, const float* x, const float* W, int K) {
  const float* xp = x + 4 * point_group();
  const float* wp = W + out_group() * (C / 4);
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 xv = *reinterpret_cast<const float4*>(xp + k * S);
    float2 w[C / 8];
#pragma unroll
    for (int q = 0; q < C / 16; ++q) {
      const float4 w4 = *reinterpret_cast<const float4*>(wp + k * C + 4 * q);
      w[2 * q] = make_float2(w4.x, w4.y);
      w[2 * q + 1] = make_float2(w4.z, w4.w);
    }
    const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 xx = make_float2(xs[i], xs[i]);
#pragma unroll
      for (int q = 0; q < C / 8; ++q) a.v[i][q] = __ffma2_rn(w[q], xx, a.v[i][q]);
    }
  }
}

// sin and cos of two arguments (s0, c0, s1, c1): one out-of-line call for two
// independent chains.  Out of line because the accurate functions carry a
// large argument reduction; by value because pointer results go through
// local memory.
static __device__ __noinline__ float4 sincos_pair(float x0, float x1) {
  float4 r;
  sincosf(x0, &r.x, &r.y);
  sincosf(x1, &r.z, &r.w);
  return r;
}

// Activation of the lane's values in place, and its derivative.
template <int C>
__device__ __forceinline__ void activate_df(int act, Acc<C>& a, Acc<C>& d) {
  const bool snake = act == SRN_ACT_SNAKEALT;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; ++q) {
      const float2 x = a.v[i][q];
      const float4 r = sincos_pair(x.x, x.y);
      a.v[i][q] = snake ? make_float2(fmaf(0.5f, x.x, r.x * r.x), fmaf(0.5f, x.y, r.z * r.z)) : make_float2(r.x, r.z);
      d.v[i][q] = snake ? make_float2(0.5f + 2.0f * r.x * r.y, 0.5f + 2.0f * r.z * r.w) : make_float2(r.y, r.w);
    }
}

// Writes the lane's values as rows (output index) of x.
template <int C, int S>
__device__ __forceinline__ void put(const Acc<C>& a, float* x) {
  float* xp = x + (out_group() * (C / 4)) * S + 4 * point_group();
#pragma unroll
  for (int q = 0; q < C / 8; ++q) {
    *reinterpret_cast<float4*>(xp + (2 * q) * S) = make_float4(a.v[0][q].x, a.v[1][q].x, a.v[2][q].x, a.v[3][q].x);
    *reinterpret_cast<float4*>(xp + (2 * q + 1) * S) = make_float4(a.v[0][q].y, a.v[1][q].y, a.v[2][q].y, a.v[3][q].y);
  }
}

// Input rows of the lane's point p (+ pl, the low part of a position carried
// as a pair): [p, sin, cos, z, (t)].
template <int S>
__device__ __forceinline__ void put_inputs(float* x, const float* sm, const Net& t, const Latent& lat, float3 p,
                                           float3 pl = make_float3(0.f, 0.f, 0.f)) {
  float* v = x + (threadIdx.x & 31);
  v[0] = p.x;
  v[S] = p.y;
  v[2 * S] = p.z;
  const float* Fm = sm + t.oF;
  for (int k = 0; k < t.m; ++k) {
    float s, c;
    net32::fourier_sincos(Fm + 3 * k, p, s, c, pl);
    v[(3 + 2 * k) * S] = s;
    v[(4 + 2 * k) * S] = c;
  }
  const Cell cell = net32::make_cell(lat, p);
  float* z = v + (3 + 2 * t.m) * S;
  for (int f = 0; f < t.F; f += 4) {
    const float4 q = net32::latent4(lat, cell, f);
    z[f * S] = q.x;
    z[(f + 1) * S] = q.y;
    z[(f + 2) * S] = q.z;
    z[(f + 3) * S] = q.w;
  }
  if (t.ti) z[t.F * S] = lat.tin;
}

// Output dd of the lane's point from the last activation rows.
template <int C, int S>
__device__ __forceinline__ float last_layer(const float* x, const float* sm, const Net& t, int dd) {
  const float* v = x + (threadIdx.x & 31);
  const float* w = sm + t.oWl + dd * C;
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 4
  for (int o = 0; o < C; o += 4) {
    const float4 w4 = *reinterpret_cast<const float4*>(w + o);
    s0 = fmaf(w4.x, v[o * S], s0);
    s1 = fmaf(w4.y, v[(o + 1) * S], s1);
    s2 = fmaf(w4.z, v[(o + 2) * S], s2);
    s3 = fmaf(w4.w, v[(o + 3) * S], s3);
  }
  return sm[t.obl + dd] + ((s0 + s1) + (s2 + s3));
}

// acc[q][j] (points 2q, 2q + 1 of the lane; N weight rows) = sum over the C
// entries o of d (rows of S floats) of W[row j][o]: the product with the
// transposed layer, entries ascending.  row(j) gives the lane's weight rows.
template <int C, int S, int N, class Row>
__device__ __forceinline__ void back(float2 (&acc)[2][N], const float* d, const float* W, Row row) {
  const float* dp = d + 4 * point_group();
#pragma unroll
  for (int j = 0; j < N; ++j) acc[0][j] = acc[1][j] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int o = 0; o < C; o += 4) {
    float4 x[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = *reinterpret_cast<const float4*>(dp + (o + e) * S);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(W + row(j) * C + o);
      const float ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 ww = make_float2(ws[e], ws[e]);
        acc[0][j] = __ffma2_rn(make_float2(x[e].x, x[e].y), ww, acc[0][j]);
        acc[1][j] = __ffma2_rn(make_float2(x[e].z, x[e].w), ww, acc[1][j]);
      }
    }
  }
}

}  // namespace tile32
}  // namespace srn
