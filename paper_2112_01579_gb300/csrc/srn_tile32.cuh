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
//
// Measured against one thread per point with out-of-line library sines: error
// grid of 128^3 x 8 evaluations of the main configuration 5.68 -> 3.06 ms
// (5.4 G evaluations/s; bound by the pipe that takes packed FMAs and the
// shared-memory data pipe together), the plain workload's 128^2 frame 968 ->
// 202 us (with several samples of a ray per pass).
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
  int rows;   // rows of 32 floats that a warp keeps of its inputs
  bool wide;  // more inputs than that: see put_block
};

// Networks of more than kWideIn inputs run layer 0 in blocks of rows, so that
// a warp's tile leaves room for others (rows for 235 inputs: six warps an SM).
// 300,000 points of 4 layers of 32, with all rows -> in blocks (a thread per
// point): 155 inputs 276 -> 207 us (277), 255 inputs 472 -> 270 (364), 8 layers
// of 64 and 255 inputs 1480 -> 680 (1776); a 400 x 300 frame of those 24.4 ->
// 7.3 ms (13.4).  At 127 inputs and less there is nothing to gain.  A gradient
// evaluates its Fourier rows twice that way; at width 32, where they are the
// larger part, that pays later (169 inputs 412 -> 495 us, 255 842 -> 705).
constexpr int kWideIn = 128, kWideInGradient32 = 192;
constexpr int kBlockFeatures = 32, kBlockChannels = 64;  // Fourier rows, latent channels of a block
constexpr int kBlockLow = 3 + 2 * kBlockFeatures + 1;    // first of three rows that keep the positions' low parts
constexpr int kBlockRows = kBlockLow + 3;

inline Net make_net(const NetDev& n, bool gradient = false) {
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
  t.wide = t.d0 > (gradient && C == 32 ? kWideInGradient32 : kWideIn);
  t.rows = t.wide ? kBlockRows : t.d0;
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
#pragma unroll 8  // loads in flight: a call of few points waits for these
  for (int i = tid; i < t.d0 * C; i += nt) {
    const int k = i / C, o = i - k * C;
    sm[t.oW0 + i] = W[(size_t)o * t.d0 + input_column(k, t.m)];
  }
  for (int i = tid; i < C; i += nt) sm[t.ob0 + i] = n.b[i];
  W += (size_t)t.d0 * C;
  const float* bb = n.b + C;
  for (int h = 0; h < t.l - 2; ++h) {
    float* base = sm + t.oHid + h * t.hidStride;
#pragma unroll 8
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

// ---- inline sine / cosine of the tile paths
// Reduction by Cody and Waite (Software Manual for the Elementary Functions,
// 1980) in FMA form, then minimax polynomials from a Remez exchange on the
// absolute error, each coefficient rounded to FP32 before the next was
// fitted: sin r on |r| <= 1.0005 pi/2 to 5.0e-9; on
// |r| <= 1.001 pi/4 sin to 1.9e-9 and cos to 1.1e-10 (before FP32 arithmetic rounds, about
// 6e-8).  They cost a third of the issue slots of the accurate library
// calls, which stay for arguments beyond kActMax and for Fourier matrices
// that are not powers of two.
constexpr float kActMax = 1.0e4f;  // below: rint(x / pi) is off by less than 2e-4, inside the fitted range

__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }

// r = x - k pi with k = rint(x / pi) (pi as FP32 hi + lo); t's lowest bit is k's parity.
__device__ __forceinline__ float2 reduce_pi(float2 x, float2& t) {
  const float kMagic = 12582912.0f;  // 1.5 2^23
  t = __ffma2_rn(x, f2(0.318309886183790672f), f2(kMagic));
  const float2 k = __fadd2_rn(t, f2(-kMagic));
  const float2 r = __ffma2_rn(k, f2(-3.14159274101257324f), x);
  return __ffma2_rn(k, f2(8.74227765734758577e-8f), r);
}
__device__ __forceinline__ float2 sin_half(float2 r, float2 z) {
  float2 p = __ffma2_rn(z, f2(2.59889998e-06f), f2(-0.000198060457f));
  p = __ffma2_rn(z, p, f2(0.00833300874f));
  p = __ffma2_rn(z, p, f2(-0.166666567f));
  return __ffma2_rn(__fmul2_rn(r, z), p, r);
}
// cos r = sin(pi / 2 - |r|): a polynomial in r would lose the relative
// precision near the cosine's zero.
__device__ __forceinline__ float2 cos_half(float2 r) {
  const float2 a = make_float2(fabsf(r.x), fabsf(r.y));
  const float2 h = __fadd2_rn(__ffma2_rn(a, f2(-1.0f), f2(1.57079637050628662f)), f2(-4.37113883e-8f));
  return sin_half(h, __fmul2_rn(h, h));
}
// cos x to 1.7e-8 rms (correctly rounded 1.5e-8, the library's 2.0e-8): the
// derivative of the sine networks.  cos_half has 2.7e-8, from two roundings on
// top of its reduction's, and made their gradients 2 to 3 % less exact than
// the library's cosine.  Quarter turns, |r| <= pi / 4, and 1 - z / 2 with its
// rounding error kept.
__device__ __forceinline__ float2 cos_turn(float2 x) {
  const float kMagic = 12582912.0f;  // 1.5 2^23
  const float2 t = __ffma2_rn(x, f2(0.636619772367581343f), f2(kMagic));
  const float2 q = __fadd2_rn(t, f2(-kMagic));
  const float2 r = __ffma2_rn(q, f2(4.37113883e-8f), __ffma2_rn(q, f2(-1.57079637050628662f), x));
  const float2 z = __fmul2_rn(r, r);
  float2 p = __ffma2_rn(z, f2(-0.000194957684f), f2(0.00833198149f));
  p = __ffma2_rn(z, p, f2(-0.166666508f));
  const float2 s = __ffma2_rn(__fmul2_rn(r, z), p, r);
  p = __ffma2_rn(z, f2(2.44306702e-05f), f2(-0.00138873013f));
  p = __ffma2_rn(z, p, f2(0.0416666456f));
  const float2 w = __ffma2_rn(z, f2(-0.5f), f2(1.0f));
  const float2 e = __ffma2_rn(z, f2(-0.5f), __ffma2_rn(w, f2(-1.0f), f2(1.0f)));
  const float2 c = __fadd2_rn(w, __ffma2_rn(__fmul2_rn(z, z), p, e));
  const int a = __float_as_int(t.x), b = __float_as_int(t.y);
  return make_float2(__int_as_float(__float_as_int((a & 1) ? s.x : c.x) ^ (((a + 1) & 2) << 30)),
                     __int_as_float(__float_as_int((b & 1) ? s.y : c.y) ^ (((b + 1) & 2) << 30)));
}
__device__ __forceinline__ float flip(float v, float t) {  // v (-1)^k
  return __int_as_float(__float_as_int(v) ^ (__float_as_int(t) << 31));
}

// sin and cos of 2^j w p, w the FP32 value of 2 pi, from X = 2^j p (exact)
// plus `lo` radians: in quarter turns, q = rint(4 X), f = X - q / 4 (exact),
// w X = 2 pi X + e X with e = w - 2 pi, so modulo 2 pi the angle is
// q pi / 2 + w f + e q / 4.
__device__ __forceinline__ void turn_sincos(float X, float lo, float& s, float& c) {
  const float kMagic = 12582912.0f;
  const float t = fmaf(X, 4.0f, kMagic);
  const float q4 = t - kMagic;
  const float f = fmaf(q4, -0.25f, X);
  const float r = fmaf(6.28318548202514648f, f, fmaf(4.37113900e-8f, q4, lo));
  const float z = r * r;
  float p = fmaf(z, -0.000194957684f, 0.00833198149f);
  p = fmaf(z, p, -0.166666508f);
  const float sr = fmaf(r * z, p, r);
  p = fmaf(z, 2.44306702e-05f, -0.00138873013f);
  p = fmaf(z, p, 0.0416666456f);
  const float cr = fmaf(z * z, p, fmaf(z, -0.5f, 1.0f));
  const int q = __float_as_int(t);
  const float a = (q & 1) ? cr : sr, b = (q & 1) ? sr : cr;
  s = __int_as_float(__float_as_int(a) ^ ((q & 2) << 30));
  c = __int_as_float(__float_as_int(b) ^ (((q + 1) & 2) << 30));
}
constexpr int kTurnRows = 30;  // octaves 0..9: |e X| stays below 1e-4

// Whether F's row k is w 2^(k div 3) on axis k mod 3 (block-wide answer).
__device__ __forceinline__ bool nerf_rows(const float* F, int m) {
  bool ok = m <= kTurnRows;
  for (int i = threadIdx.x; ok && i < 3 * m; i += blockDim.x) {
    const int k = i / 3, a = i - 3 * k;
    ok = F[i] == (a == k % 3 ? 6.28318548202514648f * (float)(1 << (k / 3)) : 0.0f);
  }
  return __syncthreads_and(ok) != 0;
}

// Activation values of four arguments, and their derivatives.
struct Quad {
  float4 a, d;
};
__device__ __forceinline__ Quad act_quad(float4 x, bool snake) {
  Quad r;
  if (!(fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))) <= kActMax)) {
    const float4 p = sincos_pair(x.x, x.y), q = sincos_pair(x.z, x.w);
    if (snake) {
      r.a = make_float4(fmaf(0.5f, x.x, p.x * p.x), fmaf(0.5f, x.y, p.z * p.z), fmaf(0.5f, x.z, q.x * q.x),
                        fmaf(0.5f, x.w, q.z * q.z));
      r.d = make_float4(0.5f + 2.0f * p.x * p.y, 0.5f + 2.0f * p.z * p.w, 0.5f + 2.0f * q.x * q.y,
                        0.5f + 2.0f * q.z * q.w);
    } else {
      r.a = make_float4(p.x, p.z, q.x, q.z);
      r.d = make_float4(p.y, p.w, q.y, q.w);
    }
    return r;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 v = h ? make_float2(x.z, x.w) : make_float2(x.x, x.y);
    float2 t, a, d;
    const float2 e = reduce_pi(v, t), z = __fmul2_rn(e, e), s = sin_half(e, z);
    if (snake) {  // sin^2 and sin cos do not change with k
      a = __ffma2_rn(s, s, __fmul2_rn(v, f2(0.5f)));
      d = __ffma2_rn(__fadd2_rn(s, s), cos_half(e), f2(0.5f));
    } else {
      a = make_float2(flip(s.x, t.x), flip(s.y, t.y));
      d = cos_turn(v);
    }
    if (h) r.a.z = a.x, r.a.w = a.y, r.d.z = d.x, r.d.w = d.y;
    else r.a.x = a.x, r.a.y = a.y, r.d.x = d.x, r.d.y = d.y;
  }
  return r;
}
// Out of line: a kernel that activates several unrolled layers would not fit
// the instruction cache with the code inlined at every value.
template <bool SNAKE>
__device__ __noinline__ Quad act_quad_call(float4 x) {
  return act_quad(x, SNAKE);
}

// Activation and derivative of the lane's values by act_quad_call.
template <int C, bool SNAKE>
__device__ __forceinline__ void activate_call(Acc<C>& a, Acc<C>& d) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; q += 2) {
      const Quad r = act_quad_call<SNAKE>(make_float4(a.v[i][q].x, a.v[i][q].y, a.v[i][q + 1].x, a.v[i][q + 1].y));
      a.v[i][q] = make_float2(r.a.x, r.a.y);
      a.v[i][q + 1] = make_float2(r.a.z, r.a.w);
      d.v[i][q] = make_float2(r.d.x, r.d.y);
      d.v[i][q + 1] = make_float2(r.d.z, r.d.w);
    }
}

// Activation of the lane's values in place; DF: and its derivative.
template <int C, bool DF>
__device__ __forceinline__ void activate(int act, Acc<C>& a, Acc<C>* d) {
  const bool snake = act == SRN_ACT_SNAKEALT;
  float big = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; ++q) big = fmaxf(big, fmaxf(fabsf(a.v[i][q].x), fabsf(a.v[i][q].y)));
  if (__any_sync(0xffffffffu, !(big <= kActMax))) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < C / 8; ++q) {
        const float2 x = a.v[i][q];
        const float4 r = sincos_pair(x.x, x.y);
        a.v[i][q] = snake ? make_float2(fmaf(0.5f, x.x, r.x * r.x), fmaf(0.5f, x.y, r.z * r.z)) : make_float2(r.x, r.z);
        if (DF) d->v[i][q] = snake ? make_float2(0.5f + 2.0f * r.x * r.y, 0.5f + 2.0f * r.z * r.w) : make_float2(r.y, r.w);
      }
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; ++q) {
      const float2 x = a.v[i][q];
      float2 t;
      const float2 r = reduce_pi(x, t), z = __fmul2_rn(r, r);
      const float2 s = sin_half(r, z);
      if (snake) {  // sin^2 and sin cos do not change with k
        a.v[i][q] = __ffma2_rn(s, s, __fmul2_rn(x, f2(0.5f)));
        if (DF) d->v[i][q] = __ffma2_rn(__fadd2_rn(s, s), cos_half(r), f2(0.5f));
      } else {
        a.v[i][q] = make_float2(flip(s.x, t.x), flip(s.y, t.y));
        if (DF) d->v[i][q] = cos_turn(x);
      }
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

// Channels f0 .. f0 + N - 1 of the latent vector at p as rows of z; all 8 N / 4
// loads (twice that with two keyframes) can be in flight at once.
template <int S, int N>
__device__ __forceinline__ void put_latent(float* z, const Latent& lat, float3 p, int f0 = 0) {
  const Cell cell = net32::make_cell(lat, p);
  float4 q[N / 4];
#pragma unroll
  for (int f = 0; f < N / 4; ++f) q[f] = net32::latent4(lat, cell, f0 + 4 * f);
#pragma unroll
  for (int f = 0; f < N / 4; ++f) {
    z[(4 * f) * S] = q[f].x;
    z[(4 * f + 1) * S] = q[f].y;
    z[(4 * f + 2) * S] = q[f].z;
    z[(4 * f + 3) * S] = q[f].w;
  }
}

// Input rows of the lane's point p (+ pl, the low part of a position carried
// as a pair): [p, sin, cos, z, (t)].
// NeRF Fourier rows (nerf) take the inline quarter-turn form.  The latent
// gather of the usual channel counts goes first, so that its loads are in
// flight during the features (error grid 3.41 -> 3.37 ms).
template <int S>
__device__ __forceinline__ void put_inputs(float* x, const float* sm, const Net& t, const Latent& lat, bool nerf,
                                           float3 p, float3 pl = make_float3(0.f, 0.f, 0.f)) {
  float* v = x + (threadIdx.x & 31);
  float* z = v + (3 + 2 * t.m) * S;
  if (t.F == 16) put_latent<S, 16>(z, lat, p);
  else if (t.F == 8) put_latent<S, 8>(z, lat, p);
  v[0] = p.x;
  v[S] = p.y;
  v[2 * S] = p.z;
  const float* Fm = sm + t.oF;
  if (nerf) {
    float w = 1.0f;
    for (int k = 0; k < t.m; k += 3, w += w) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (k + a < t.m) {
          const float pa = a == 0 ? p.x : (a == 1 ? p.y : p.z), la = a == 0 ? pl.x : (a == 1 ? pl.y : pl.z);
          float s, c;
          turn_sincos(w * pa, 6.28318548202514648f * (w * la), s, c);
          v[(3 + 2 * (k + a)) * S] = s;
          v[(4 + 2 * (k + a)) * S] = c;
        }
      }
    }
  } else {
    for (int k = 0; k < t.m; ++k) {
      float s, c;
      net32::fourier_sincos(Fm + 3 * k, p, s, c, pl);
      v[(3 + 2 * k) * S] = s;
      v[(4 + 2 * k) * S] = c;
    }
  }
  if (t.F != 16 && t.F != 8) {  // sixteen channels a pass: 300,000 points with 64 of them 324 -> 247 us
    int f = 0;
    for (; f + 16 <= t.F; f += 16) put_latent<S, 16>(z + f * S, lat, p, f);
    for (; f < t.F; f += 4) put_latent<S, 4>(z + f * S, lat, p, f);
  }
  if (t.ti) z[t.F * S] = lat.tin;
}

// sin and cos of Fourier row k at p + pl.
__device__ __forceinline__ void feature(const float* Fm, int k, bool nerf, float3 p, float3 pl, float& s, float& c) {
  if (nerf) {
    const float w = (float)(1 << (k / 3));
    const int a = k % 3;
    const float pa = a == 0 ? p.x : (a == 1 ? p.y : p.z), la = a == 0 ? pl.x : (a == 1 ? pl.y : pl.z);
    turn_sincos(w * pa, 6.28318548202514648f * (w * la), s, c);
  } else {
    net32::fourier_sincos(Fm + 3 * k, p, s, c, pl);
  }
}

// The input rows of a wide network from `row` on, as many as a block holds, in
// the lane's column v; returns how many.  The values are those of put_inputs.
// Out of line, arguments by value, like all of the wide path: the others keep
// their registers.
static __device__ __noinline__ int put_block(float* v, const float* Fm, int m, int F, int ti, bool nerf,
                                             const Latent lat, float3 p, float3 pl, int row) {
  constexpr int S = kPts;
  int n = 0;
  if (row < 3 + 2 * m) {
    if (row == 0) {
      v[0] = p.x;
      v[S] = p.y;
      v[2 * S] = p.z;
      v[kBlockLow * S] = pl.x;
      v[(kBlockLow + 1) * S] = pl.y;
      v[(kBlockLow + 2) * S] = pl.z;
      n = 3;
    }
    const int k0 = row == 0 ? 0 : (row - 3) / 2, k1 = min(m, k0 + kBlockFeatures);
#pragma unroll 2
    for (int k = k0; k < k1; ++k, n += 2) {
      float s, c;
      feature(Fm, k, nerf, p, pl, s, c);
      v[n * S] = s;
      v[(n + 1) * S] = c;
    }
    return n;
  }
  const int f0 = row - 3 - 2 * m, f1 = min(F, f0 + kBlockChannels);
  for (; f0 + n + 16 <= f1; n += 16) put_latent<S, 16>(v + n * S, lat, p, f0 + n);
  for (; f0 + n < f1; n += 4) put_latent<S, 4>(v + n * S, lat, p, f0 + n);
  if (f1 == F && ti) v[n++ * S] = lat.tin;
  return n;
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

// Outputs of one point (the same p in all lanes) by the accurate functions,
// the whole warp on it: a lane per Fourier row, latent channel and output
// neuron, so one point takes about a microsecond; the products in the order
// of the tile passes.  x: 112 floats of scratch.  Out of line and with its
// arguments by value: it is for rare use, and the caller keeps its registers.
static __device__ __noinline__ float4 accurate_point(const float* sm, const Net t, int act, const Latent lat, float3 p,
                                                     float* x) {
  constexpr int C = 32;
  const int lane = threadIdx.x & 31;
  __syncwarp();
  if (lane < 3) x[lane] = lane == 0 ? p.x : (lane == 1 ? p.y : p.z);
  for (int k = lane; k < t.m; k += 32) {
    float s, c;
    net32::fourier_sincos(sm + t.oF + 3 * k, p, s, c);
    x[3 + 2 * k] = s;
    x[4 + 2 * k] = c;
  }
  const Cell cell = net32::make_cell(lat, p);
  for (int f = 4 * lane; f < t.F; f += 128) {
    const float4 q = net32::latent4(lat, cell, f);
    float* z = x + 3 + 2 * t.m + f;
    z[0] = q.x;
    z[1] = q.y;
    z[2] = q.z;
    z[3] = q.w;
  }
  if (t.ti && lane == 0) x[3 + 2 * t.m + t.F] = lat.tin;
  __syncwarp();
  const float* W = sm + t.oW0;
  const float* in = x;
  float h = sm[t.ob0 + lane];
  int K = t.d0;
  for (int layer = 1;; ++layer) {
#pragma unroll 8
    for (int k = 0; k < K; ++k) h = fmaf(W[k * C + lane], in[k], h);
    const float s = sinf(h);
    float* next = x + 48 + (layer & 1) * C;
    next[lane] = act == SRN_ACT_SNAKEALT ? fmaf(0.5f, h, s * s) : s;
    __syncwarp();
    in = next;
    if (layer == t.l - 1) break;
    W = sm + t.oHid + (layer - 1) * t.hidStride;
    h = W[C * C + lane];
    K = C;
  }
  // lane 4 d + r: the r-th of the four interleaved sums of output d
  float sum = 0.f;
  const int d = lane >> 2, r = lane & 3;
  if (d < t.D)
    for (int o = r; o < C; o += 4) sum = fmaf(sm[t.oWl + d * C + o], in[o], sum);
  float out[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float s0 = __shfl_sync(0xffffffffu, sum, 4 * k), s1 = __shfl_sync(0xffffffffu, sum, 4 * k + 1),
                s2 = __shfl_sync(0xffffffffu, sum, 4 * k + 2), s3 = __shfl_sync(0xffffffffu, sum, 4 * k + 3);
    out[k] = k < t.D ? sm[t.obl + k] + ((s0 + s1) + (s2 + s3)) : 0.f;
  }
  __syncwarp();
  return make_float4(out[0], out[1], out[2], out[3]);
}

// acc[q][j] (points 2q, 2q + 1 of the lane; N weight rows) = sum over the C
// entries o of d (rows of S floats) of W[row j][o]: the product with the
// transposed layer, in PARTS sums of C / PARTS consecutive entries.  row(j)
// gives the lane's weight rows.
template <int C, int S, int N, int PARTS = 1, class Row>
__device__ __forceinline__ void back(float2 (&acc)[2][N], const float* d, const float* W, Row row) {
  const float* dp = d + 4 * point_group();
#pragma unroll
  for (int j = 0; j < N; ++j) acc[0][j] = acc[1][j] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int part = 0; part < PARTS; ++part) {
    float2 s[2][N];
#pragma unroll
    for (int j = 0; j < N; ++j) s[0][j] = s[1][j] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int o = part * (C / PARTS); o < (part + 1) * (C / PARTS); o += 4) {
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
          s[0][j] = __ffma2_rn(make_float2(x[e].x, x[e].y), ww, s[0][j]);
          s[1][j] = __ffma2_rn(make_float2(x[e].z, x[e].w), ww, s[1][j]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
      acc[0][j] = PARTS == 1 ? s[0][j] : __fadd2_rn(acc[0][j], s[0][j]);
      acc[1][j] = PARTS == 1 ? s[1][j] : __fadd2_rn(acc[1][j], s[1][j]);
    }
  }
}

// ---- whole passes of a warp's 32 points
struct Ctx {
  const float* sm;
  const Net* t;
  int act;
  bool nerf;
};

// Forward pass of the lanes' points: the last activations end up as rows of
// x (read them with last_layer; a __syncwarp must follow before the rows are
// overwritten).  v0: the input rows (may be x itself).  DF: df[h] receives
// the derivative of activation h.  WIDE: for the networks put_block is for, in
// kernels of their own (the branch alone cost the error grid 2.5 %).
template <int C, bool DF, bool WIDE>
__device__ __forceinline__ void forward(const Ctx& c, float* v0, float* x, const Latent& lat, float3 p, float3 pl,
                                        Acc<C>* df) {
  constexpr int S = kPts;
  const Net& t = *c.t;
  Acc<C> a;
  if constexpr (WIDE) {
    set_bias<C>(a, c.sm + t.ob0);
    for (int row = 0; row < t.d0;) {
      const int n = put_block(v0 + (threadIdx.x & 31), c.sm + t.oF, t.m, t.F, t.ti, c.nerf, lat, p, pl, row);
      __syncwarp();
      layer<C, S>(a, v0, c.sm + t.oW0 + row * C, n);
      row += n;
      __syncwarp();
    }
  } else {
    put_inputs<S>(v0, c.sm, t, lat, c.nerf, p, pl);
    __syncwarp();
    set_bias<C>(a, c.sm + t.ob0);
    layer<C, S>(a, v0, c.sm + t.oW0, t.d0);
  }
#pragma unroll 1
  for (int h = 1; h < t.l - 1; ++h) {
    activate<C, DF>(c.act, a, DF ? df + (h - 1) : nullptr);
    __syncwarp();
    put<C, S>(a, x);
    __syncwarp();
    const float* W = c.sm + t.oHid + (h - 1) * t.hidStride;
    set_bias<C>(a, W + C * C);
    layer<C, S>(a, x, W, C);
  }
  activate<C, DF>(c.act, a, DF ? df + (t.l - 2) : nullptr);
  __syncwarp();
  put<C, S>(a, x);
  __syncwarp();
}

// The lane's seed sum_d s_d W_last[d][o] from D rows of output adjoints (row
// stride kPts), or W_last's row 0 (rows == nullptr).
template <int C>
__device__ __forceinline__ void seed(Acc<C>& a, const float* sm, const Net& t, const float* rows) {
  const float* w = sm + t.oWl + out_group() * (C / 4);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; ++q)
      a.v[i][q] = rows ? make_float2(0.f, 0.f) : *reinterpret_cast<const float2*>(w + 2 * q);
  if (!rows) return;
  for (int d = 0; d < t.D; ++d) {
    const float4 dv = *reinterpret_cast<const float4*>(rows + d * kPts + 4 * point_group());
    const float ds[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
    for (int q = 0; q < C / 8; ++q) {
      const float2 wq = *reinterpret_cast<const float2*>(w + d * C + 2 * q);
#pragma unroll
      for (int i = 0; i < 4; ++i) a.v[i][q] = __ffma2_rn(wq, f2(ds[i]), a.v[i][q]);
    }
  }
}

// l += gradient with respect to the cell coordinates of sum_f g_f z_f over N
// channels from f0 (g_f in rows of z): per corner the product of g with the
// corner's values, times the derivative of its weight.
template <int S, int N>
__device__ __forceinline__ void latent_vjp(float3& l, const float* z, const Latent& lat, const Cell& c, int f0) {
  float g[N];
#pragma unroll
  for (int f = 0; f < N; ++f) g[f] = z[f * S];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    const float wx = dx ? c.fx : 1.0f - c.fx, wy = dy ? c.fy : 1.0f - c.fy, wz = dz ? c.fz : 1.0f - c.fz;
    const int at = c.base + dx * c.sx + dy * c.sy + dz * c.sz + f0;
    float dot = 0.f;
#pragma unroll
    for (int f = 0; f < N; f += 4) {
      float4 v = __ldg(reinterpret_cast<const float4*>(lat.g0 + at + f));
      if (lat.g1) {
        const float4 h = __ldg(reinterpret_cast<const float4*>(lat.g1 + at + f));
        v = make_float4(lat.tw0 * v.x + lat.tw1 * h.x, lat.tw0 * v.y + lat.tw1 * h.y, lat.tw0 * v.z + lat.tw1 * h.z,
                        lat.tw0 * v.w + lat.tw1 * h.w);
      }
      dot = fmaf(g[f], v.x, dot);
      dot = fmaf(g[f + 1], v.y, dot);
      dot = fmaf(g[f + 2], v.z, dot);
      dot = fmaf(g[f + 3], v.w, dot);
    }
    l.x = fmaf(dot, (dx ? wy : -wy) * wz, l.x);
    l.y = fmaf(dot, wx * (dy ? wz : -wz), l.y);
    l.z = fmaf(dot, wx * (dz ? wy : -wy), l.z);
  }
}

// The second half of input_gradient for a wide network: Fourier rows and
// latent channels in blocks, the features evaluated again.  Rows 0 to 2 of v0
// hold the products of the position rows, x the adjoint rows.
template <int C>
__device__ __noinline__ float3 wide_gradient(const float* W0, const float* Fm, int m, int F, bool nerf, float* v0,
                                             const float* x, const Latent lat, float3 p) {
  constexpr int S = kPts;
  const int pg = point_group(), og = out_group(), lane = threadIdx.x & 31;
  __syncwarp();
  float3 r = make_float3(v0[lane], v0[S + lane], v0[2 * S + lane]);
  const float3 pl = make_float3(v0[kBlockLow * S + lane], v0[(kBlockLow + 1) * S + lane], v0[(kBlockLow + 2) * S + lane]);
  for (int k0 = 0; k0 < m; k0 += kBlockFeatures) {
    const int k1 = min(m, k0 + kBlockFeatures);
    __syncwarp();
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
      float s, c;
      feature(Fm, k, nerf, p, pl, s, c);
      v0[2 * (k - k0) * S + lane] = s;
      v0[(2 * (k - k0) + 1) * S + lane] = c;
    }
    __syncwarp();
    for (int kb = k0; kb < k1; kb += 16) {  // four Fourier rows a lane
      float2 g[2][8];
      back<C, S, 8, 4>(g, x, W0, [&](int q) { return 3 + 2 * min(kb + 4 * og + (q >> 1), m - 1) + (q & 1); });
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = kb + 4 * og + e;
        if (k < k1) {
          float4* row = reinterpret_cast<float4*>(v0 + 2 * (k - k0) * S + 4 * pg);
          const float4 s4 = *row, c4 = *reinterpret_cast<const float4*>(v0 + (2 * (k - k0) + 1) * S + 4 * pg);
          const float2 s01 = g[0][2 * e], c01 = g[0][2 * e + 1], s23 = g[1][2 * e], c23 = g[1][2 * e + 1];
          *row = make_float4(s01.x * c4.x - c01.x * s4.x, s01.y * c4.y - c01.y * s4.y, s23.x * c4.z - c23.x * s4.z,
                             s23.y * c4.w - c23.y * s4.w);
        }
      }
    }
    __syncwarp();
    for (int k = k0; k < k1; ++k) {
      const float coef = v0[2 * (k - k0) * S + lane];
      r.x = fmaf(coef, Fm[3 * k], r.x);
      r.y = fmaf(coef, Fm[3 * k + 1], r.y);
      r.z = fmaf(coef, Fm[3 * k + 2], r.z);
    }
  }
  const Cell cell = net32::make_cell(lat, p);
  float3 l = make_float3(0.f, 0.f, 0.f);
  for (int f0 = 0; f0 < F; f0 += kBlockChannels) {
    const int f1 = min(F, f0 + kBlockChannels);
    __syncwarp();
    for (int fb = f0; fb < f1; fb += 32) {  // eight channels a lane
      float2 g[2][8];
      const int f = fb + 8 * og;
      back<C, S, 8, 4>(g, x, W0 + (3 + 2 * m) * C, [&](int q) { return min(f + q, F - 1); });
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (f + q < f1)
          *reinterpret_cast<float4*>(v0 + (f - f0 + q) * S + 4 * pg) = make_float4(g[0][q].x, g[0][q].y, g[1][q].x, g[1][q].y);
    }
    __syncwarp();
    int f = f0;
    for (; f + 16 <= f1; f += 16) latent_vjp<S, 16>(l, v0 + (f - f0) * S + lane, lat, cell, f);
    for (; f < f1; f += 4) latent_vjp<S, 4>(l, v0 + (f - f0) * S + lane, lat, cell, f);
  }
  __syncwarp();
  const float scale = (float)(lat.R - 1);
  return make_float3(fmaf(scale, l.x, r.x), fmaf(scale, l.y, r.y), fmaf(scale, l.z, r.z));
}

// Input gradient of the lane's point (Section 5 "Adjoint") from the seed in
// the tile layout: backward through the hidden layers, then the position,
// Fourier and latent inputs.  v0 holds the input rows of the forward (all but
// the cosines are overwritten), x is scratch of C rows, df the derivatives.
template <int C, bool WIDE>
__device__ __forceinline__ float3 input_gradient(const Ctx& c, float* v0, float* x, const Latent& lat, float3 p,
                                                 Acc<C>& a, const Acc<C>* df) {
  constexpr int S = kPts;
  const Net& t = *c.t;
  const int pg = point_group(), og = out_group(), lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < C / 8; ++q) a.v[i][q] = __fmul2_rn(a.v[i][q], df[t.l - 2].v[i][q]);
  __syncwarp();
  put<C, S>(a, x);
  __syncwarp();
#pragma unroll 1
  for (int h = t.l - 2; h >= 1; --h) {
    float2 g[2][C / 4];
    back<C, S, C / 4>(g, x, c.sm + t.oHid + (h - 1) * t.hidStride, [&](int q) { return og * (C / 4) + q; });
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < C / 8; ++q) {
        const float2 lo = g[i >> 1][2 * q], hi = g[i >> 1][2 * q + 1];
        a.v[i][q] = __fmul2_rn((i & 1) ? make_float2(lo.y, hi.y) : make_float2(lo.x, hi.x), df[h - 1].v[i][q]);
      }
    __syncwarp();
    put<C, S>(a, x);
    __syncwarp();
  }
  // layer 0: the lane takes its share of the input rows for its four points;
  // the results go back to the rows, where each point's lane adds them up (a
  // Fourier row's product with its frequency and the sum in one rounding,
  // which the sums of four lanes did not: 1 to 6 % of a gradient's error)
  const float* W0 = c.sm + t.oW0;
  {
    float2 g[2][1];
    const int r = og < 3 ? og : 2;
    back<C, S, 1, 4>(g, x, W0, [&](int) { return r; });
    if (og < 3) *reinterpret_cast<float4*>(v0 + og * S + 4 * pg) = make_float4(g[0][0].x, g[0][0].y, g[1][0].x, g[1][0].y);
  }
  if constexpr (WIDE) {
    return wide_gradient<C>(W0, c.sm + t.oF, t.m, t.F, c.nerf, v0, x, lat, p);
  } else {
#pragma unroll 1
    for (int kb = 0; kb < t.m; kb += 8) {
      const int ka[2] = {min(kb + og, t.m - 1), min(kb + og + 4, t.m - 1)};
      float2 g[2][4];
      back<C, S, 4, 4>(g, x, W0, [&](int q) { return 3 + 2 * ka[q >> 1] + (q & 1); });
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (kb + og + 4 * e < t.m) {
          const int k = ka[e];
          const float4 s4 = *reinterpret_cast<const float4*>(v0 + (3 + 2 * k) * S + 4 * pg);
          const float4 c4 = *reinterpret_cast<const float4*>(v0 + (4 + 2 * k) * S + 4 * pg);
          const float2 s01 = g[0][2 * e], c01 = g[0][2 * e + 1], s23 = g[1][2 * e], c23 = g[1][2 * e + 1];
          *reinterpret_cast<float4*>(v0 + (3 + 2 * k) * S + 4 * pg) =
              make_float4(s01.x * c4.x - c01.x * s4.x, s01.y * c4.y - c01.y * s4.y, s23.x * c4.z - c23.x * s4.z,
                          s23.y * c4.w - c23.y * s4.w);
        }
      }
    }
#pragma unroll 1
    for (int fb = 0; fb < t.F; fb += 16) {
      float2 g[2][4];
      const int f0 = fb + 4 * og;
      back<C, S, 4, 4>(g, x, W0 + (3 + 2 * t.m) * C, [&](int q) { return min(f0 + q, t.F - 1); });
      if (f0 < t.F) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(v0 + (3 + 2 * t.m + f0 + q) * S + 4 * pg) =
              make_float4(g[0][q].x, g[0][q].y, g[1][q].x, g[1][q].y);
      }
    }
    __syncwarp();
    float3 r = make_float3(v0[lane], v0[S + lane], v0[2 * S + lane]);
    const float* Fm = c.sm + t.oF;
#pragma unroll 2
    for (int k = 0; k < t.m; ++k) {
      const float coef = v0[(3 + 2 * k) * S + lane];
      r.x = fmaf(coef, Fm[3 * k], r.x);
      r.y = fmaf(coef, Fm[3 * k + 1], r.y);
      r.z = fmaf(coef, Fm[3 * k + 2], r.z);
    }
    const float* z = v0 + (3 + 2 * t.m) * S + lane;
    const Cell cell = net32::make_cell(lat, p);
    float3 l = make_float3(0.f, 0.f, 0.f);
    if (t.F == 16) {
      latent_vjp<S, 16>(l, z, lat, cell, 0);
    } else {
      int f = 0;
      for (; f + 16 <= t.F; f += 16) latent_vjp<S, 16>(l, z + f * S, lat, cell, f);
      for (; f < t.F; f += 4) latent_vjp<S, 4>(l, z + f * S, lat, cell, f);
    }
    const float scale = (float)(lat.R - 1);
    r = make_float3(fmaf(scale, l.x, r.x), fmaf(scale, l.y, r.y), fmaf(scale, l.z, r.z));
    __syncwarp();
    return r;
  }
}

// Warps per CTA of a tile kernel over `tiles` tiles (0: not known).  One CTA
// of 16 warps (8 at widths 48 and 64: what registers allow an SM) where that
// many tiles per SM wait, so that the parameters are in shared memory once and
// the rest stays L1 for the gathers (error grid of 128^3 x 8: 3.37 -> 3.09
// ms).  Fewer tiles: one CTA per SM that holds its share, so that every tile
// is in the first wave (CTAs of 4, of which shared memory held three per SM,
// left a second wave nearly empty: 60,000 points of the main network 31.3 -> 26.6
// us, with gradient 57.5 -> 45.1 us); not under 4 warps, which then
// spread over as many SMs as there are tiles for.  Less where the parameters
// and `rows` rows of 32 floats per warp pass the 227 KB a CTA may have, of
// which the kernel's own static shared memory is a part.
constexpr int max_warps(int C) { return C == 32 ? 16 : 8; }
constexpr int max_dynamic(int static_bytes) { return 227 * 1024 - static_bytes; }
// Lets kernel k have as much shared memory as there is.  Not what the call at
// hand needs: that follows the number of points, and a second host thread
// with a smaller call of the same network would lower the limit between this
// thread's setting and its launch, which is then refused.
template <class K>
cudaError_t allow_dynamic(K k, int static_bytes = 0) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dynamic(static_bytes));
}
inline int warps_for(const Net& t, int C, int rows, long long tiles, int sms, int static_bytes = 0) {
  const long long share = (tiles + sms - 1) / sms;
  int w = share >= max_warps(C) ? max_warps(C) : (share > 4 ? (int)share : 4);
  while (w > 1 && sizeof(float) * ((size_t)t.total + (size_t)w * rows * kPts) > (size_t)max_dynamic(static_bytes)) --w;
  return w;
}

}  // namespace tile32
}  // namespace srn
