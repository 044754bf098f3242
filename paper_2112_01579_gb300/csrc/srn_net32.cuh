// FP32 network device code, one thread per point: the latent gather (Section
// 4.2) and the Fourier features (Eq. 1-2) that all FP32 kernels share, and the
// shared-memory staging and forward pass (Section 3 layer equation) of the fit
// point kernel for networks the tiled kernel does not take.
#pragma once

#include "srn_device.cuh"

namespace srn {
namespace net32 {

constexpr int kMaxL = 8;  // deepest network the FP32 kernels stash for the adjoint

// Shared-memory image of the network, offsets in floats (multiples of 4).
struct Layout {
  int d0, l, D, m, F, ti;
  int oF, oW0T, ob0, oHid, hidStride, oWl, obl, total;
};

inline Layout make_layout(const NetDev& n) {
  Layout L;
  const int C = n.c;
  L.d0 = net_d0(n); L.l = n.l; L.D = n.D; L.m = n.m; L.F = n.F; L.ti = n.ti;
  int o = 0;
  L.oF = o; o += ((3 * n.m + 3) / 4) * 4;
  L.oW0T = o; o += L.d0 * C;
  L.ob0 = o; o += C;
  L.oHid = o; L.hidStride = 2 * C * C + C;
  o += (n.l - 2) * L.hidStride;
  L.oWl = o; o += n.D * C;
  L.obl = o; o += 4;
  L.total = o;
  return L;
}

// Stage the FP32 parameters: W0 and hidden layers transposed ([in][out]) so a
// thread adds one input's contribution to all outputs with float4 reads; the
// last layer row-major; hidden layers also row-major for the adjoint.
template <int C>
__device__ void load_net(float* sm, const Layout& L, const NetDev& n) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < 3 * L.m; i += nt) sm[L.oF + i] = n.fourier[i];
  const float* W = n.W;
  for (int i = tid; i < L.d0 * C; i += nt) {
    int o = i / L.d0, j = i - o * L.d0;
    sm[L.oW0T + j * C + o] = W[i];
  }
  for (int i = tid; i < C; i += nt) sm[L.ob0 + i] = n.b[i];
  W += (size_t)L.d0 * C;
  const float* bb = n.b + C;
  for (int h = 0; h < L.l - 2; ++h) {
    float* base = sm + L.oHid + h * L.hidStride;
    for (int i = tid; i < C * C; i += nt) {
      int o = i / C, j = i - o * C;
      base[j * C + o] = W[i];
      base[C * C + C + i] = W[i];
    }
    for (int i = tid; i < C; i += nt) base[C * C + i] = bb[i];
    W += C * C;
    bb += C;
  }
  for (int i = tid; i < L.D * C; i += nt) sm[L.oWl + i] = W[i];
  for (int i = tid; i < L.D; i += nt) sm[L.obl + i] = bb[i];
  __syncthreads();
}

// h += a * row, two outputs per packed FP32x2 FMA (each lane a correctly
// rounded FMA, so the same bits as scalar fmaf).
template <int C>
__device__ __forceinline__ void axpy(float (&h)[C], const float* __restrict__ row, float a) {
  const float2 aa = make_float2(a, a);
#pragma unroll
  for (int o = 0; o < C; o += 4) {
    const float4 w = *reinterpret_cast<const float4*>(row + o);
    const float2 r0 = __ffma2_rn(make_float2(w.x, w.y), aa, make_float2(h[o], h[o + 1]));
    const float2 r1 = __ffma2_rn(make_float2(w.z, w.w), aa, make_float2(h[o + 2], h[o + 3]));
    h[o] = r0.x;
    h[o + 1] = r0.y;
    h[o + 2] = r1.x;
    h[o + 3] = r1.y;
  }
}

template <int C>
__device__ __forceinline__ float dotrow(const float* __restrict__ row, const float (&a)[C]) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
  for (int o = 0; o < C; o += 4) {
    float4 w = *reinterpret_cast<const float4*>(row + o);
    s0 = fmaf(w.x, a[o], s0);
    s1 = fmaf(w.y, a[o + 1], s1);
    s2 = fmaf(w.z, a[o + 2], s2);
    s3 = fmaf(w.w, a[o + 3], s3);
  }
  return (s0 + s1) + (s2 + s3);
}

// Eq. 3 SnakeAlt(x) = 0.5 x + sin^2 x, or sin(x); and the derivatives.
// Out-of-line sin / cos: the accurate functions carry a large argument-
// reduction path, and inlined once per hidden unit of the unrolled layers
// they overflow the instruction cache (the fit kernel stalled mostly on
// instruction fetch).
static __device__ __noinline__ void sincos_call(float x, float* s, float* c) { sincosf(x, s, c); }
static __device__ __noinline__ float sin_call(float x) { return sinf(x); }

__device__ __forceinline__ float act_f(int act, float x) {
  float s = sin_call(x);
  return act == SRN_ACT_SNAKEALT ? fmaf(0.5f, x, s * s) : s;
}
// Activation value and derivative from one sin/cos evaluation.
__device__ __forceinline__ void act_and_df(int act, float x, float& a, float& d) {
  float s, c;
  sincos_call(x, &s, &c);
  if (act == SRN_ACT_SNAKEALT) {
    a = fmaf(0.5f, x, s * s);
    d = 0.5f + 2.0f * s * c;
  } else {
    a = s;
    d = c;
  }
}
// Latent grid source of one frame: z = tw0 G_k0(p) + tw1 G_k0+1(p).
struct Latent {
  const float* g0;
  const float* g1;
  float tw0, tw1;
  float tin;  // time value (the extra input of the direct time encoding)
  int R, F;
};

__device__ __forceinline__ Latent make_latent(const NetDev& n, float t) {
  int k0;
  float f;
  time_weights(n, t, k0, f);
  size_t gsz = (size_t)n.R * n.R * n.R * n.F;
  Latent L;
  L.g0 = n.grid + (size_t)k0 * gsz;
  L.g1 = n.nkey > 1 ? L.g0 + gsz : nullptr;
  L.tw0 = n.nkey > 1 ? 1.0f - f : 1.0f;
  L.tw1 = f;
  L.tin = t;
  L.R = n.R;
  L.F = n.F;
  return L;
}

struct Cell {
  int base, sx, sy, sz;   // element offsets of vertex (ix,iy,iz) and of +x, +y, +z
  float fx, fy, fz;
};

__device__ __forceinline__ Cell make_cell(const Latent& lat, float3 p) {
  Cell c;
  int ix, iy, iz;
  cell_coord(p.x, lat.R, ix, c.fx);
  cell_coord(p.y, lat.R, iy, c.fy);
  cell_coord(p.z, lat.R, iz, c.fz);
  c.sx = lat.F;
  c.sy = lat.R * lat.F;
  c.sz = lat.R * lat.R * lat.F;
  c.base = iz * c.sz + iy * c.sy + ix * c.sx;
  return c;
}

// Channels f..f+3 of the latent vector (trilinear, time-blended).
__device__ __forceinline__ float4 latent4(const Latent& lat, const Cell& c, int f) {
  float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    float w = (dx ? c.fx : 1.0f - c.fx) * (dy ? c.fy : 1.0f - c.fy) * (dz ? c.fz : 1.0f - c.fz);
    int off = c.base + dx * c.sx + dy * c.sy + dz * c.sz + f;
    float4 g = __ldg(reinterpret_cast<const float4*>(lat.g0 + off));
    float w0 = w * lat.tw0;
    z.x = fmaf(w0, g.x, z.x); z.y = fmaf(w0, g.y, z.y); z.z = fmaf(w0, g.z, z.z); z.w = fmaf(w0, g.w, z.w);
    if (lat.g1) {
      float4 h = __ldg(reinterpret_cast<const float4*>(lat.g1 + off));
      float w1 = w * lat.tw1;
      z.x = fmaf(w1, h.x, z.x); z.y = fmaf(w1, h.y, z.y); z.z = fmaf(w1, h.z, z.z); z.w = fmaf(w1, h.w, z.w);
    }
  }
  return z;
}

// sin and cos of the Fourier argument e = F_k . p (Eq. 2) with e carried to
// about twice FP32 precision: each product split exactly into hi + lo by an
// FMA, the three products summed with error-free two-sums, then
// sin(hi + lo) = sin hi + lo cos hi and cos(hi + lo) = cos hi - lo sin hi.
// A plain FP32 dot product would lose |e| * 2^-24 of the argument, which for
// the high NeRF octaves (|e| in the thousands) dominates the error; the
// rounded-to-nearest intrinsics keep the compiler from contracting the steps.
// pl is the low part of a position carried as a pair p + pl (the render's
// sample positions); F_k . pl joins the low part of the argument.
__device__ __forceinline__ void fourier_sincos(const float* f, float3 p, float& s, float& c,
                                               float3 pl = make_float3(0.f, 0.f, 0.f)) {
  const float p0 = __fmul_rn(f[0], p.x), e0 = fmaf(f[0], p.x, -p0);
  const float p1 = __fmul_rn(f[1], p.y), e1 = fmaf(f[1], p.y, -p1);
  const float p2 = __fmul_rn(f[2], p.z), e2 = fmaf(f[2], p.z, -p2);
  const float s1 = __fadd_rn(p0, p1);
  const float b1 = __fsub_rn(s1, p0);
  const float t1 = __fadd_rn(__fsub_rn(p0, __fsub_rn(s1, b1)), __fsub_rn(p1, b1));
  const float hi = __fadd_rn(s1, p2);
  const float b2 = __fsub_rn(hi, s1);
  const float t2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(hi, b2)), __fsub_rn(p2, b2));
  const float lo = e0 + e1 + e2 + t1 + t2 + (f[0] * pl.x + f[1] * pl.y + f[2] * pl.z);
  float sh, ch;
  sincosf(hi, &sh, &ch);
  s = fmaf(ch, lo, sh);
  c = fmaf(-sh, lo, ch);
}

// Full forward pass at p.  out[0..D-1]; hs[i] receives the pre-activation of
// layer i (i = 0..l-2) for the backward.
template <int C>
__device__ __forceinline__ void forward(const float* sm, const Layout& L, int act, const Latent& lat, float3 p,
                                        float (&out)[4], float (*hs)[C]) {
  float h[C];
  const float* W0T = sm + L.oW0T;
#pragma unroll
  for (int o = 0; o < C; ++o) h[o] = sm[L.ob0 + o];
  axpy<C>(h, W0T, p.x);
  axpy<C>(h, W0T + C, p.y);
  axpy<C>(h, W0T + 2 * C, p.z);
  const float* Fm = sm + L.oF;
  for (int k = 0; k < L.m; ++k) {
    float s, c;
    fourier_sincos(Fm + 3 * k, p, s, c);
    axpy<C>(h, W0T + (3 + k) * C, s);
    axpy<C>(h, W0T + (3 + L.m + k) * C, c);
  }
  Cell cell = make_cell(lat, p);
  for (int f = 0; f < L.F; f += 4) {
    float4 z = latent4(lat, cell, f);
    const float* r = W0T + (3 + 2 * L.m + f) * C;
    axpy<C>(h, r, z.x);
    axpy<C>(h, r + C, z.y);
    axpy<C>(h, r + 2 * C, z.z);
    axpy<C>(h, r + 3 * C, z.w);
  }
  if (L.ti) axpy<C>(h, W0T + (3 + 2 * L.m + L.F) * C, lat.tin);  // Section 7 "direct" time input
  for (int i = 1; i < L.l - 1; ++i) {
    const float* base = sm + L.oHid + (i - 1) * L.hidStride;
    float a[C];
#pragma unroll
    for (int o = 0; o < C; ++o) {
      hs[i - 1][o] = h[o];
      a[o] = act_f(act, h[o]);
    }
#pragma unroll
    for (int o = 0; o < C; ++o) h[o] = base[C * C + o];
#pragma unroll
    for (int j = 0; j < C; ++j) axpy<C>(h, base + j * C, a[j]);
  }
  float a[C];
#pragma unroll
  for (int o = 0; o < C; ++o) {
    hs[L.l - 2][o] = h[o];
    a[o] = act_f(act, h[o]);
  }
#pragma unroll
  for (int d = 0; d < 4; ++d)
    out[d] = d < L.D ? sm[L.obl + d] + dotrow<C>(sm + L.oWl + d * C, a) : 0.0f;
}

__device__ __forceinline__ float3 clamp_p(float3 p) { return make_float3(clamp01f(p.x), clamp01f(p.y), clamp01f(p.z)); }

}  // namespace net32
}  // namespace srn
