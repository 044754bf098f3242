// FP16 tensor-core fV-SRN render for sm_103a: tcgen05.mma with TMEM
// accumulators, persistent CTAs, one thread per ray.
//
// Design (GB300-first restatement of the fused TensorCore network of
// Section 4.1):
// * A CTA holds 7 (6 with finite-difference shading), 4 or 3 warpgroups for
//   hidden width 32, 48 or 64 (what registers allow: 72, 128 and 168 a
//   thread; one more warpgroup at widths 48 and 64 spills and is 3 % slower).
//   Each warpgroup owns a tile of 128 rays, one per thread; thread i of the
//   warpgroup is row i of the MMA operand A and TMEM lane i of the
//   accumulator, so the per-ray work (ray stepping,
//   latent-grid trilinear fetch, Fourier features, transfer function,
//   compositing, early termination) stays one thread per ray as in the paper,
//   while the layers run as M=128 x N=C tensor-core MMAs.
// * Every sample: the thread writes its FP16 layer-0 input row into tensor
//   memory (operand A of the MMA, see tmem_st8); one elected thread
//   issues tcgen05.mma
//   (kind::f16, FP32 accumulate in TMEM); the thread reads its row back with
//   tcgen05.ld, applies the activation in FP32 and writes it into the same
//   columns as the next layer's A row as an FP16 hi + lo pair (a = hi + lo to
//   ~2^-22 relative; the B tile holds [W | W]), so the hidden activations
//   keep FP32 accuracy through the FP16 tensor cores.  Inside the tile the input columns are
//   [sin_0, cos_0, ..., sin_{m-1}, cos_{m-1}, p, z, 1, 1]; the B tile of
//   layer 0 is permuted to match, so the arithmetic is that of [p, sin, cos,
//   z].  Biases ride in the MMA as an FP16 hi + lo pair against two
//   constant-1 columns (layer 0: columns of its own row; hidden layers: one
//   extra K=16 MMA against a constant tile), which keeps them FP32-exact.  The last layer
//   (C -> D) runs on the CUDA cores in FP32.
// * SnakeAlt(x) = 0.5 x + sin^2 x = (x - cos 2x + 1) / 2 (Eq. 3).  Every MMA
//   layer is staged to produce u = 2x (weights and bias doubled, which is
//   exact in FP16), the epilogue hands a = u / 2 - cos u = 2 SnakeAlt(x) - 1
//   to the next layer, and the factor 1/2 and the shift 1/2 are folded into
//   that layer's weights and bias: the doubled next layer then simply uses W
//   and 2b + sum_j W_j (width 32: -a and -W, see act_fold).
// * Rays are claimed dynamically from a work counter, a warp at a time: when
//   every lane's ray has terminated (box exit or opacity >= threshold), the
//   warp takes the next 8 x 4 pixel tile.  The lanes then march neighbouring
//   rays in step, so their latent-grid gathers mostly hit the same cells and
//   the L1 serves a warp's loads in few wavefronts (per-lane refill, which
//   keeps every lane busy but scatters the lanes over the volume, was 10 %
//   slower on the main configuration's frame).
// * Every mbarrier wait is bounded; on timeout the warpgroup stops, records
//   SRN_ERR_TIMEOUT in the status word and the CTA frees its TMEM.
// * A non-finite network output (an input or activation beyond the FP16
//   range, 65504) is recorded as SRN_ERR_NONFINITE.
#pragma once
#include <string.h>

#include <type_traits>

#include "srn_device.cuh"
#include "srn_mma.h"

namespace srn {
namespace mma {

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(a), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase: gives up after kWaitCycles.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t a, uint32_t parity) {
  if (mbar_try_wait(a, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(a, parity)) {
    if (clock64() - t0 > kWaitCycles) return false;
  }
  return true;
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ bool bar_red_or(int id, int n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred q, p;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, %2, %3, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (FP16 inputs, FP32 accumulate).
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The same with A in tensor memory (lane = row, two FP16 of K per column).
__device__ __forceinline__ void mma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
               : "memory");
}

// Thread's TMEM lane, 32 consecutive FP32 columns, waited for.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row atoms
// 1024 bytes apart (SBO), sm100 descriptor version 1.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;              // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024u >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1u << 46;              // descriptor version
  d |= (uint64_t)2u << 61;              // SWIZZLE_128B
  return d;
}

// A descriptor moved by `bytes` (a multiple of 16; addresses stay below 2^18).
__device__ __forceinline__ uint64_t desc_at(uint64_t d, uint32_t bytes) { return d + (uint64_t)(bytes >> 4); }

// Instruction descriptor: kind::f16, A = B = FP16, D = FP32, both K-major,
// M = 128, N = the layer's output width.
constexpr uint32_t idesc_n(int N) { return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24); }

// Byte offset of 16-byte chunk j of row r in a 128B-swizzled tile.
__device__ __forceinline__ uint32_t sw_off(int r, int j) { return (uint32_t)(r * 128 + ((j ^ (r & 7)) << 4)); }

__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
  __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// FP16 hi + lo split of a pair: hi = fp16(a), lo = fp16(a - hi).  The
// residual a - hi is exact in FP32; it is formed by one mixed-precision FMA
// per element (hi in FP16 times the FP16 constant -1, plus a in FP32), so
// neither widening nor negating hi costs an instruction.
__device__ __forceinline__ void split_h2(float a0, float a1, uint32_t& hi, uint32_t& lo) {
  hi = pack_h2(a0, a1);
  float r0, r1;
  asm("{.reg .b16 x, y, m;\n\t"
      "mov.b32 {x, y}, %2;\n\t"
      "mov.b16 m, 0xBC00;\n\t"
      "fma.rn.f32.f16 %0, x, m, %3;\n\t"
      "fma.rn.f32.f16 %1, y, m, %4;}"
      : "=f"(r0), "=f"(r1)
      : "r"(hi), "f"(a0), "f"(a1));
  lo = pack_h2(r0, r1);
}

// Activation values handed to the next layer from two accumulator values:
// sin(x) for the sine network; for SnakeAlt the accumulator holds u = 2x and
// the value is u / 2 - cos u = 2 SnakeAlt(x) - 1, or its negative with NEG
// (the next layer's weights then carry the minus sign), which with PACK is one
// packed FMA for two.  Width 32 takes NEG; at width 48 the schedule it led to
// was 1 % slower.
template <int ACT, bool PACK, bool NEG>
__device__ __forceinline__ float2 act_fold(float x, float y) {
  if (ACT != SRN_ACT_SNAKEALT) return make_float2(__sinf(x), __sinf(y));
  if (PACK) return __ffma2_rn(make_float2(x, y), make_float2(-0.5f, -0.5f), make_float2(__cosf(x), __cosf(y)));
  if (!NEG) return make_float2(fmaf(0.5f, x, -__cosf(x)), fmaf(0.5f, y, -__cosf(y)));
  return make_float2(fmaf(-0.5f, x, __cosf(x)), fmaf(-0.5f, y, __cosf(y)));
}

// Byte offset of 16-byte chunk cg (= column / 8) of row r in a tile of
// 128B-swizzled 128-row K-atoms (the fit kernel's operand tiles).
__device__ __forceinline__ uint32_t sw_tile_off(int r, int cg) {
  return (uint32_t)((cg >> 3) * kTile) + sw_off(r, cg & 7);
}

// The per-ray operand rows (layer inputs, activations, adjoint rows) live in
// tensor memory: row = lane, two FP16 of K per 32-bit column.  A thread
// stores its own row with tcgen05.st, eight columns (16 FP16) at a time, so a
// row takes four stores instead of eight 16-byte shared-memory stores (and
// the proxy fence they need before the MMA), and the MMA leaves the L1 /
// shared-memory pipe to the latent gathers.  The same bits as operand rows in
// shared memory, and faster on every variant: main configuration at 1024^2
// 10.61 -> 9.81 ms, four keyframed 517 x 333 frames 7.69 -> 7.12 ms, adjoint
// shading at 512^2 20.0 -> 18.4 ms, six layers of 48 channels at 512^2 3.91 ->
// 3.57 ms, 2^20 points 96 -> 82 us.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&w)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

struct RayLat {
  int g0, g1;     // element offsets of the bracketing keyframe grids (g1 < 0: single grid)
  float w0, w1;   // time weights
  float tin;      // time value (input of the direct time encoding)
};

// Latent vector (Section 4.2 trilinear latent grid; Section 7 time blend)
// from the FP16 grid, accumulated in FP32.  Each corner's weight is rounded
// to FP16 and the products taken by mixed-precision FMAs (FP16 weight times
// FP16 grid value, exact, plus the FP32 sum): one instruction per channel
// and corner instead of a widening and an FMA.  The weight rounding (2^-11
// relative) moves z_c by at most 2^-11 sum_k w_k |G_kc|, about as much as the
// FP16 rounding of z itself for the A tile.
// ST: one latent grid (no keyframes), known at compile time: no time blend.
// WIDE: 32-byte loads (grid rows of 32 bytes, aligned), for points that do not
// share cells: a warp's lanes then hit 32 lines whatever the load's width, and
// the L1 takes a wavefront per line and load (2^20 random points 70.0 -> 61.6
// us; rays of one tile share cells, where the width makes no difference).
template <int F, int ST, bool WIDE = false>
__device__ __forceinline__ void latent_h(const __half* __restrict__ G, int R, const RayLat& rl, float3 p,
                                         float (&z)[F]) {
  int ix, iy, iz;
  float fx, fy, fz;
  cell_coord(p.x, R, ix, fx);
  cell_coord(p.y, R, iy, fy);
  cell_coord(p.z, R, iz, fz);
  const int sx = F, sy = R * F, sz = R * R * F;
  const int base = iz * sz + iy * sy + ix * sx;
#pragma unroll
  for (int f = 0; f < F; ++f) z[f] = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    const float w = (dx ? fx : 1.0f - fx) * (dy ? fy : 1.0f - fy) * (dz ? fz : 1.0f - fz);
    const int off = base + dx * sx + dy * sy + dz * sz;
#pragma unroll
    for (int kk = 0; kk < (ST ? 1 : 2); ++kk) {
      const int g = ST ? 0 : (kk ? rl.g1 : rl.g0);
      if (!ST && kk && g < 0) break;
      const __half wh = __float2half_rn(ST ? w : w * (kk ? rl.w1 : rl.w0));
      const uint16_t wb = *reinterpret_cast<const uint16_t*>(&wh);
      uint4 wide[2];
      if constexpr (WIDE) ldg32(G + g + off, wide[0], wide[1]);
#pragma unroll
      for (int c = 0; c < F; c += 8) {
        const uint4 q = WIDE ? wide[(c / 8) & 1] : __ldg(reinterpret_cast<const uint4*>(G + g + off + c));
        const uint32_t qq[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          asm("{.reg .b16 x, y, w;\n\t"
              "mov.b32 {x, y}, %2;\n\t"
              "mov.b16 w, %3;\n\t"
              "fma.rn.f32.f16 %0, x, w, %0;\n\t"
              "fma.rn.f32.f16 %1, y, w, %1;}"
              : "+f"(z[c + 2 * e]), "+f"(z[c + 2 * e + 1])
              : "r"(qq[e]), "h"(wb));
        }
      }
    }
  }
}

// Latent vector from the 8-bit grid (Section 4.2: per-channel codes, value
// lo + step * code).  F = 16 codes of a vertex are one 16-byte load; each
// byte is spliced into the FP16 value 1024 + code and 1152 subtracted in
// FP16, both exact, giving the centred code c - 128.  As in latent_h the
// corner weight is rounded to FP16 and sum_k w_k (c_k - 128) accumulated by
// mixed-precision FMAs; since the weights sum to 1,
// z = (lo + 128 step) + step * sum_k w_k (c_k - 128), with lo + 128 step
// staged per channel in qp[2 f].  The weight rounding moves z by at most
// 2^-11 step sum_k w_k |c_k - 128| (half the channel's range, at most).
template <int F, int ST>
__device__ __forceinline__ void latent_q(const uint8_t* __restrict__ Q, const float* qp, int R, const RayLat& rl,
                                         float3 p, float (&z)[F]) {
  static_assert(F == 16, "one 16-byte load per vertex");
  int ix, iy, iz;
  float fx, fy, fz;
  cell_coord(p.x, R, ix, fx);
  cell_coord(p.y, R, iy, fy);
  cell_coord(p.z, R, iz, fz);
  const int sx = F, sy = R * F, sz = R * R * F;
  const int base = iz * sz + iy * sy + ix * sx;
  const __half2 k1152 = __float2half2_rn(1152.0f);
#pragma unroll
  for (int f = 0; f < F; ++f) z[f] = 0.0f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    const float w = (dx ? fx : 1.0f - fx) * (dy ? fy : 1.0f - fy) * (dz ? fz : 1.0f - fz);
    const int off = base + dx * sx + dy * sy + dz * sz;
#pragma unroll
    for (int kk = 0; kk < (ST ? 1 : 2); ++kk) {
      const int g = ST ? 0 : (kk ? rl.g1 : rl.g0);
      if (!ST && kk && g < 0) break;
      const __half wh = __float2half_rn(ST ? w : w * (kk ? rl.w1 : rl.w0));
      const uint16_t wb = *reinterpret_cast<const uint16_t*>(&wh);
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(Q + g + off));
      const uint32_t words[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t lo2 = __byte_perm(words[e], 0x64646464u, 0x4140u);
        uint32_t hi2 = __byte_perm(words[e], 0x64646464u, 0x4342u);
        const __half2 a2 = __hsub2(*reinterpret_cast<const __half2*>(&lo2), k1152);
        const __half2 b2 = __hsub2(*reinterpret_cast<const __half2*>(&hi2), k1152);
        const uint32_t au = *reinterpret_cast<const uint32_t*>(&a2), bu = *reinterpret_cast<const uint32_t*>(&b2);
        asm("{.reg .b16 x, y, w;\n\t"
            "mov.b32 {x, y}, %4;\n\t"
            "mov.b16 w, %6;\n\t"
            "fma.rn.f32.f16 %0, x, w, %0;\n\t"
            "fma.rn.f32.f16 %1, y, w, %1;\n\t"
            "mov.b32 {x, y}, %5;\n\t"
            "fma.rn.f32.f16 %2, x, w, %2;\n\t"
            "fma.rn.f32.f16 %3, y, w, %3;}"
            : "+f"(z[4 * e]), "+f"(z[4 * e + 1]), "+f"(z[4 * e + 2]), "+f"(z[4 * e + 3])
            : "r"(au), "r"(bu), "h"(wb));
      }
    }
  }
#pragma unroll
  for (int f = 0; f < F; ++f) z[f] = fmaf(qp[2 * f + 1], z[f], qp[2 * f]);
}

// Layer-0 input row (Eq. 1-2 features, Section 4.2 latent vector, Section 7
// time input when TI) in the tile's column order [sin_0, cos_0, ...,
// sin_{m-1}, cos_{m-1}, p, z, (t), 1, 1, 0...] over the K0 columns layer 0
// reads.  Values are packed to FP16 pairs
// and stored to the thread's TMEM row 16 at a time as they are produced; the
// whole warp takes part (tcgen05.st is warp-collective), lanes without a
// sample write a row nothing reads.  SCATTERED: points of no common cell.
template <int M, int F, int K0, int TI, int GQ, int ST, bool SCATTERED>
__device__ __forceinline__ void write_input_row(uint32_t t_a, float3 p, bool nerf, const float* fm,
                                                const __half* G, const uint8_t* Q, const float* qp, int R,
                                                const RayLat& rl) {
  constexpr int D0 = 3 + 2 * M + F + TI;
  static_assert(M >= 3, "the NeRF recurrence needs the three base rows");
  float z[F];
  if constexpr (GQ != 0) {
    latent_q<F, ST>(Q, qp, R, rl, p, z);
  } else if constexpr (SCATTERED && F == 16) {
    if (aligned32(G)) latent_h<F, ST, true>(G, R, rl, p, z);
    else latent_h<F, ST>(G, R, rl, p, z);
  } else {
    latent_h<F, ST>(G, R, rl, p, z);
  }
  uint32_t w[8];
  int nw = 0, col = 0;
  auto emit = [&](float a, float b) {
    w[nw++] = pack_h2(a, b);
    if (nw == 8) {
      tmem_st8(t_a + col, w);
      col += 8;
      nw = 0;
    }
  };
  if (nerf) {
    // NeRF rows are 2^j w along axis k mod 3 (octave j = k div 3, w the
    // stored FP32 value of 2 pi): one sin/cos per axis, then angle doubling
    // sin 2t = 2 s c, cos 2t = 1 - 2 s^2 (three instructions; the FMA form's
    // absolute error, about 2^-23, is far below the FP16 rounding of the
    // features for the A tile, 2^-12).  Doubling doubles the error of
    // the base angle, so with more than five octaves the base is recomputed
    // every fourth octave from the reduced argument: with x = 2^j p_a and
    // r = round(x) (both exact in FP32), 2^j w p_a = w (x - r) + (w - 2 pi) r
    // modulo 2 pi.
    constexpr int kReseed = M > 15 ? 4 : 64;
    constexpr float kW = 6.28318548202514648f;         // FP32 2 pi
    constexpr float kWErr = 1.74845560252379070e-7f;    // FP32 2 pi - 2 pi
    float s[3], c[3];
#pragma unroll
    for (int k = 0; k < M; ++k) {
      const int a = k % 3, j = k / 3;
      const float pa = a == 0 ? p.x : (a == 1 ? p.y : p.z);
      if (j % kReseed == 0) {
        const float x = pa * (float)(1 << j);
        const float r = rintf(x);
        __sincosf(fmaf(kW, x - r, kWErr * r), &s[a], &c[a]);
      } else {
        const float ss = s[a], cc = c[a], t2 = ss + ss;
        s[a] = t2 * cc;
        c[a] = fmaf(-t2, ss, 1.0f);
      }
      emit(s[a], c[a]);
    }
  } else {
#pragma unroll
    for (int k = 0; k < M; ++k) {
      const float e = fm[3 * k] * p.x + fm[3 * k + 1] * p.y + fm[3 * k + 2] * p.z;
      float sv, cv;
      sincosf(e, &sv, &cv);
      emit(sv, cv);
    }
  }
  // remaining columns 2M .. K0-1: p, z, the two bias ones, zeros
  float tail[K0 - 2 * M];
#pragma unroll
  for (int i = 0; i < K0 - 2 * M; ++i) {
    const int cc = 2 * M + i;
    float v = 0.0f;
    if (cc < 2 * M + 3) v = cc == 2 * M ? p.x : (cc == 2 * M + 1 ? p.y : p.z);
    else if (cc < 2 * M + 3 + F) v = z[cc - 2 * M - 3];
    else if (cc < D0) v = rl.tin;  // Section 7 "direct" time input
    else if (cc == D0 || cc == D0 + 1) v = 1.0f;
    tail[i] = v;
  }
#pragma unroll
  for (int i = 0; i < K0 - 2 * M; i += 2) emit(tail[i], tail[i + 1]);
}

// ---------------------------------------------------------------- kernel
// Thread's TMEM lane, 16 consecutive FP32 columns, waited for.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Thread's TMEM lane, C consecutive FP32 columns (C a multiple of 16).
template <int C>
__device__ __forceinline__ void tmem_ld_row(uint32_t taddr, float (&v)[C]) {
#pragma unroll
  for (int c = 0; c + 32 <= C; c += 32) tmem_ld32(taddr + c, *reinterpret_cast<float(*)[32]>(v + c));
  if constexpr (C % 32 != 0) tmem_ld16(taddr + (C - 16), v + (C - 16));
}

// Thread's TMEM lane, 32 consecutive FP32 columns written, store waited for.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n\t"
      "tcgen05.wait::st.sync.aligned;"
      ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]),
        "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]),
        "f"(v[16]), "f"(v[17]), "f"(v[18]), "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]),
        "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]), "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
      : "memory");
}

// Thread's TMEM lane, 16 consecutive FP32 columns written, store waited for.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};\n\t"
      "tcgen05.wait::st.sync.aligned;"
      ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]),
        "f"(v[8]), "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}

// Thread's TMEM lane, C consecutive FP32 columns written (C a multiple of 16).
template <int C>
__device__ __forceinline__ void tmem_st_row(uint32_t taddr, const float (&v)[C]) {
#pragma unroll
  for (int c = 0; c + 32 <= C; c += 32) tmem_st32(taddr + c, *reinterpret_cast<const float(*)[32]>(v + c));
  if constexpr (C % 32 != 0) tmem_st16(taddr + (C - 16), v + (C - 16));
}

// Gradient with respect to p of sum_c gz[c] z_c(p), z the latent vector
// (trilinear in p inside the cell chosen by cell_coord, time-blended):
// sum over corners and keyframes of w_time (gz . g_corner) grad w_corner(p),
// with d f / d p = R - 1 per axis.
template <int F, int ST>
__device__ __forceinline__ float3 latent_grad_h(const __half* __restrict__ G, int R, const RayLat& rl, float3 p,
                                                const float* gz) {
  int ix, iy, iz;
  float fx, fy, fz;
  cell_coord(p.x, R, ix, fx);
  cell_coord(p.y, R, iy, fy);
  cell_coord(p.z, R, iz, fz);
  const int sx = F, sy = R * F, sz = R * R * F;
  const int base = iz * sz + iy * sy + ix * sx;
  float3 g = make_float3(0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    const float wx = dx ? fx : 1.0f - fx, wy = dy ? fy : 1.0f - fy, wz = dz ? fz : 1.0f - fz;
    const int off = base + dx * sx + dy * sy + dz * sz;
#pragma unroll
    for (int kk = 0; kk < (ST ? 1 : 2); ++kk) {
      const int gb = ST ? 0 : (kk ? rl.g1 : rl.g0);
      if (!ST && kk && gb < 0) break;
      float dot = 0.0f;
#pragma unroll
      for (int c = 0; c < F; c += 8) {
        uint4 q = __ldg(reinterpret_cast<const uint4*>(G + gb + off + c));
        const __half2* h = reinterpret_cast<const __half2*>(&q);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 v = __half22float2(h[e]);
          dot = fmaf(gz[c + 2 * e], v.x, dot);
          dot = fmaf(gz[c + 2 * e + 1], v.y, dot);
        }
      }
      if (!ST) dot *= kk ? rl.w1 : rl.w0;
      g.x = fmaf(dot, (dx ? wy : -wy) * wz, g.x);
      g.y = fmaf(dot, wx * (dy ? wz : -wz), g.y);
      g.z = fmaf(dot, wx * (dz ? wy : -wy), g.z);
    }
  }
  const float s = (float)(R - 1);
  return make_float3(s * g.x, s * g.y, s * g.z);
}

template <int C, int M, int F, int ACT, int SH, int TI, int GQ, int LF, int ST>
__global__ void __launch_bounds__(128 * wgs_for(C, SH), 1)
    render_mma_kernel(const NetDev net, const std::conditional_t<is_points(SH), PointsBatch, BatchDev> b, const PointsDev pd, const SmemPlan plan,
                      unsigned long long* __restrict__ ray_counter, unsigned int* __restrict__ status) {
  constexpr int WGS = wgs_for(C, SH), THREADS = 128 * WGS;
  constexpr int D0 = 3 + 2 * M + F + TI;
  constexpr int K0 = ((D0 + 2 + 15) / 16) * 16;  // inputs + two bias columns
  constexpr int NAH = (2 * C + 63) / 64;         // K-atoms of a hidden layer's B tile
  constexpr int BT = C * 128;                    // bytes of one K-atom of a B tile (C rows)
  constexpr uint32_t IDESC = idesc_n(C);
  static_assert(C % 16 == 0 && C <= 64 && K0 <= 128, "shape outside the kernel's tiling");
  constexpr int NP = SH == SRN_SHADE_FD ? 7 : 1;  // network passes per sample
  constexpr bool POINTS = is_points(SH);
  constexpr bool SNAKE = ACT == SRN_ACT_SNAKEALT;
  constexpr bool ADJ = is_adjoint(SH);  // input gradient by backward MMAs (Section 5 "adjoint")
  constexpr int TMC = kTmemCols;
  constexpr int NACC = adj_acc_cols(C, K0);  // adjoint: accumulator columns before the derivative stash
  static_assert(!ADJ || (TI == 0 && GQ == 0), "tensor-core adjoint: no time input, FP16 grid");
  static_assert(WGS * tmem_wg_cols(C, SH, K0) <= TMC, "TMEM layout exceeds the allocation");

  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* B0 = sm + plan.oB0;
  uint8_t* Bh = sm + plan.oBh;
  uint8_t* Bb = sm + plan.oBb;
  uint8_t* BhT = sm + plan.oBhT;
  uint8_t* B0T = sm + plan.oB0T;
  float* wl = reinterpret_cast<float*>(sm + plan.oWl);
  TFSeg& tf = *reinterpret_cast<TFSeg*>(sm + plan.oTF);
  float* fm = reinterpret_cast<float*>(sm + plan.oFm);
  float* qp = reinterpret_cast<float*>(sm + plan.oQp);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + plan.oMbar);
  volatile int* misc = reinterpret_cast<volatile int*>(sm + plan.oMisc);  // [0] tmem base, [4+wg] fail

  const int tid = threadIdx.x;
  // the warp's index by a broadcast is known to be uniform, so addresses made
  // from it stay in uniform registers: 3 % of a frame; point evaluation is
  // 12 % slower that way (81 against 72 us for 2^20 points)
  const int warp_id = POINTS ? tid >> 5 : __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int wg = warp_id >> 2, row = tid & 127, lane = tid & 31;
  const bool issuer = (warp_id & 3) == 0;  // the warp whose elected lane issues its warpgroup's MMAs
  // LF > 0: a network of LF layers and D = 1 output (4 for the gradient
  // head), both fixed at compile time (the layer loop unrolls, the output
  // loop has its exact trip count); the dispatch picks such an instantiation
  // only for such a network
  constexpr int DF = SH == SRN_SHADE_HEAD ? 4 : 1;
  // The activations and the last layer in packed FMAs (two channels each)
  // where that was faster: the single-grid width-32 march without shading or
  // with the adjoint gradient (main configuration, 1024^2: 8.61 -> 8.37 ms;
  // 512^2 shaded, with the packed products of the backward below: 13.68 ->
  // 12.94 ms).  Elsewhere the register pairs cost as much as they save or
  // more: keyframes 6.30 -> 6.38 ms, width 48 2.89 -> 2.91.
  constexpr bool PACK = ST == 1 && C == 32 && (SH == SRN_SHADE_NONE || SH == SRN_SHADE_ADJOINT);
  // The last layer as a sum over the even and one over the odd channels with
  // 16-byte weight loads, the same at width 32 with and without PACK (every
  // march of a network gives the same bits); keyframes 6.30 -> 6.25 ms.  One
  // sum at widths 48 and 64 (the other form: 2.89 -> 2.93 ms) and for points
  // with gradient (166 -> 170 us for 2^20).
  constexpr bool SUM2 = C == 32 && SH != kPointsAdj;
  constexpr bool NEG = C == 32;  // see act_fold
  const int L = LF > 0 ? LF : net.l;
  const int D = LF > 0 ? DF : net.D;
  // the FP16 latent grid holds G 2^-gexp: the latent columns' layer-0 weights
  // are staged times 2^gexp (exact), the 8-bit grid's lo / step times 2^-gexp
  const int gexp = net.grid_exp ? *net.grid_exp : 0;
  const float gscale = __int_as_float((127 + gexp) << 23);  // 2^gexp, gexp <= 113

  // ---- stage parameters as FP16 B tiles (row o = output neuron, K-major,
  // 128B-swizzled K-atoms).  Layer 0: columns in the tile's input order, FP32
  // bias as hi + lo at D0, D0+1.  Hidden layer h: [W | W] over 2C columns
  // (hi and lo halves of the activation); its bias hi, lo in columns
  // 16(h-1), 16(h-1)+1 of the bias tile (multiplied by the constant tile).
  // SnakeAlt folding as described at the top of the file.  A thread stages
  // 16-byte chunks (8 columns of one row), one or two of them, so the loads
  // of all weights are in flight at once: a call of few points is mostly this
  // staging (with one thread per row of a layer and a memset of the work
  // counter before the launch, 1000 points took 21.4 us a call and 2^20 81.9;
  // so 16.5 and 72.7).
  constexpr int CH0 = K0 / 8, CHH = 2 * C / 8;  // chunks of a row, layer 0 and hidden
  for (int it = tid; it < C * CH0 + (L - 2) * C * CHH; it += THREADS) {
    const int r = it < C * CH0 ? it / CH0 : (it - C * CH0) / CHH;  // row over all (hidden) layers
    const int cg = it < C * CH0 ? it - r * CH0 : (it - C * CH0) - r * CHH;
    const int layer = it < C * CH0 ? 0 : 1 + r / C, o = layer == 0 ? r : r - (layer - 1) * C;
    const int din = layer == 0 ? D0 : C;
    const __half* Wsrc = net.W_h + (layer == 0 ? 0 : (size_t)C * D0 + (size_t)(layer - 1) * C * C) + (size_t)o * din;
    const float scale = SNAKE && layer == 0 ? 2.0f : 1.0f;
    uint8_t* Wt = layer == 0 ? B0 : Bh + (layer - 1) * NAH * BT;
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      __half h2[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int col = 8 * cg + 2 * e + q;
        __half v = __float2half_rn(0.0f);
        if (layer == 0) {
          int src = -1;
          if (col < 2 * M) src = (col & 1) ? 3 + M + (col >> 1) : 3 + (col >> 1);
          else if (col < 2 * M + 3) src = col - 2 * M;
          else if (col < D0) src = col;
          const bool lat = src >= 3 + 2 * M && src < 3 + 2 * M + F;
          if (src >= 0) v = __float2half_rn(ldexpf(scale * __half2float(Wsrc[src]), lat ? gexp : 0));
          if (col == D0 || col == D0 + 1) {
            const float bias = scale * net.b[o];
            const __half bh = __float2half_rn(bias);
            v = col == D0 ? bh : __float2half_rn(bias - __half2float(bh));
          }
        } else {
          v = __float2half_rn((SNAKE && NEG ? -1.0f : 1.0f) * __half2float(Wsrc[col % C]));  // see act_fold
        }
        h2[q] = v;
      }
      __half2 hh = __halves2half2(h2[0], h2[1]);
      w[e] = *reinterpret_cast<uint32_t*>(&hh);
    }
    *reinterpret_cast<uint4*>(Wt + (cg >> 3) * BT + sw_off(o, cg & 7)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  // hidden biases, the last threads first (the chunks above take the first ones twice)
  for (int it = THREADS - 1 - tid; it < (L - 2) * C; it += THREADS) {
    const int layer = 1 + it / C, o = it - (layer - 1) * C;
    const __half* Wsrc = net.W_h + (size_t)C * D0 + (size_t)(layer - 1) * C * C + (size_t)o * C;
    float bias = net.b[layer * C + o];
    if (SNAKE) {
      float rs = 0.0f;
      for (int c = 0; c < C; ++c) rs += __half2float(Wsrc[c]);
      bias = 2.0f * bias + rs;
    }
    const int cg = 2 * (layer - 1);  // the layer's 16-column K-block: chunks cg, cg + 1
    const __half bh = __float2half_rn(bias);
    __half2 hb = __halves2half2(bh, __float2half_rn(bias - __half2float(bh)));
    const uint32_t wb = *reinterpret_cast<uint32_t*>(&hb);
    *reinterpret_cast<uint4*>(Bb + (cg >> 3) * BT + sw_off(o, cg & 7)) = make_uint4(wb, 0u, 0u, 0u);
    *reinterpret_cast<uint4*>(Bb + ((cg + 1) >> 3) * BT + sw_off(o, (cg + 1) & 7)) = make_uint4(0u, 0u, 0u, 0u);
  }
  if constexpr (ADJ) {
    // backward B tiles, unscaled FP16 weights, K = 2C (hi and lo halves of
    // the adjoint row): hidden layer h (1 <= h <= l-2): row n = input n of
    // the layer, column c -> W_h[c mod C][n]; layer 0: row n = tile input
    // column n (same order as the forward tile; zero for the bias columns and
    // the padding), column c -> W_0[c mod C][src(n)].
    const int rows = (L - 2) * C + K0;
    for (int it = tid; it < rows; it += THREADS) {
      const bool in0 = it >= (L - 2) * C;
      const int h = in0 ? 0 : 1 + it / C;
      const int n = in0 ? it - (L - 2) * C : it - (h - 1) * C;
      int src = n;
      if (in0) {
        if (n < 2 * M) src = (n & 1) ? 3 + M + (n >> 1) : 3 + (n >> 1);
        else if (n < 2 * M + 3) src = n - 2 * M;
        else if (n >= D0) src = -1;
      }
      const int din = in0 ? D0 : C;
      const __half* Wsrc = net.W_h + (in0 ? 0 : (size_t)C * D0 + (size_t)(h - 1) * C * C);
      uint8_t* Wt = in0 ? B0T : BhT + (h - 1) * NAH * BT;
      const int atom = in0 ? K0 * 128 : BT;  // bytes of one K-atom of this tile
      for (int cg = 0; cg < 2 * C / 8; ++cg) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c0 = (8 * cg + 2 * e) % C, c1 = (8 * cg + 2 * e + 1) % C;
          const __half v0 = src >= 0 ? Wsrc[(size_t)c0 * din + src] : __float2half_rn(0.0f);
          const __half v1 = src >= 0 ? Wsrc[(size_t)c1 * din + src] : __float2half_rn(0.0f);
          __half2 hh = __halves2half2(v0, v1);
          w[e] = *reinterpret_cast<uint32_t*>(&hh);
        }
        *reinterpret_cast<uint4*>(Wt + (cg >> 3) * atom + sw_off(n, cg & 7)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
  {
    // last layer on the CUDA cores: folded like the hidden layers
    const __half* Wl = net.W_h + (size_t)C * D0 + (size_t)(L - 2) * C * C;
    for (int i = tid; i < D * C; i += THREADS) wl[i] = (SNAKE ? (NEG ? -0.5f : 0.5f) : 1.0f) * __half2float(Wl[i]);
    if (tid < D) {
      float bias = net.b[(L - 1) * C + tid];
      if (SNAKE) {
        float rs = 0.0f;
        for (int c = 0; c < C; ++c) rs += __half2float(Wl[tid * C + c]);
        bias += 0.5f * rs;
      }
      wl[D * C + tid] = bias;
    }
    for (int i = tid; i < 3 * M; i += THREADS) fm[i] = net.fourier[i];
    if (GQ)
      for (int i = tid; i < 2 * F; i += THREADS)  // [lo + 128 step, step] per channel (latent_q)
        qp[i] = ldexpf((i & 1) ? net.grid_qp[i] : fmaf(128.0f, net.grid_qp[i + 1], net.grid_qp[i]), -gexp);
  }
  if constexpr (!POINTS) load_tf_segments(tf, b.tf);
  // the constant tile has ones in columns 0 and 1 of every row (the bias MMA
  // of the hidden layers)
  if (wg == 0) {
    uint8_t* One = sm + plan.oOne;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      *reinterpret_cast<uint4*>(One + sw_off(row, j)) = make_uint4(j == 0 ? pack_h2(1.0f, 1.0f) : 0u, 0u, 0u, 0u);
  }
  if (row == 0) {
    mbar_init(smem_u32(&mbar[wg]), 1);
    misc[4 + wg] = 0;
  }
  if (tid < 32) {
    tmem_alloc(smem_u32((const void*)&misc[0]), TMC);
    tmem_relinquish();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // row k of a NeRF matrix: 2 pi 2^(k div 3) on axis k mod 3, zero elsewhere
  bool ok = true;
  for (int i = tid; i < 3 * M; i += THREADS) {
    const int k = i / 3, a = i - 3 * k;
    ok &= fm[i] == (a == k % 3 ? 6.2831855f * (float)(1 << (k / 3)) : 0.0f);
  }
  const bool nerf = __syncthreads_and(ok) != 0;
  const uint32_t tmem = (uint32_t)misc[0];
  const uint32_t d_tmem = tmem + (uint32_t)(wg * tmem_wg_cols(C, SH, K0));
  const uint32_t t_row = d_tmem + ((uint32_t)((row >> 5) * 32) << 16);  // warp's lane quarter
  // operand rows: behind the accumulator (adjoint: in the upper half of the
  // wide accumulator, which only the last, N = K0 MMA fills; that MMA's row
  // takes the place of the consumed derivative stash)
  constexpr int ACOL = C;
  const uint32_t a_tmem = d_tmem + ACOL, t_a = t_row + ACOL;
  const uint64_t b0_desc = sw128_desc(smem_u32(B0)), bh_desc = sw128_desc(smem_u32(Bh)),
                 bb_desc = sw128_desc(smem_u32(Bb)), one_desc = sw128_desc(smem_u32(sm + plan.oOne));
  const uint64_t bht_desc = sw128_desc(smem_u32(BhT)), b0t_desc = sw128_desc(smem_u32(B0T));
  const uint32_t mb = smem_u32(&mbar[wg]);
  const int bar_id = 1 + wg;

  // ---- ray state
  const int tiles_x = (b.W + 7) / 8, tiles_y = (b.H + 3) / 4;
  const long long tpf = (long long)tiles_x * tiles_y;
  const long long n_rays = POINTS ? pd.n : tpf * 32 * b.n_views * b.n_times;
  const size_t gsz = (size_t)net.R * net.R * net.R * net.F;
  bool active = false, exhausted = false, failed = false;
  bool overflow = false;  // a non-finite network output (FP16 range exceeded)
  long long pix = 0;
  float3 o = make_float3(0.f, 0.f, 0.f), d = o;
  float t0 = 0.f, t1 = 0.f, C0 = 0.f, C1 = 0.f, C2 = 0.f, Acc = 0.f;
  int k = 0, pass = 0;
  RayLat rl{0, -1, 1.0f, 0.0f, 0.0f};
  float rho_c = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
  float3 ppos = make_float3(0.f, 0.f, 0.f);
  unsigned int ns = 0;
  uint32_t phase = 0;
  if (POINTS) {
    int k0;
    float f;
    time_weights(net, pd.time, k0, f);
    rl.g0 = (int)(k0 * gsz);
    rl.g1 = net.nkey > 1 ? (int)((k0 + 1) * gsz) : -1;
    rl.w0 = net.nkey > 1 ? 1.0f - f : 1.0f;
    rl.w1 = f;
    rl.tin = pd.time;
  }

  // Points are taken by the warp's place in the grid, then a grid stride on,
  // without round trips to the counter (1000 points 16.5 -> 12.3 us), so point
  // calls of one context may overlap on several streams.  Rays go
  // by the counter: they differ in length, and the choice at run time costs
  // the march 2 % (registers).
  uint32_t place = 32u * (blockIdx.x + gridDim.x * (unsigned)(tid >> 5));
  while (true) {
    // ---- refill: a warp whose lanes are all done claims the next 32 rays
    // (one 8 x 4 pixel tile), so its lanes march neighbouring rays together
    while (true) {
      bool need = !__any_sync(0xffffffffu, active) && !exhausted && !failed;
      if (POINTS && (long long)place >= n_rays) {
        exhausted = exhausted || need;
        need = false;
      }
      const unsigned int mask = __ballot_sync(0xffffffffu, need);
      if (mask == 0) break;
      unsigned long long base = 0;
      if constexpr (POINTS) {
        base = place;
        place += gridDim.x * THREADS;
      } else {
        const int leader = __ffs(mask) - 1;
        if (lane == leader) base = atomicAdd(ray_counter, (unsigned long long)__popc(mask));
        base = __shfl_sync(0xffffffffu, base, leader);
      }
      if (need) {
        const long long r = (long long)base + __popc(mask & ((1u << lane) - 1u));
        if (r >= n_rays) {
          exhausted = true;
        } else if (POINTS) {
          pix = r;
          ppos = make_float3(clamp01f(pd.pts[3 * r]), clamp01f(pd.pts[3 * r + 1]), clamp01f(pd.pts[3 * r + 2]));
          active = true;
        } else {
          const long long tile = r >> 5;
          const int li = (int)(r & 31);
          const long long frame = tile / tpf;
          const int tt = (int)(tile - frame * tpf);
          const int px = (tt % tiles_x) * 8 + (li & 7), py = (tt / tiles_x) * 4 + (li >> 3);
          if (px < b.W && py < b.H) {
            const int view = (int)(frame % b.n_views), ti = (int)(frame / b.n_views);
            pix = (frame * b.H + py) * (long long)b.W + px;
            camera_ray(b.cams[view], b.W, b.H, px, py, o, d);
            if (box_intersect(o, d, t0, t1)) {
              int k0;
              float f;
              time_weights(net, b.times[ti], k0, f);
              rl.g0 = (int)(k0 * gsz);
              rl.g1 = net.nkey > 1 ? (int)((k0 + 1) * gsz) : -1;
              rl.w0 = net.nkey > 1 ? 1.0f - f : 1.0f;
              rl.w1 = f;
              rl.tin = b.times[ti];
              C0 = C1 = C2 = Acc = 0.f;
              k = 0;
              pass = 0;
              active = true;
            } else {
              reinterpret_cast<float4*>(b.out)[pix] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
        }
      }
    }

    // ---- layer-0 input of this pass
    float len = 0.f;
    float3 qs = make_float3(0.f, 0.f, 0.f);  // sample position of this pass
    if (POINTS) {
      qs = ppos;
    } else if (active && !failed) {
      const float ta = fmaf((float)k, b.step, t0);
      const float tb = fminf(fmaf((float)(k + 1), b.step, t0), t1);
      len = tb - ta;
      const float tm = 0.5f * (ta + tb);
      float3 q = make_float3(clamp01f(fmaf(tm, d.x, o.x) + 0.5f), clamp01f(fmaf(tm, d.y, o.y) + 0.5f),
                             clamp01f(fmaf(tm, d.z, o.z) + 0.5f));
      if (SH == SRN_SHADE_FD && pass > 0) {
        const int ax = (pass - 1) >> 1;
        const float h = (pass & 1) ? b.fd_h : -b.fd_h;
        if (ax == 0) q.x = clamp01f(q.x + h);
        if (ax == 1) q.y = clamp01f(q.y + h);
        if (ax == 2) q.z = clamp01f(q.z + h);
      }
      qs = q;
    }
    if (__any_sync(0xffffffffu, active && !failed)) {
      write_input_row<M, F, K0, TI, GQ, ST, POINTS>(t_a, qs, nerf, fm, net.grid_h, net.grid_q, qp, net.R, rl);
      tmem_wait_st();
    }
    tc_fence_before();
    const bool any = bar_red_or(bar_id, 128, active && !failed);
    if (!any || misc[4 + wg]) break;
    if (issuer && !b.stall_test && elect_one()) {  // stall_test: no MMA, no commit, nothing in flight
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < K0 / 16; ++kk) {
        const uint32_t ka = ((16 * kk) >> 6), kb = ((16 * kk) & 63) * 2;
        mma_f16_ta(d_tmem, a_tmem + 8 * kk, desc_at(b0_desc, ka * BT + kb), IDESC, kk > 0);
      }
      mma_commit(mb);
    }

    // ---- layers: wait, read the accumulator row, activation, next MMA
    float out[4] = {0.f, 0.f, 0.f, 0.f};
    float dl[C];  // adjoint variant: d out / d (pre-activation) of the current layer
    bool stop = false;
#pragma unroll(LF > 0 ? LF - 1 : 1)
    for (int layer = 0; layer < L - 1; ++layer) {
      // the failure decision is warp-uniform so tcgen05.ld stays convergent;
      // a failed thread keeps arriving at the warpgroup barriers, which all
      // threads leave together once the flag is visible
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(mb, phase))) {
        failed = true;
        misc[4 + wg] = 1;
      }
      phase ^= 1u;
      tc_fence_after();
      float x[C];
      if (!failed) tmem_ld_row<C>(t_row, x);
      if (layer < L - 2) {
        if (!failed) {
          // activation as FP16 hi (columns 0..C-1) + lo (columns C..2C-1)
#pragma unroll
          for (int j = 0; j < C / 16; ++j) {
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float2 a = act_fold<ACT, PACK, NEG>(x[16 * j + 2 * e], x[16 * j + 2 * e + 1]);
              split_h2(a.x, a.y, hi[e], lo[e]);
            }
            tmem_st8(t_a + 8 * j, hi);
            tmem_st8(t_a + C / 2 + 8 * j, lo);
          }
          tmem_wait_st();
          if constexpr (ADJ) {
            // activation derivative of this hidden layer, kept in TMEM for the
            // backward: SnakeAlt' = 0.5 + sin(2x) (the accumulator holds 2x); sin' = cos
            float dv[C];
#pragma unroll
            for (int j = 0; j < C; j += 2) {
              const float2 p = SNAKE ? __fadd2_rn(make_float2(0.5f, 0.5f), make_float2(__sinf(x[j]), __sinf(x[j + 1])))
                                     : make_float2(__cosf(x[j]), __cosf(x[j + 1]));
              dv[j] = p.x;
              dv[j + 1] = p.y;
            }
            tmem_st_row<C>(t_row + NACC + C * layer, dv);
          }
        }
        tc_fence_before();
        if (bar_red_or(bar_id, 128, failed)) { stop = true; break; }
        if (issuer && elect_one()) {
          tc_fence_after();
          const uint64_t bw = desc_at(bh_desc, layer * NAH * BT);
          const uint32_t kbias = 16 * layer;  // this layer's K-block of the bias tile
          mma_f16(d_tmem, one_desc, desc_at(bb_desc, (kbias >> 6) * BT + (kbias & 63) * 2), IDESC,
                  0u);
#pragma unroll
          for (int kk = 0; kk < 2 * C / 16; ++kk) {
            const uint32_t ka = ((16 * kk) >> 6), kb = ((16 * kk) & 63) * 2;
            mma_f16_ta(d_tmem, a_tmem + 8 * kk, desc_at(bw, ka * BT + kb), IDESC, 1u);
          }
          mma_commit(mb);
        }
      } else if (!failed) {
        if constexpr (SUM2) {
          float2 a[C / 2];
#pragma unroll
          for (int j = 0; j < C / 2; ++j) a[j] = act_fold<ACT, PACK, NEG>(x[2 * j], x[2 * j + 1]);
#pragma unroll
          for (int dd = 0; dd < 4; ++dd) {
            if (dd < D) {
              float2 sacc = make_float2(wl[D * C + dd], 0.0f);
#pragma unroll
              for (int j = 0; j < C / 2; j += 2) {
                const float4 w = *reinterpret_cast<const float4*>(wl + dd * C + 2 * j);
                if (PACK) {
                  sacc = __ffma2_rn(make_float2(w.x, w.y), a[j], sacc);
                  sacc = __ffma2_rn(make_float2(w.z, w.w), a[j + 1], sacc);
                } else {
                  sacc = make_float2(fmaf(w.x, a[j].x, sacc.x), fmaf(w.y, a[j].y, sacc.y));
                  sacc = make_float2(fmaf(w.z, a[j + 1].x, sacc.x), fmaf(w.w, a[j + 1].y, sacc.y));
                }
              }
              out[dd] = sacc.x + sacc.y;
            }
          }
        } else {
          float a[C];
#pragma unroll
          for (int j = 0; j < C; j += 2) {
            const float2 v = act_fold<ACT, false, NEG>(x[j], x[j + 1]);
            a[j] = v.x;
            a[j + 1] = v.y;
          }
#pragma unroll
          for (int dd = 0; dd < 4; ++dd) {
            if (dd < D) {
              float sacc = wl[D * C + dd];
#pragma unroll
              for (int j = 0; j < C; ++j) sacc = fmaf(wl[dd * C + j], a[j], sacc);
              out[dd] = sacc;
            }
          }
        }
        if constexpr (ADJ) {
          // d out / d x of the last hidden layer; wl holds W / 2 (NEG: -W / 2) for SnakeAlt
#pragma unroll
          for (int j = 0; j < C; ++j) dl[j] = SNAKE ? (NEG ? -wl[j] : wl[j]) * fmaf(2.0f, __sinf(x[j]), 1.0f) : wl[j] * __cosf(x[j]);
        }
      }
    }
    if (stop) break;

    // ---- adjoint input gradient (Section 5): backward through the hidden
    // layers and layer 0 on the tensor cores, the adjoint row split into FP16
    // hi + lo like the activations; then the Fourier and latent Jacobians.
    float3 gadj = make_float3(0.f, 0.f, 0.f);
    if constexpr (ADJ) {
      for (int h = L - 2; h >= 0; --h) {
        const int acol = h >= 1 ? ACOL : NACC;
        if (!failed) {
#pragma unroll
          for (int j = 0; j < C / 16; ++j) {
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              split_h2(dl[16 * j + 2 * e], dl[16 * j + 2 * e + 1], hi[e], lo[e]);
            }
            tmem_st8(t_row + acol + 8 * j, hi);
            tmem_st8(t_row + acol + C / 2 + 8 * j, lo);
          }
          tmem_wait_st();
        }
        tc_fence_before();
        if (bar_red_or(bar_id, 128, failed)) { stop = true; break; }
        if (issuer && elect_one()) {
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 2 * C / 16; ++kk) {
            const uint32_t ka = ((16 * kk) >> 6), kb = ((16 * kk) & 63) * 2;
            const uint32_t ad = d_tmem + acol + 8 * kk;
            if (h >= 1)
              mma_f16_ta(d_tmem, ad, desc_at(bht_desc, (h - 1) * NAH * BT + ka * BT + kb), IDESC, kk > 0);
            else
              mma_f16_ta(d_tmem, ad, desc_at(b0t_desc, ka * (K0 * 128) + kb), idesc_n(K0), kk > 0);
          }
          mma_commit(mb);
        }
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(mb, phase))) {
          failed = true;
          misc[4 + wg] = 1;
        }
        phase ^= 1u;
        tc_fence_after();
        if (failed) continue;
        if (h >= 1) {
          // packed here and where dv is made: 512^2 shaded 13.3 -> 12.9 ms
          float g[C], dv[C];
          tmem_ld_row<C>(t_row, g);
          tmem_ld_row<C>(t_row + NACC + C * (h - 1), dv);
#pragma unroll
          for (int j = 0; j < C; j += 2) {
            const float2 p = __fmul2_rn(make_float2(g[j], g[j + 1]), make_float2(dv[j], dv[j + 1]));
            dl[j] = p.x;
            dl[j + 1] = p.y;
          }
        } else {
          // in two parts, so that half the registers hold it at a time: the
          // Fourier and position columns with what shares their last 16, then
          // the rest of the latent columns
          constexpr int P1 = (2 * M + 3 + 15) / 16 * 16, P2 = (2 * M + 3 + F - P1 + 15) / 16 * 16;
          float gv[P1], gl[F];
          tmem_ld_row<P1>(t_row, gv);
          float3 gp = make_float3(gv[2 * M], gv[2 * M + 1], gv[2 * M + 2]);
          if (active) {
            // the Fourier features: d sin e = cos e F_k, d cos e = -sin e F_k
            if (nerf) {
              constexpr int kReseed = M > 15 ? 4 : 64;
              constexpr float kW = 6.28318548202514648f, kWErr = 1.74845560252379070e-7f;
              float sn[3], cs[3];
              float ga[3] = {0.f, 0.f, 0.f};
#pragma unroll
              for (int kq = 0; kq < M; ++kq) {
                const int a = kq % 3, j = kq / 3;
                const float pa = a == 0 ? qs.x : (a == 1 ? qs.y : qs.z);
                if (j % kReseed == 0) {
                  const float xx = pa * (float)(1 << j);
                  const float r = rintf(xx);
                  __sincosf(fmaf(kW, xx - r, kWErr * r), &sn[a], &cs[a]);
                } else {
                  const float ss = sn[a], cc = cs[a];
                  sn[a] = 2.0f * ss * cc;
                  cs[a] = (cc - ss) * (cc + ss);
                }
                ga[a] = fmaf(fm[3 * kq + a], gv[2 * kq] * cs[a] - gv[2 * kq + 1] * sn[a], ga[a]);
              }
              gp.x += ga[0];
              gp.y += ga[1];
              gp.z += ga[2];
            } else {
#pragma unroll
              for (int kq = 0; kq < M; ++kq) {
                const float e = fm[3 * kq] * qs.x + fm[3 * kq + 1] * qs.y + fm[3 * kq + 2] * qs.z;
                float sv, cv;
                sincosf(e, &sv, &cv);
                const float coef = gv[2 * kq] * cv - gv[2 * kq + 1] * sv;
                gp.x = fmaf(coef, fm[3 * kq], gp.x);
                gp.y = fmaf(coef, fm[3 * kq + 1], gp.y);
                gp.z = fmaf(coef, fm[3 * kq + 2], gp.z);
              }
            }
          }
#pragma unroll
          for (int c = 0; c < F; ++c)
            if (2 * M + 3 + c < P1) gl[c] = gv[2 * M + 3 + c];
          float g2[P2];
          tmem_ld_row<P2>(t_row + P1, g2);
#pragma unroll
          for (int c = 0; c < F; ++c)
            if (2 * M + 3 + c >= P1) gl[c] = g2[2 * M + 3 + c - P1];
          if (active) {
            const float3 l = latent_grad_h<F, ST>(net.grid_h, net.R, rl, qs, gl);
            // grid_h = G 2^-gexp
            gadj = make_float3(fmaf(l.x, gscale, gp.x), fmaf(l.y, gscale, gp.y), fmaf(l.z, gscale, gp.z));
          }
        }
      }
      if (stop) break;
    }

    if (POINTS) {
      if (active && !failed) {
        if constexpr (ADJ) {
          // density and gradient mode: out is the density [n] (output 0 of a
          // 4-output head), grad [n][3]
          pd.out[pix] = out[0];
          if (pd.grad) {
            pd.grad[3 * pix] = gadj.x;
            pd.grad[3 * pix + 1] = gadj.y;
            pd.grad[3 * pix + 2] = gadj.z;
          }
        } else {
          for (int dd = 0; dd < D; ++dd) pd.out[pix * D + dd] = out[dd];
        }
        overflow |= !(fabsf(out[0]) < INFINITY);
        ++ns;
        active = false;
      }
      continue;
    }
    // ---- transfer function, shading, compositing, termination
    if (active && !failed) {
      bool sample_done = true;
      float3 g = make_float3(0.f, 0.f, 0.f);
      if (SH == SRN_SHADE_FD) {
        if (pass == 0) rho_c = out[0];
        else if (pass == 1) gx = out[0];
        else if (pass == 2) gx = (gx - out[0]) / (2.0f * b.fd_h);
        else if (pass == 3) gy = out[0];
        else if (pass == 4) gy = (gy - out[0]) / (2.0f * b.fd_h);
        else if (pass == 5) gz = out[0];
        else gz = (gz - out[0]) / (2.0f * b.fd_h);
        sample_done = pass == NP - 1;
        pass = sample_done ? 0 : pass + 1;
        g = make_float3(gx, gy, gz);
      } else {
        rho_c = out[0];
        if (SH == SRN_SHADE_HEAD) g = make_float3(out[1], out[2], out[3]);
        if (ADJ) g = gadj;
      }
      if (sample_done) {
        ++ns;
        overflow |= !(fabsf(rho_c) < INFINITY);
        float4 c = tf_segment_eval(tf, (b.tf.n + 2) / 4, rho_c);
        const float alpha = 1.0f - __expf(-c.w * b.tf.opacity_scale * len);
        if (SH != SRN_SHADE_NONE) shade(c, g, d);
        const float w = (1.0f - Acc) * alpha;
        C0 = fmaf(w, c.x, C0);
        C1 = fmaf(w, c.y, C1);
        C2 = fmaf(w, c.z, C2);
        Acc += w;
        ++k;
        if (Acc >= b.et || fmaf((float)k, b.step, t0) >= t1) {
          reinterpret_cast<float4*>(b.out)[pix] = make_float4(C0, C1, C2, Acc);
          active = false;
        }
      }
    }
  }

  if (failed || misc[4 + wg]) {
    if (row == 0) atomicExch(status, (unsigned int)SRN_ERR_TIMEOUT);
  } else if (__any_sync(0xffffffffu, overflow) && lane == 0) {
    // an input or activation outside the FP16 range made the output
    // non-finite; the FP32 path evaluates such networks
    atomicCAS(status, (unsigned int)SRN_OK, (unsigned int)SRN_ERR_NONFINITE);
  }
  if (!POINTS) add_samples(b.samples, ns);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid < 32) tmem_dealloc(tmem, TMC);
}

template <int C, int M, int F, int ACT, int SH, int TI, int GQ, int LF, int ST>
cudaError_t launch_t(const NetDev& net, const BatchDev& b, const PointsDev& pd, unsigned long long* ctr,
                     unsigned int* status, cudaStream_t s) {
  if (LF > 0 && (net.l != LF || net.D != (SH == SRN_SHADE_HEAD ? 4 : 1))) return cudaErrorInvalidValue;
  if (ST && net.nkey != 1) return cudaErrorInvalidValue;
  SmemPlan plan = make_plan(net, C, wgs_for(C, SH), is_adjoint(SH));
  auto k = render_mma_kernel<C, M, F, ACT, SH, TI, GQ, LF, ST>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.total);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // one CTA per SM, or one per 32 points / pixel tile where there are fewer:
  // a warp claims 32 at a time
  const long long claims = is_points(SH) ? (pd.n + 31) / 32
                                         : (long long)((b.W + 7) / 8) * ((b.H + 3) / 4) * b.n_views * b.n_times;
  const unsigned grid = (unsigned)(claims < sms ? claims : sms);
  if constexpr (is_points(SH)) {
    k<<<grid, 128 * wgs_for(C, SH), plan.total, s>>>(net, PointsBatch{}, pd, plan, ctr, status);
  } else {
    // Cleared here and not by the launch before: what overlapping calls of
    // one context leave in the counter reaches no later frame.
    e = cudaMemsetAsync(ctr, 0, sizeof(*ctr), s);
    if (e != cudaSuccess) return e;
    k<<<grid, 128 * wgs_for(C, SH), plan.total, s>>>(net, b, pd, plan, ctr, status);
  }
  return cudaGetLastError();
}

// Explicit instantiation of one variant (used by the srn_mma_w*.cu units);
// SRN_MMA_INSTANTIATE_L fixes the layer count (LF) and whether the network
// has a single latent grid (ST).
#define SRN_MMA_INSTANTIATE_L(C, M, F, ACT, SH, TI, GQ, LF, ST)                                                  \
  template cudaError_t launch_t<C, M, F, ACT, SH, TI, GQ, LF, ST>(const NetDev&, const BatchDev&,               \
                                                                  const PointsDev&, unsigned long long*,        \
                                                                  unsigned int*, cudaStream_t);
#define SRN_MMA_INSTANTIATE(C, M, F, ACT, SH, TI, GQ) SRN_MMA_INSTANTIATE_L(C, M, F, ACT, SH, TI, GQ, 0, 0)

}  // namespace mma
}  // namespace srn
