// Declarations shared by the tensor-core render kernel (srn_mma_kernel.cuh),
// its explicit instantiations (srn_mma_k*.cu) and the dispatcher
// (srn_mma.cu).  Each kernel variant is compiled in exactly one translation
// unit, so the variants build in parallel.
#pragma once
#include "srn_internal.h"

namespace srn {
namespace mma {


constexpr int kPoints = 4;     // kernel mode: network output at given points (no ray march)
constexpr int kPointsAdj = 5;  // kernel mode: density and adjoint input gradient at given points
constexpr bool is_adjoint(int SH) { return SH == SRN_SHADE_ADJOINT || SH == kPointsAdj; }
constexpr bool is_points(int SH) { return SH == kPoints || SH == kPointsAdj; }

// Warpgroups per CTA for hidden width C and shading mode SH (one CTA per
// SM): what the register file and TMEM allow.  Width 32 runs 7 (72 registers a thread), except the
// finite-difference variant, whose extra state needs the 80 registers of 6,
// and the adjoint variants, whose TMEM stash limits them to 4.
constexpr int wgs_for(int C, int SH) {
  return is_adjoint(SH) ? (C == 32 ? 4 : 2)
                        : (C == 32 ? (SH == SRN_SHADE_FD ? 6 : 7) : (C == 48 ? 4 : 3));
}
constexpr int kAdjMaxLayers = 4;  // layers of the networks the tensor-core adjoint takes
// TMEM columns a CTA allocates (all 512: one CTA holds an SM's registers, so
// no second CTA of these kernels waits for columns), and the columns of one
// warpgroup.  A warpgroup holds its accumulator (C columns) and, from column
// C on, its operand rows: max(K0, 2C) FP16, two per column (C = 32: 64
// columns, seven warpgroups 448; 48: 96, four; 64: 128, three).  The adjoint
// variants widen the accumulator for the input-gradient MMA (N = K0 columns,
// which overlap the operand rows of the other layers: its own row lies in the
// stash, consumed by then) and append the stashed activation derivatives of
// the (at most two) hidden layers, C columns each: 64 + 64 (width 32, four
// warpgroups), 96 + 96 (48, two), 128 + 128 (64, two).
constexpr int kTmemCols = 512;
constexpr int a_cols(int C, int K0) { return K0 / 2 > C ? K0 / 2 : C; }
constexpr int adj_acc_cols(int C, int K0) {
  return K0 > C + a_cols(C, K0) ? ((K0 + 31) / 32) * 32 : C + a_cols(C, K0);
}
constexpr int tmem_wg_cols(int C, int SH, int K0) {
  return is_adjoint(SH) ? adj_acc_cols(C, K0) + (kAdjMaxLayers - 2) * C : C + a_cols(C, K0);
}
constexpr int kTile = 128 * 128;       // 128 rows x 128 B (64 FP16 columns): the constant tile

constexpr long long kWaitCycles = 2000000000ll;  // ~1 s at 2 GHz

// Point-evaluation arguments (modes kPoints, kPointsAdj).
struct PointsDev {
  const float* pts;  // [n][3]
  float* out;        // [n][D] (kPointsAdj: density [n])
  long long n;
  float time;
  float* grad;       // kPointsAdj: d rho / d p [n][3], or null
};

// What the point modes take in place of a batch of frames: the same names
// without the cameras, times and transfer function, 7 KB of kernel arguments
// that a call of few points would wait for.
struct PointsBatch {
  CamDev cams[1];
  float times[1];
  int n_views, n_times, W, H;
  float step, et, fd_h;
  struct {
    int n;
    float opacity_scale;
  } tf;
  float* out;
  unsigned long long* samples;
  int stall_test;
};

// ---------------------------------------------------------------- layout
struct SmemPlan {
  int oOne, oB0, oBh, oBb, oBhT, oB0T, oWl, oTF, oFm, oQp, oMbar, oMisc, total;
};

// Shared memory for hidden width C and WGS warpgroups: the weights (B tiles,
// 128B-swizzled K-atoms C * 128 bytes apart) and small tables.  The per-ray
// operand rows are in tensor memory, so most of the SM's 256 KB stay L1.
inline SmemPlan make_plan(const NetDev& n, int C, int WGS, bool adjoint = false) {
  const int D0 = net_d0(n);
  const int K0 = ((D0 + 2 + 15) / 16) * 16;
  const int NA0 = (K0 + 63) / 64, NAH = (2 * C + 63) / 64;
  const int BT = C * 128;
  const int NBB = n.l > 2 ? (16 * (n.l - 2) + 63) / 64 : 1;
  SmemPlan s;
  int o = 0;
  s.oOne = o; o += kTile;                   // constant tile: columns 0, 1 = 1
  s.oB0 = o; o += NA0 * BT;                 // layer 0
  s.oBh = o; o += (n.l - 2) * NAH * BT;     // hidden layers: [W | W]
  s.oBb = o; o += NBB * BT;                 // hidden biases, one 16-column K-block per layer
  s.oBhT = o; if (adjoint) o += (n.l - 2) * NAH * BT;      // adjoint: [W_h^T | W_h^T] of the hidden layers
  s.oB0T = o; if (adjoint) o += NAH * (NA0 * 64) * 128;    // adjoint: [W_0^T | W_0^T], K0 rows
  s.oWl = o; o += (n.D * C + 4) * 4;
  o = (o + 15) & ~15;
  s.oTF = o; o += (int)sizeof(TFSeg);
  o = (o + 15) & ~15;
  s.oFm = o; o += ((3 * n.m + 3) & ~3) * 4 + 16;
  s.oQp = o; o += 2 * 32 * 4;
  o = (o + 7) & ~7;
  s.oMbar = o; o += 8 * WGS;
  s.oMisc = o; o += 16 * 4;
  s.total = o + 1024;  // alignment slack
  return s;
}

// One kernel variant: hidden width C, M Fourier rows, F latent channels,
// activation ACT, shading SH (or kPoints), direct time input TI, 8-bit grid
// GQ; LF > 0: a network of LF layers and D = 1 output (4 with head
// shading), both fixed at compile time (0: read from the network); ST = 1:
// a single latent grid (no keyframes), so the gather has no time blend.
// Defined in srn_mma_kernel.cuh, instantiated in srn_mma_w*.cu.
template <int C, int M, int F, int ACT, int SH, int TI, int GQ, int LF = 0, int ST = 0>
cudaError_t launch_t(const NetDev& net, const BatchDev& b, const PointsDev& pd, unsigned long long* ctr,
                     unsigned int* status, cudaStream_t s);

}  // namespace mma
}  // namespace srn
