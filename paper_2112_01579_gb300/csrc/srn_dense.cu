// Dense-grid direct volume rendering of a float32 volume: the plain method
// the fV-SRN network stands in for, and the reference renderer of the paper's
// quality comparisons (Section 4 / 6).  Same ray march, transfer function,
// compositing and shading as the network renderer; density = trilinear
// interpolation of the volume.
//
// One thread per ray, 32 pixels a warp.  Bound by issue slots and by the L1
// data pipe at once (a warp's corner load takes one wavefront per cache line
// it touches), so both are kept low: the sample position is carried in voxel
// units (one FMA per axis), offsets are 32 bits where the volume has fewer
// than 2^31 voxels, the interpolation is seven nested lerps by two weights (a
// difference of two voxels would lose infinities), the transfer
// function's segment comes from counting control points out of two 16-byte
// loads, and the corner values stay in registers while a ray stays in its
// cell (two samples in five at half a voxel a step).  A 1024^2 frame of a
// 256^3 volume: 1427 -> 1062 us; without the kept corners 6 % more, and pixel
// tiles chosen per view to cross the fewest rows gained nothing.

#include "srn_device.cuh"

namespace srn {
namespace {

constexpr int kThreads = 128;

// The cell a ray is in and its corner values.
template <class I>
struct Cell {
  I at;
  float c[8];
};

// Trilinear density at voxel coordinates g (vertex i at coordinate i).  The
// lerps are (1 - f) a + f b and not a + f (b - a): infinite or very large
// voxels next to each other or to small ones keep their values.
template <class I, bool CACHED>
__device__ __forceinline__ float sample(const VolDev& v, I sy, I sz, float3 g, Cell<I>& k) {
  const int ix = min(max(__float2int_rd(g.x), 0), v.nx - 2), iy = min(max(__float2int_rd(g.y), 0), v.ny - 2),
            iz = min(max(__float2int_rd(g.z), 0), v.nz - 2);
  // saturated: a coordinate outside the volume (the rounding of a ray from
  // far away) takes the value at the face, in no more instructions
  const float fx = __saturatef(g.x - (float)ix), fy = __saturatef(g.y - (float)iy), fz = __saturatef(g.z - (float)iz);
  const I at = (I)iz * sz + (I)iy * sy + (I)ix;
  if (!CACHED || at != k.at) {
    k.at = at;
    k.c[0] = __ldg(v.vol + at); k.c[1] = __ldg(v.vol + at + 1);
    k.c[2] = __ldg(v.vol + at + sy); k.c[3] = __ldg(v.vol + at + sy + 1);
    k.c[4] = __ldg(v.vol + at + sz); k.c[5] = __ldg(v.vol + at + sz + 1);
    k.c[6] = __ldg(v.vol + at + sz + sy); k.c[7] = __ldg(v.vol + at + sz + sy + 1);
  }
  const float ex = 1.0f - fx, ey = 1.0f - fy, ez = 1.0f - fz;
  const float x0 = fmaf(fx, k.c[1], ex * k.c[0]), x1 = fmaf(fx, k.c[3], ex * k.c[2]);
  const float x2 = fmaf(fx, k.c[5], ex * k.c[4]), x3 = fmaf(fx, k.c[7], ex * k.c[6]);
  const float y0 = fmaf(fy, x1, ey * x0), y1 = fmaf(fy, x3, ey * x2);
  return fmaf(fz, y1, ez * y0);
}

// 1 - exp(-x): the series for |x| below 1/4 (the first term left out is
// 5e-8 of the value there), where 1 - exp would cancel; steps are short, so
// that is nearly every sample.  x is negative where a control point's alpha is.
__device__ __forceinline__ float opacity(float x) {
  if (fabsf(x) < 0.25f) {
    float p = fmaf(x, -1.0f / 720.0f, 1.0f / 120.0f);
    p = fmaf(x, p, -1.0f / 24.0f);
    p = fmaf(x, p, 1.0f / 6.0f);
    p = fmaf(x, p, -0.5f);
    return fmaf(x * x, p, x);
  }
  return 1.0f - expf(-x);
}

template <bool FD, class I>
__global__ void __launch_bounds__(kThreads) dvr_dense_kernel(const VolDev v, const BatchDev b) {
  __shared__ TFSeg tf;
  load_tf_segments(tf, b.tf);
  __syncthreads();
  const int quads = (b.tf.n + 2) / 4;  // n - 1 bounds
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const int tiles_x = (b.W + 7) / 8, tiles_y = (b.H + 3) / 4;
  const long long tpf = (long long)tiles_x * tiles_y;
  const long long frame = warp / tpf;
  if (frame >= (long long)b.n_times * b.n_views) return;
  const int t = (int)(warp - frame * tpf);
  const int px = (t % tiles_x) * 8 + (lane & 7), py = (t / tiles_x) * 4 + (lane >> 3);
  const int view = (int)(frame % b.n_views);
  if (px >= b.W || py >= b.H) return;

  float3 o, d;
  camera_ray(b.cams[view], b.W, b.H, px, py, o, d);
  float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
  unsigned int ns = 0;
  float t0, t1;
  if (box_intersect(o, d, t0, t1)) {
    const I sy = (I)v.nx, sz = (I)v.nx * (I)v.ny;
    const float mx = (float)(v.nx - 1), my = (float)(v.ny - 1), mz = (float)(v.nz - 1);
    const float3 gd = make_float3(d.x * mx, d.y * my, d.z * mz);
    const float3 go = make_float3((o.x + 0.5f) * mx, (o.y + 0.5f) * my, (o.z + 0.5f) * mz);
    const float scale = b.tf.opacity_scale;
    Cell<I> cell, side;
    cell.at = ~(I)0;
    float ta = t0;
    for (float k = 1.0f; ta < t1; k += 1.0f) {
      const float tb = fminf(fmaf(k, b.step, t0), t1);
      const float len = tb - ta, tm = 0.5f * (ta + tb);
      // inside the box up to rounding; sample() clamps, the neighbours need it here
      float3 g = make_float3(fmaf(tm, gd.x, go.x), fmaf(tm, gd.y, go.y), fmaf(tm, gd.z, go.z));
      if (FD) g = make_float3(fminf(fmaxf(g.x, 0.0f), mx), fminf(fmaxf(g.y, 0.0f), my), fminf(fmaxf(g.z, 0.0f), mz));
      const float rho = sample<I, true>(v, sy, sz, g, cell);
      ++ns;
      float4 c = tf_segment_eval(tf, quads, rho);
      const float alpha = opacity(scale * c.w * len);
      if (FD) {
        // central differences one voxel apart, clamped to the volume
        float3 n;
        n.x = 0.5f * mx * (sample<I, false>(v, sy, sz, make_float3(fminf(g.x + 1.0f, mx), g.y, g.z), side) -
                           sample<I, false>(v, sy, sz, make_float3(fmaxf(g.x - 1.0f, 0.0f), g.y, g.z), side));
        n.y = 0.5f * my * (sample<I, false>(v, sy, sz, make_float3(g.x, fminf(g.y + 1.0f, my), g.z), side) -
                           sample<I, false>(v, sy, sz, make_float3(g.x, fmaxf(g.y - 1.0f, 0.0f), g.z), side));
        n.z = 0.5f * mz * (sample<I, false>(v, sy, sz, make_float3(g.x, g.y, fminf(g.z + 1.0f, mz)), side) -
                           sample<I, false>(v, sy, sz, make_float3(g.x, g.y, fmaxf(g.z - 1.0f, 0.0f)), side));
        shade(c, n, d);
      }
      const float w = (1.0f - A) * alpha;
      C0 = fmaf(w, c.x, C0);
      C1 = fmaf(w, c.y, C1);
      C2 = fmaf(w, c.z, C2);
      A += w;
      ta = tb;
      if (A >= b.et) break;
    }
  }
  size_t idx = ((size_t)frame * b.H + py) * b.W + px;
  reinterpret_cast<float4*>(b.out)[idx] = make_float4(C0, C1, C2, A);
  add_samples(b.samples, ns);
}

}  // namespace

cudaError_t launch_dvr_dense(const VolDev& v, const BatchDev& b, cudaStream_t s) {
  const long long tiles = (long long)((b.W + 7) / 8) * ((b.H + 3) / 4) * b.n_views * b.n_times;
  const unsigned blocks = (unsigned)((tiles + (kThreads / 32) - 1) / (kThreads / 32));
  const bool small = (long long)v.nx * v.ny < (1ll << 31) && (long long)v.nx * v.ny * v.nz < (1ll << 31);
  if (b.shading == SRN_SHADE_NONE) {
    if (small) dvr_dense_kernel<false, unsigned int><<<blocks, kThreads, 0, s>>>(v, b);
    else dvr_dense_kernel<false, unsigned long long><<<blocks, kThreads, 0, s>>>(v, b);
  } else {
    if (small) dvr_dense_kernel<true, unsigned int><<<blocks, kThreads, 0, s>>>(v, b);
    else dvr_dense_kernel<true, unsigned long long><<<blocks, kThreads, 0, s>>>(v, b);
  }
  return cudaGetLastError();
}

}  // namespace srn
