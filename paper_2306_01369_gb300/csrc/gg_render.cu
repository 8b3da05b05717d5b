// gg_render.cu -- depth observations computed on the device (the paper's Sec. III-A
// "sky" and "ego" cameras): an orthographic height map of the particle surface and a
// perspective depth image of particles and rigid bodies.
//
// Particles are splatted: one thread per sphere visits the pixels its conservative
// footprint covers, tests each pixel exactly (FP32, fixed order) and folds its value
// into the pixel with an integer atomic max / min on the float's ordered bits, so the
// image does not depend on the order of the spheres.  Bodies are sphere traced per
// pixel (FP32, fixed order) and merged.  The decisions (coverage, ray-sphere hit,
// every tracing step) use the same operations in the same order as the oracle.
//
// An image is a chain of short kernels, so they are chained with programmatic dependent
// launch and each does as little as it can: the spheres are taken last id first (beds are
// laid down bottom up, so what a camera above sees comes early), and a ray stops being traced
// where the spheres already block it.  A look at a pixel before its atomic does not pay: the
// atomics are not waited for, the look is, at every pixel of a sphere's loop (height map of
// 4,000 spheres at 640 x 480 178 us without and 775 with it, of 16,000 at 160 x 96 14.5 and
// 34.3, of 262,144 at 72 x 36 9.7 and 10.4; only 600,000 at 640 x 480 gained, 79 and 70).
#include <algorithm>

#include <cuda_runtime.h>

#include "gg_device.cuh"
#include "gg_internal.h"

namespace gg {

namespace {

// Order-preserving map of a float onto uint32 (for atomicMax over signed values);
// 0 is below every image of a float.
__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_ordered(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__global__ void k_fill(uint32_t *img, uint32_t count, uint32_t v) {
  pdl_enter();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < count) img[p] = v;
}

__device__ __forceinline__ float pixel_centre(float base, uint32_t u, float step) {
  return __fadd_rn(base, __fmul_rn(__fadd_rn((float)u, 0.5f), step));
}

__global__ void k_splat_height(StepArgs a, uint32_t off, uint32_t n, RenderArgs c, uint32_t *img) {
  pdl_enter();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 p = a.pos_id[off + (n - 1u - i)];
  // conservative pixel range: |x - px| <= r with px = bx + (u + 1/2) sx
  const int u0 = max(0, (int)floorf((p.x - p.w - c.bx) / c.sx - 0.5f) - 1);
  const int u1 = min((int)c.W - 1, (int)ceilf((p.x + p.w - c.bx) / c.sx - 0.5f) + 1);
  const int v0 = max(0, (int)floorf((p.y - p.w - c.by) / c.sy - 0.5f) - 1);
  const int v1 = min((int)c.H - 1, (int)ceilf((p.y + p.w - c.by) / c.sy - 0.5f) + 1);
  const float r2 = __fmul_rn(p.w, p.w);
  for (int v = v0; v <= v1; ++v) {
    const float py = pixel_centre(c.by, (uint32_t)v, c.sy);
    const float dy = __fsub_rn(p.y, py);
    for (int u = u0; u <= u1; ++u) {
      const float px = pixel_centre(c.bx, (uint32_t)u, c.sx);
      const float dx = __fsub_rn(p.x, px);
      const float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
      if (!(d2 <= r2)) continue;
      const float h = __fadd_rn(p.z, __fsqrt_rn(__fsub_rn(r2, d2)));
      atomicMax(&img[(size_t)v * c.W + u], ordered(h));  // (nothing waits for it; a look first made its loop wait)
    }
  }
}

__global__ void k_finish_height(const uint32_t *img, uint32_t count, float empty, float *out) {
  pdl_enter();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < count) out[p] = img[p] ? from_ordered(img[p]) : empty;
}

// Unit ray of pixel (u, v) in the world frame, FP32 in the oracle's order.
__device__ __forceinline__ float3 pixel_ray(const RenderArgs &c, uint32_t u, uint32_t v) {
  const float ax = __fsub_rn(__fadd_rn((float)u, 0.5f), __fmul_rn(0.5f, (float)c.W));
  const float ay = __fsub_rn(__fadd_rn((float)v, 0.5f), __fmul_rn(0.5f, (float)c.H));
  const float dxc = __fdiv_rn(ax, c.f), dyc = __fdiv_rn(ay, c.f);
  const float s = __fadd_rn(__fadd_rn(__fmul_rn(dxc, dxc), __fmul_rn(dyc, dyc)), 1.0f);
  const float nr = __fsqrt_rn(s);
  const float dc[3] = {__fdiv_rn(dxc, nr), __fdiv_rn(dyc, nr), __fdiv_rn(1.0f, nr)};
  float d[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    d[k] = __fadd_rn(__fadd_rn(__fmul_rn(c.R[3 * k], dc[0]), __fmul_rn(c.R[3 * k + 1], dc[1])),
                     __fmul_rn(c.R[3 * k + 2], dc[2]));
  return make_float3(d[0], d[1], d[2]);
}

// Every pixel's ray, once per image (the splat tests many spheres against each), and its
// empty value.
__global__ void k_begin_depth(RenderArgs c, uint32_t *img) {
  pdl_enter();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= c.W * c.H) return;
  const float3 d = pixel_ray(c, p % c.W, p / c.W);
  c.rays[p] = make_float4(d.x, d.y, d.z, 0.f);
  img[p] = 0x7f800000u;
}

// Distance used to step the tracing: the body's SDF; outside a GRID body's sampled box
// the distance to that box, at least eps.
__device__ __forceinline__ float march_sdf(const DevBody &b, float3 y, float eps) {
  int br;
  const float f = body_sdf(b, y, &br);
  if (b.kind != 4 || br >= 0) return f;
  const float yy[3] = {y.x, y.y, y.z};
  float q[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float lo = b.shape[k];
    const float hi = __fadd_rn(b.shape[k], __fmul_rn(b.shape[3], (float)(b.gn[k] - 1u)));
    q[k] = fmaxf(fmaxf(__fsub_rn(lo, yy[k]), __fsub_rn(yy[k], hi)), 0.0f);
  }
  const float s = __fadd_rn(__fadd_rn(__fmul_rn(q[0], q[0]), __fmul_rn(q[1], q[1])), __fmul_rn(q[2], q[2]));
  return fmaxf(__fsqrt_rn(s), eps);
}

__device__ __forceinline__ void splat_depth(const StepArgs &a, uint32_t off, uint32_t n, const RenderArgs &c, uint32_t i,
                                            uint32_t *img) {
  const float4 p = a.pos_id[off + (n - 1u - i)];
  const float oc0 = __fsub_rn(p.x, c.o[0]), oc1 = __fsub_rn(p.y, c.o[1]), oc2 = __fsub_rn(p.z, c.o[2]);
  const float rr = __fmul_rn(p.w, p.w);
  // conservative footprint from the centre in the camera frame (any rounding here
  // only widens or narrows the box by far less than the one-pixel margin)
  const float cx = c.R[0] * oc0 + c.R[3] * oc1 + c.R[6] * oc2;
  const float cy = c.R[1] * oc0 + c.R[4] * oc1 + c.R[7] * oc2;
  const float cz = c.R[2] * oc0 + c.R[5] * oc1 + c.R[8] * oc2;
  int u0 = 0, u1 = (int)c.W - 1, v0 = 0, v1 = (int)c.H - 1;
  if (cz - p.w > 0.5f * c.near) {
    const float zl = cz - p.w, zh = cz + p.w;
    const float xlo = fminf((cx - p.w) / zl, (cx - p.w) / zh), xhi = fmaxf((cx + p.w) / zl, (cx + p.w) / zh);
    const float ylo = fminf((cy - p.w) / zl, (cy - p.w) / zh), yhi = fmaxf((cy + p.w) / zl, (cy + p.w) / zh);
    u0 = max(u0, (int)floorf(c.f * xlo + 0.5f * c.W - 0.5f) - 1);
    u1 = min(u1, (int)ceilf(c.f * xhi + 0.5f * c.W - 0.5f) + 1);
    v0 = max(v0, (int)floorf(c.f * ylo + 0.5f * c.H - 0.5f) - 1);
    v1 = min(v1, (int)ceilf(c.f * yhi + 0.5f * c.H - 0.5f) + 1);
  } else if (cz + p.w <= 0.f) {
    return;  // entirely behind the camera
  }
  const float cc = __fsub_rn(__fadd_rn(__fadd_rn(__fmul_rn(oc0, oc0), __fmul_rn(oc1, oc1)), __fmul_rn(oc2, oc2)), rr);
  for (int v = v0; v <= v1; ++v)
    for (int u = u0; u <= u1; ++u) {
      const float4 d = c.rays[(size_t)v * c.W + u];
      const float b = __fadd_rn(__fadd_rn(__fmul_rn(d.x, oc0), __fmul_rn(d.y, oc1)), __fmul_rn(d.z, oc2));
      const float disc = __fsub_rn(__fmul_rn(b, b), cc);
      if (!(disc >= 0.0f)) continue;
      const float t0 = __fsub_rn(b, __fsqrt_rn(disc));
      if (!(t0 >= c.near && t0 <= c.far)) continue;
      atomicMin(&img[(size_t)v * c.W + u], __float_as_uint(t0));  // t0 > 0: bits order as floats
    }
}

// The spheres' and the bodies' depths of a pixel meet in its atomic, so both are made in one
// launch: the first blocks trace, the blocks after them splat the spheres meanwhile.  A traced
// ray is a chain of up to c.steps evaluations: that chain is what the launch takes, until the
// image fills the chip.  A ray ends where the spheres already block it (their depth is looked
// up every fourth step: it only falls, and a later hit would lie behind it).  Two forms, equal
// to the bit:
//  - k_depth: a block traces 32 pixels with a warp per body, so that a step's bodies are
//    evaluated side by side and without divergence between their kinds.  Every warp keeps the
//    state of all the block's pixels, so a step has one barrier (the distances are
//    double-buffered).  Shortens the chain: 36 x 36 rays past two bodies and 262,144 spheres
//    26.8 us, 32.9 in the other form; past eight 49 and 170.
//  - k_depth_pixels: a thread per pixel, the bodies in turn, no barrier.  Less work in all, so
//    it is the form of images that fill the chip: 640 x 480 past two bodies and 600,000 spheres
//    161 us, 255 in the other form.
// (As launches of their own, splat then trace: 47.3, 178 and 215 us.)
constexpr uint32_t kTraceBodies = 32;  // as many as the mask has bits

// Pixels up to which the bodies get a warp each.  The two forms cross between these sizes (us
// of the whole image, k_depth and k_depth_pixels): two bodies 320 x 200 (70-72, 74-78) and 512
// x 384 (91-119, 86-92), three 400 x 300 (45, 46), four to eight 640 x 480 (111-223, 140-273)
// and 1280 x 720 (253-572, 212-404), sixteen 640 x 480 (568, 591), 32 at 512 x 384 (1129, 1120).
// One body has nothing to share out.
__host__ __forceinline__ uint32_t warp_pixels(uint32_t bodies) {
  return bodies < 2u ? 0u : (bodies < 4u ? 100000u : std::min(400000u, 5500000u / bodies));
}

__device__ __forceinline__ float nearest_body(const StepArgs &a, uint32_t gb0, uint32_t nb, uint32_t mask, float3 x, float eps) {
  float fmin = __int_as_float(0x7f800000);
  for (uint32_t b = 0; b < nb; ++b) {
    if (!((mask >> b) & 1u)) continue;
    const DevBody &B = a.bodies[gb0 + b];
    fmin = fminf(fmin, march_sdf(B, world_to_body(B, x), eps));
  }
  return fmin;
}

constexpr int kDepthThreads = 128;
__global__ void __launch_bounds__(kDepthThreads) k_depth_pixels(StepArgs a, uint32_t off, uint32_t n, uint32_t gb0, uint32_t nb,
                                                                uint32_t tblocks, RenderArgs c, uint32_t *img) {
  pdl_enter();
  if (blockIdx.x >= tblocks) {
    const uint32_t i = (blockIdx.x - tblocks) * blockDim.x + threadIdx.x;
    if (i < n) splat_depth(a, off, n, c, i, img);
    return;
  }
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= c.W * c.H) return;
  const float4 d = c.rays[p];
  float t = c.near, seen = __int_as_float(0x7f800000);
  for (uint32_t k = 0; k < c.steps; ++k) {
    const float block_at = seen;
    if ((k & 3u) == 0u) seen = __uint_as_float(__ldcg(&img[p]));
    const float3 x = make_float3(__fadd_rn(c.o[0], __fmul_rn(t, d.x)), __fadd_rn(c.o[1], __fmul_rn(t, d.y)),
                                 __fadd_rn(c.o[2], __fmul_rn(t, d.z)));
    const float fmin = nearest_body(a, gb0, nb, c.mask, x, c.eps);
    if (fmin < c.eps) {
      atomicMin(&img[p], __float_as_uint(t));  // t >= near > 0
      return;
    }
    t = __fadd_rn(t, fmin);
    if (!(t <= c.far) || t >= block_at) return;
  }
}

__global__ void __launch_bounds__(32 * kTraceBodies) k_depth(StepArgs a, uint32_t off, uint32_t n, uint32_t gb0, uint32_t nb,
                                                             uint32_t tblocks, RenderArgs c, uint32_t *img) {
  pdl_enter();
  if (blockIdx.x >= tblocks) {
    const uint32_t i = (blockIdx.x - tblocks) * blockDim.x + threadIdx.x;
    if (i < n) splat_depth(a, off, n, c, i, img);
    return;
  }
  __shared__ float dist[2][kTraceBodies][32], block_at[2][32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t p = blockIdx.x * 32u + lane;
  const bool in = p < c.W * c.H;
  const bool mine = warp < nb && ((c.mask >> warp) & 1u);
  const DevBody B = a.bodies[gb0 + (warp < nb ? warp : 0u)];
  const float4 d = in ? c.rays[p] : make_float4(0.f, 0.f, 1.f, 0.f);
  const float inf = __int_as_float(0x7f800000);
  float t = c.near, hit = inf, seen = inf;
  bool live = in;
  for (uint32_t k = 0; k < c.steps && __any_sync(0xffffffffu, live); ++k) {
    const uint32_t h = k & 1u;
    float f = inf;
    if (live && mine) {
      const float3 x = make_float3(__fadd_rn(c.o[0], __fmul_rn(t, d.x)), __fadd_rn(c.o[1], __fmul_rn(t, d.y)),
                                   __fadd_rn(c.o[2], __fmul_rn(t, d.z)));
      f = march_sdf(B, world_to_body(B, x), c.eps);
    }
    dist[h][warp][lane] = f;
    if (warp == 0) {
      block_at[h][lane] = seen;
      if ((k & 3u) == 0u && in) seen = __uint_as_float(__ldcg(&img[p]));
    }
    __syncthreads();
    if (!live) continue;
    float fmin = dist[h][0][lane];
    for (uint32_t w = 1; w < nb; ++w) fmin = fminf(fmin, dist[h][w][lane]);
    if (fmin < c.eps) {
      hit = t;
      live = false;
    } else {
      t = __fadd_rn(t, fmin);
      if (!(t <= c.far) || t >= block_at[h][lane]) live = false;
    }
  }
  if (warp == 0 && in && hit < inf) atomicMin(&img[p], __float_as_uint(hit));  // hit >= near > 0
}

__global__ void k_finish_depth(const uint32_t *img, uint32_t count, float far, float *out) {
  pdl_enter();
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= count) return;
  const float best = __uint_as_float(img[p]);
  out[p] = best <= far ? best : far;
}

inline unsigned cdiv(uint32_t a, unsigned b) { return a ? (a + b - 1) / b : 1; }

}  // namespace

cudaError_t enqueue_render(const StepArgs &a, uint32_t env_off, uint32_t env_n, uint32_t gb0, uint32_t nb,
                           const RenderArgs &c, uint32_t *img, float *out, cudaStream_t st) {
  const uint32_t np = c.W * c.H;
  cudaError_t e;
  bool first = true;
#define GG_CHAIN(kern, count, block, ...)                                                        \
  do {                                                                                           \
    if ((e = launch(!first, kern, dim3(cdiv(count, block)), block, 0, st, __VA_ARGS__)) != cudaSuccess) return e; \
    first = false;                                                                               \
  } while (0)
  if (c.kind == 0) {
    GG_CHAIN(k_fill, np, 256, img, np, 0u);
    if (env_n) GG_CHAIN(k_splat_height, env_n, 128, a, env_off, env_n, c, img);
    GG_CHAIN(k_finish_height, np, 256, (const uint32_t *)img, np, c.empty, out);
  } else {
    GG_CHAIN(k_begin_depth, np, 128, c, img);
    const uint32_t nt = std::min(nb, kTraceBodies);
    // (of two bodies' four warps two only wait, but 64-thread blocks took 77 us where these take 70)
    const bool warps = np <= warp_pixels(nt);
    const unsigned threads = warps ? 32u * std::max(4u, nt) : (unsigned)kDepthThreads;
    const uint32_t tblocks = nt && c.mask ? cdiv(np, warps ? 32u : threads) : 0u;
    if (tblocks || env_n) {
      e = launch(true, warps ? k_depth : k_depth_pixels, dim3(tblocks + (env_n ? cdiv(env_n, threads) : 0u)), threads, 0, st, a, env_off, env_n, gb0,
                 nt, tblocks, c, img);
      if (e != cudaSuccess) return e;
    }
    GG_CHAIN(k_finish_depth, np, 128, (const uint32_t *)img, np, c.far, out);
  }
#undef GG_CHAIN
  return cudaGetLastError();
}

}  // namespace gg
