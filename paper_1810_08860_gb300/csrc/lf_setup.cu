// lf_setup.cu - per-view and per-triangle set-up kernels.
//
//   grid_tables_kernel   once per mesh build: per-view ray directions of the
//                        grid columns/rows, a_j = (j W/(G-1) - cx)/fx, b_k likewise.
//   view_setup_kernel    per call, one thread per (eye, view): FP64 composition
//                        of the view's camera->eye transform, its source
//                        projection, disk constants, and a conservative screen
//                        footprint of the disk, which is OR-ed into per-tile view
//                        masks (the culling of disks against the eye, Sec. 4.2.1).
//   cluster_bounds_kernel  once per mesh build: the depth range of every cluster
//                        of 4x4 cells.
//   tri_setup_kernel     per call, one CTA per (eye, view, part) with a non-empty
//                        footprint: clusters culled by their depth ranges, then
//                        vertex transform and 1/256-pixel snap, near clip, int64
//                        triangle set-up and footprint culling; it bins the view's
//                        triangles when the grid is one part.
//   bin_records_kernel, bin_scan_kernel  the binning of grids of several parts.
//
// Every float operation that feeds an integer decision (snapped position, depth
// winner, disk membership) uses explicit round-to-nearest intrinsics in a fixed
// order, so the decision is the same on any compiler setting.
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "lf_internal.h"
#include "lf_launch.h"
#include "lf_ray.h"

namespace lfk {

// ------------------------------------------------------------------ small helpers

__device__ __forceinline__ bool snap_rn(float x, float y, float z, float fx, float fy, float cx, float cy,
                                        int32_t& sx, int32_t& sy) {
  float qx = __fdiv_rn(x, z), qy = __fdiv_rn(y, z);
  float u = __fmaf_rn(fx, qx, cx), v = __fmaf_rn(fy, qy, cy);
  float su = __fmul_rn(u, 256.0f), sv = __fmul_rn(v, 256.0f);
  const float lim = (float)kSnapLimit;
  if (!(fabsf(su) < lim) || !(fabsf(sv) < lim)) return false;
  sx = __float2int_rn(su);  // |su| < 2^29: the 32-bit round-to-nearest-even conversion is exact
  sy = __float2int_rn(sv);
  return true;
}

// ------------------------------------------------------------------ grid tables

__global__ void grid_tables_kernel(const ViewStatic* __restrict__ views, int n_views, int src_w, int src_h,
                                   int G, float* __restrict__ a, float* __restrict__ b) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n_views * G) return;
  int v = (int)(idx / G), j = (int)(idx % G);
  const ViewStatic& V = views[v];
  double s = __ddiv_rn(__dmul_rn((double)j, (double)src_w), (double)(G - 1));
  double t = __ddiv_rn(__dmul_rn((double)j, (double)src_h), (double)(G - 1));
  a[idx] = __double2float_rn(__ddiv_rn(__dsub_rn(s, V.cx), V.fx));
  b[idx] = __double2float_rn(__ddiv_rn(__dsub_rn(t, V.cy), V.fy));
}

cudaError_t launch_grid_tables(const ViewStatic* views, int n_views, int src_w, int src_h, int G, float* a,
                               float* b, cudaStream_t s) {
  int64_t n = (int64_t)n_views * G;
  grid_tables_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(views, n_views, src_w, src_h, G, a, b);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ texture conversion

__global__ void convert_textures_kernel(const uchar4* __restrict__ src, void* __restrict__ dst, int64_t n,
                                        int fmt, const float* __restrict__ view_scale, int64_t per_view) {
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (; idx < n; idx += stride) {
    uchar4 c = src[idx];
    float r = __fdiv_rn((float)c.x, 255.0f), g = __fdiv_rn((float)c.y, 255.0f), bl = __fdiv_rn((float)c.z, 255.0f);
    if (fmt == LF_TEX_F32) {
      reinterpret_cast<float4*>(dst)[idx] = make_float4(r, g, bl, 1.0f);
    } else if (fmt == LF_TEX_BF16) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(r, g);
      __nv_bfloat162 hi = __floats2bfloat162_rn(bl, 1.0f);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo);
      pk.y = *reinterpret_cast<uint32_t*>(&hi);
      reinterpret_cast<uint2*>(dst)[idx] = pk;
    } else if (fmt == LF_TEX_FP8E4M3) {
      float inv = __frcp_rn(view_scale[idx / per_view]);
      __nv_fp8x4_e4m3 q(make_float4(__fmul_rn(r, inv), __fmul_rn(g, inv), __fmul_rn(bl, inv), 0.0f));
      reinterpret_cast<__nv_fp8x4_storage_t*>(dst)[idx] = q.__x;
    }
  }
}

cudaError_t launch_convert_textures(const uint8_t* src, void* dst, int64_t n_texels, int fmt,
                                    const float* view_scale, int64_t texels_per_view, cudaStream_t s) {
  int64_t blocks = (n_texels + 255) / 256;
  if (blocks > 152 * 64) blocks = 152 * 64;
  if (blocks < 1) blocks = 1;
  convert_textures_kernel<<<(unsigned)blocks, 256, 0, s>>>(reinterpret_cast<const uchar4*>(src), dst, n_texels,
                                                          fmt, view_scale, texels_per_view);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ per-view reductions

__global__ void view_scale_kernel(const uchar4* __restrict__ src, int64_t per_view, float* __restrict__ scale,
                                  ViewStatic* __restrict__ views) {
  __shared__ int s_max;
  if (threadIdx.x == 0) s_max = 1;
  __syncthreads();
  const uchar4* p = src + (int64_t)blockIdx.x * per_view;
  int m = 1;
  for (int64_t i = threadIdx.x; i < per_view; i += blockDim.x) {
    uchar4 c = p[i];
    m = max(m, max((int)c.x, max((int)c.y, (int)c.z)));
  }
  atomicMax(&s_max, m);
  __syncthreads();
  if (threadIdx.x == 0) {
    float sc = __fdiv_rn(__fdiv_rn((float)s_max, 255.0f), 448.0f);
    scale[blockIdx.x] = sc;
    views[blockIdx.x].tex_scale = sc;
  }
}

cudaError_t launch_view_scale(const uint8_t* rgba8, int n_views, int64_t per_view, float* scale, ViewStatic* views,
                              cudaStream_t s) {
  view_scale_kernel<<<n_views, 256, 0, s>>>(reinterpret_cast<const uchar4*>(rgba8), per_view, scale, views);
  return cudaGetLastError();
}

__global__ void depth_offsets_kernel(const float* __restrict__ depth, int per_view, __half* __restrict__ dst,
                                     ViewStatic* __restrict__ views) {
  __shared__ float s_min[256];
  const float* p = depth + (int64_t)blockIdx.x * per_view;
  float m = INFINITY;
  for (int i = threadIdx.x; i < per_view; i += blockDim.x) m = fminf(m, p[i]);
  s_min[threadIdx.x] = m;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) s_min[threadIdx.x] = fminf(s_min[threadIdx.x], s_min[threadIdx.x + o]);
    __syncthreads();
  }
  const float z0 = s_min[0];
  if (threadIdx.x == 0) views[blockIdx.x].depth_origin = z0;
  __half* q = dst + (int64_t)blockIdx.x * per_view;
  for (int i = threadIdx.x; i < per_view; i += blockDim.x) q[i] = __float2half_rn(__fsub_rn(p[i], z0));
}

cudaError_t launch_depth_offsets(const float* depth, int n_views, int per_view, void* dst_half, ViewStatic* views,
                                 cudaStream_t s) {
  depth_offsets_kernel<<<n_views, 256, 0, s>>>(depth, per_view, static_cast<__half*>(dst_half), views);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ view set-up

// Range of x/z over forward rays (z > 0) that meet a ball of radius rho whose
// centre projects to (c, cz) in the plane of one image axis and the optical
// axis: the directions within asin(rho/L) of the centre's direction, clipped to
// the forward half-plane.  Returns false when no forward ray meets it; an
// infinite bound is returned as +-inf.  FP32 is enough: the caller pads the
// ball and the pixel range, and the result only culls.
__device__ bool axis_extent(float c, float cz, float rho, float& lo, float& hi) {
  const float half_pi = 1.57079632679f;
  const float L2 = c * c + cz * cz;
  if (L2 <= rho * rho * 1.0001f) {  // the eye's projection lies inside the ball's
    lo = -INFINITY;
    hi = INFINITY;
    return true;
  }
  const float th = atan2f(c, cz), de = asinf(fminf(1.0f, rho * rsqrtf(L2)) ) + 1e-5f;
  const float a = fmaxf(th - de, -half_pi), b = fminf(th + de, half_pi);
  if (!(a < b)) return false;
  lo = (a <= -half_pi + 1e-4f) ? -INFINITY : tanf(a);
  hi = (b >= half_pi - 1e-4f) ? INFINITY : tanf(b);
  return true;
}

// Pixel-index range [i0, i1] whose centres' x/z lies in [lo, hi], padded by two pixels.
__device__ void pixel_range(float lo, float hi, float f, float c, int n, int& i0, int& i1) {
  const float u0 = f * lo + c, u1 = f * hi + c;
  i0 = (int)fmaxf(-1.0f, fminf((float)n, floorf(u0 - 0.5f) - 2.0f));
  i1 = (int)fmaxf(-1.0f, fminf((float)n, ceilf(u1 - 0.5f) + 2.0f));
}

constexpr int kViewsPerSetupBlock = 16;
constexpr int kViewSetupThreads = 128;
constexpr int kViewSetupSlices = 8;  // blocks sharing one group of views' (view, tile) cone tests

// Two-level frames, round disks: a first look at which views an eye selects, 64 pixels
// spread over each view's footprint (the block's slice takes two views).  What it finds
// is exact; the views it misses are left to select_kernel, which tests every pixel of
// the tiles that may see them.  With it select_kernel takes 9 us of a 2 x 1440x1600
// frame of 640 views instead of 85.
__device__ void mark_visible(const FrameArgs& A, const EyeParams& E, const EyeFloat& F, int e, int v0, const int4* s_bb) {
  constexpr int kPer = kViewsPerSetupBlock / kViewSetupSlices, kLanes = kViewSetupThreads / kPer;  // 2 views, 64 pixels
  const int k = blockIdx.z * kPer + threadIdx.x / kLanes, q = threadIdx.x % kLanes, v = v0 + k;
  if (v >= A.n_views) return;
  const int4 bb = s_bb[k];
  if (bb.x > bb.z || bb.y > bb.w) return;
  const int x = bb.x + (int)((int64_t)(2 * (q & 7) + 1) * (bb.z - bb.x + 1) / 16);
  const int y = bb.y + (int)((int64_t)(2 * (q >> 3) + 1) * (bb.w - bb.y + 1) / 16);
  float p[3];
  sphere_crossing(F.ray, F.centre, ray_slope(x, F.cx, F.fx), ray_row(F, ray_slope(y, F.cy, F.fy)), p);
  const ViewStatic& V = A.views[v];
  const float4 cc = make_float4(__double2float_rn(__dsub_rn((double)V.disk_c[0], A.sphere_c[0])),
                                __double2float_rn(__dsub_rn((double)V.disk_c[1], A.sphere_c[1])),
                                __double2float_rn(__dsub_rn((double)V.disk_c[2], A.sphere_c[2])),
                                __fmul_rn(V.disk_r, V.disk_r));
  if (disk_d2(cc, p) < cc.w) A.visible[(int64_t)e * A.n_views + v] = 1;
}

// A block takes 16 views of one eye.  Threads 0-15 do the per-view set-up
// (FP64 composition, FP32 shading map and disk constants, conservative
// footprint); then all threads test every (view, tile) pair of the block's
// footprints and OR the view's bit into the masks of the tiles it can reach.
// The tile test compares cones from the eye: a pixel whose sphere crossing
// lies in the disk has its ray within asin(rho/|c|) of the direction to the
// disk centre c, and every pixel ray of a tile lies within (half diagonal)/f
// of the tile's centre ray (rays through image points s apart differ by at
// most s/f in angle), so a tile is skipped only when the two cones are apart.
__global__ void __launch_bounds__(kViewSetupThreads) view_setup_kernel(FrameArgs A, const __grid_constant__ InlineEyes given) {
  __shared__ float s_dir[kViewsPerSetupBlock][4];   // unit direction to the disk centre, cos of the cone limit
  __shared__ int s_off[kViewsPerSetupBlock + 1];   // exclusive prefix of the footprints' tile counts
  __shared__ int s_tile[kViewsPerSetupBlock][3];    // footprint: first tile column and row, tile columns
  __shared__ int4 s_tile_bb[kViewsPerSetupBlock];   // footprint in pixels
  const int e = blockIdx.y;
  const int v0 = blockIdx.x * kViewsPerSetupBlock;
  const EyeParams& E = given.n ? given.eye[e] : A.eyes[e];
  if (given.n && blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x == 64) A.eyes[e] = given.eye[e];
  const float tile_half_diag = 0.5f * sqrtf((float)(A.tile_w * A.tile_w + A.tile_h * A.tile_h));
  const float alpha_tile = tile_half_diag / fminf((float)E.fx, (float)E.fy);
  const bool writer = blockIdx.z == 0;  // the other slices only share the cone tests
  // Triangle set-up may launch now: it waits for this grid to complete before
  // it reads anything the grid writes.
  griddep_wait();
  griddep_release();
  if (writer && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    // the frame's counters start at zero (no kernel before this one uses them)
    *A.pool_counter = 0ull;
    *A.error_word = 0u;
    *A.work_counter = 0;
    *A.bin_offsets_counter = 0ull;
    *A.bin_entries_counter = 0ull;
  }
  // the eye's FP32 decision constants, each rounded once from FP64 (every block for itself: its share of the ray tables)
  __shared__ EyeFloat F;
  if (threadIdx.x >= 32 && threadIdx.x < 32 + 16) {
    const int k = threadIdx.x - 32;
    if (k < 9) F.R[k] = __double2float_rn(E.R[k]);
    else if (k < 12) F.o[k - 9] = __double2float_rn(__dsub_rn(E.t[k - 9], A.sphere_c[k - 9]));
    else (&F.fx)[k - 12] = __double2float_rn((&E.fx)[k - 12]);
    __syncwarp(0xffffu);
    if (k == 0) {
      const float R2 = __double2float_rn(__dmul_rn(A.sphere_r, A.sphere_r));
      F.ray = make_float4(F.R[0], F.R[3], F.R[6],
                          __fsub_rn(dot3_rn(F.o[0], F.o[1], F.o[2], F.o[0], F.o[1], F.o[2]), R2));
      F.centre = make_float4(F.o[0], F.o[1], F.o[2], 0.0f);
      if (writer && blockIdx.x == 0) A.eyes_f[e] = F;
    }
  }
  int n_tiles = 0;  // tiles of this thread's view's footprint (threads 0-15)
  if (threadIdx.x < kViewsPerSetupBlock) {
    const int v = v0 + threadIdx.x;
    int bb[4] = {1, 1, 0, 0};
    float dir[4] = {0.f, 0.f, 1.f, 2.f};
    if (v < A.n_views) {
      const ViewStatic& V = A.views[v];
      if (writer) {
      A.active[(int64_t)e * A.n_views + v] = 0;  // set by the raster when a pixel sees the view
      ViewRec& R = A.vrecs[(int64_t)e * A.n_views + v];
      // A1: M = R_eye^T R_i, m = R_eye^T (t_i - t_eye) in FP64, fixed order, no fusion.
      double M[9], m[3];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          double s = __dmul_rn(E.R[0 * 3 + r], V.R[0 * 3 + c]);
          s = __dadd_rn(s, __dmul_rn(E.R[1 * 3 + r], V.R[1 * 3 + c]));
          s = __dadd_rn(s, __dmul_rn(E.R[2 * 3 + r], V.R[2 * 3 + c]));
          M[r * 3 + c] = s;
        }
      const double d[3] = {__dsub_rn(V.t[0], E.t[0]), __dsub_rn(V.t[1], E.t[1]), __dsub_rn(V.t[2], E.t[2])};
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        double s = __dmul_rn(E.R[0 * 3 + r], d[0]);
        s = __dadd_rn(s, __dmul_rn(E.R[1 * 3 + r], d[1]));
        s = __dadd_rn(s, __dmul_rn(E.R[2 * 3 + r], d[2]));
        m[r] = s;
      }
      float Mc[9], mc[3];
#pragma unroll
      for (int k = 0; k < 9; ++k) R.Mf[k] = Mc[k] = __double2float_rn(M[k]);
#pragma unroll
      for (int k = 0; k < 3; ++k) R.Mf[9 + k] = mc[k] = __double2float_rn(m[k]);

      // Source projection for shading: h = K_i' M^T (Kinv_e [x, y, 1] - m / z), with
      // K_i' using (cx - 1/2, cy - 1/2) so h.x/h.z is the bilinear coordinate u = s - 1/2.
      // FP32 from the composition: it only places texture samples.
      const float Ki[9] = {(float)V.fx, 0.f, (float)(V.cx - 0.5), 0.f, (float)V.fy, (float)(V.cy - 0.5),
                           0.f, 0.f, 1.f};
      const float ifx = 1.0f / (float)E.fx, ify = 1.0f / (float)E.fy;
      const float Ke[9] = {ifx, 0.f, -(float)E.cx * ifx, 0.f, ify, -(float)E.cy * ify, 0.f, 0.f, 1.f};
      float KM[9];  // Ki M^T
      for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
          KM[r * 3 + c] = Ki[r * 3 + 0] * Mc[c * 3 + 0] + Ki[r * 3 + 1] * Mc[c * 3 + 1] + Ki[r * 3 + 2] * Mc[c * 3 + 2];
      for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c)
          R.Hm[r][c] = KM[r * 3 + 0] * Ke[0 * 3 + c] + KM[r * 3 + 1] * Ke[1 * 3 + c] + KM[r * 3 + 2] * Ke[2 * 3 + c];
        R.Hm[r][3] = -(KM[r * 3 + 0] * mc[0] + KM[r * 3 + 1] * mc[1] + KM[r * 3 + 2] * mc[2]);
      }

      // Disk (Sec. 4.1): centre relative to the sphere centre in FP32, r^2.
      for (int k = 0; k < 3; ++k) R.cc[k] = __double2float_rn(__dsub_rn((double)V.disk_c[k], A.sphere_c[k]));
      R.cc[3] = __fmul_rn(V.disk_r, V.disk_r);
      R.inv_r = __frcp_rn(V.disk_r);
      R.tex_scale = V.tex_scale;
      if (A.disk_mode == 1) {
        // Oval disk (Sec. 4.4): its plane's normal and axes are the columns of M; the
        // centre in the eye frame and the dot products in FP64, fixed order, each
        // rounded once.
        const double dcw[3] = {__dsub_rn((double)V.disk_c[0], E.t[0]), __dsub_rn((double)V.disk_c[1], E.t[1]),
                               __dsub_rn((double)V.disk_c[2], E.t[2])};
        double cp[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          double s = __dmul_rn(E.R[0 * 3 + r], dcw[0]);
          s = __dadd_rn(s, __dmul_rn(E.R[1 * 3 + r], dcw[1]));
          s = __dadd_rn(s, __dmul_rn(E.R[2 * 3 + r], dcw[2]));
          cp[r] = s;
        }
        auto dotc = [&](int col) {
          return __dadd_rn(__dadd_rn(__dmul_rn(M[0 * 3 + col], cp[0]), __dmul_rn(M[1 * 3 + col], cp[1])),
                           __dmul_rn(M[2 * 3 + col], cp[2]));
        };
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          R.ov[k] = Mc[k * 3 + 2];      // n
          R.ov[3 + k] = Mc[k * 3 + 0];  // x
          R.ov[6 + k] = Mc[k * 3 + 1];  // y
        }
        R.ov[9] = __double2float_rn(dotc(2));
        R.ov[10] = __double2float_rn(dotc(0));
        R.ov[11] = __double2float_rn(dotc(1));
        R.ov[12] = __double2float_rn(__ddiv_rn(1.0, (double)V.disk_ext[0]));
        R.ov[13] = __double2float_rn(__ddiv_rn(1.0, (double)V.disk_ext[1]));
        R.ov[14] = __double2float_rn(__ddiv_rn(1.0, (double)V.disk_ext[2]));
        R.ov[15] = __double2float_rn(__ddiv_rn(1.0, (double)V.disk_ext[3]));
      }
      // the view's texels: its page in a two-level frame, else its slice of the texture array
      const int tb = A.tex_format == LF_TEX_F32 ? 16 : A.tex_format == LF_TEX_BF16 ? 8 : 4;
      R.tex = A.tex_table ? A.tex_table[v]
                          : static_cast<const char*>(A.textures) + (int64_t)v * A.src_w * A.src_h * tb;
      R.parts_done = 0;
      R.bin_off = -1;
      R.big_base = 0;
      R.big_count = 0;
      R.tri_count = 0;
      }

      // Conservative footprint: a pixel whose sphere crossing can fall inside the
      // disk has a forward ray passing within r of c_i, so it lies in the screen
      // extent of the ball of radius r (padded) about c_i.
      float cw[3], ce[3];
      for (int k = 0; k < 3; ++k) cw[k] = (float)((double)V.disk_c[k] - E.t[k]);
      for (int r = 0; r < 3; ++r)
        ce[r] = (float)E.R[0 * 3 + r] * cw[0] + (float)E.R[1 * 3 + r] * cw[1] + (float)E.R[2 * 3 + r] * cw[2];
      // an oval lies in the disk of its largest extent about c_i, in its plane
      const float r_out = A.disk_mode == 1 ? fmaxf(fmaxf(V.disk_ext[0], V.disk_ext[1]),
                                                    fmaxf(V.disk_ext[2], V.disk_ext[3]))
                                           : V.disk_r;
      const float rho = r_out * 1.001f + 1e-4f;
      float xlo, xhi, ylo, yhi;
      if (axis_extent(ce[0], ce[2], rho, xlo, xhi) && axis_extent(ce[1], ce[2], rho, ylo, yhi)) {
        int x0, x1, y0, y1;
        pixel_range(xlo, xhi, (float)E.fx, (float)E.cx, E.W, x0, x1);
        pixel_range(ylo, yhi, (float)E.fy, (float)E.cy, E.H, y0, y1);
        x0 = max(x0, 0); y0 = max(y0, 0);
        x1 = min(x1, E.W - 1); y1 = min(y1, E.H - 1);
        if (x0 <= x1 && y0 <= y1) { bb[0] = x0; bb[1] = y0; bb[2] = x1; bb[3] = y1; }
      }
      if (writer) {
        ViewRec& R = A.vrecs[(int64_t)e * A.n_views + v];
        R.bb[0] = bb[0]; R.bb[1] = bb[1]; R.bb[2] = bb[2]; R.bb[3] = bb[3];
      }
      // cone of the ball seen from the eye, widened by a tile's angular radius
      const float L = sqrtf(ce[0] * ce[0] + ce[1] * ce[1] + ce[2] * ce[2]);
      if (L > rho) {
        const float lim = asinf(rho / L) + alpha_tile + 1e-4f;
        dir[0] = ce[0] / L; dir[1] = ce[1] / L; dir[2] = ce[2] / L;
        dir[3] = lim < 3.14159f ? cosf(lim) : -2.0f;
      } else {
        dir[3] = -2.0f;  // the eye is inside the ball: every tile of the footprint
      }
    }
    for (int k = 0; k < 4; ++k) s_dir[threadIdx.x][k] = dir[k];
    s_tile_bb[threadIdx.x] = make_int4(bb[0], bb[1], bb[2], bb[3]);
    int tx0 = 0, ty0 = 0, ntx = 1;
    if (bb[0] <= bb[2] && bb[1] <= bb[3]) {
      tx0 = bb[0] / A.tile_w;
      ty0 = bb[1] / A.tile_h;
      ntx = bb[2] / A.tile_w - tx0 + 1;
      n_tiles = ntx * (bb[3] / A.tile_h - ty0 + 1);
    }
    s_tile[threadIdx.x][0] = tx0;
    s_tile[threadIdx.x][1] = ty0;
    s_tile[threadIdx.x][2] = ntx;
  }
  // the footprints' tile counts, scanned by warp 0 (which holds threads 0-15)
  if (threadIdx.x < 32) {
    int incl = n_tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if ((int)threadIdx.x >= o) incl += y;
    }
    if (threadIdx.x < kViewsPerSetupBlock) s_off[threadIdx.x] = incl - n_tiles;
    if (threadIdx.x == kViewsPerSetupBlock - 1) s_off[kViewsPerSetupBlock] = incl;
  }
  __syncthreads();
  // the eye's ray tables, shared by all its blocks: the raster reads a column's slope and a row's terms instead of
  // dividing for every pixel
  {
    const int step = gridDim.x * gridDim.z * kViewSetupThreads;
    for (int i = (blockIdx.z * gridDim.x + blockIdx.x) * kViewSetupThreads + threadIdx.x; i < E.W + E.H; i += step) {
      if (i < E.W) A.ray_cols[4 * (int64_t)E.line_base + i] = ray_slope(i, F.cx, F.fx);
      else A.ray_rows[(int64_t)E.line_base + i - E.W] = ray_row(F, ray_slope(i - E.W, F.cy, F.fy));
    }
  }
  if (A.visible && A.disk_mode == 0) mark_visible(A, E, F, e, v0, s_tile_bb);
  const int total = s_off[kViewsPerSetupBlock];
  const float fx = (float)E.fx, fy = (float)E.fy, cx = (float)E.cx, cy = (float)E.cy;
  for (int f = threadIdx.x + blockIdx.z * kViewSetupThreads; f < total; f += kViewSetupThreads * kViewSetupSlices) {
    int k = 0;  // the view whose range [s_off[k], s_off[k + 1]) holds f
#pragma unroll
    for (int step = kViewsPerSetupBlock / 2; step > 0; step >>= 1)
      if (s_off[k + step] <= f) k += step;
    const int q = f - s_off[k];
    const int ntx = s_tile[k][2];
    const int tx = s_tile[k][0] + q % ntx, ty = s_tile[k][1] + q / ntx;
    // centre ray of the tile's pixel-centre rectangle
    const float xc = (float)(tx * A.tile_w) + 0.5f * (float)(A.tile_w - 1) + 0.5f;
    const float yc = (float)(ty * A.tile_h) + 0.5f * (float)(A.tile_h - 1) + 0.5f;
    const float rx = (xc - cx) / fx, ry = (yc - cy) / fy;
    const float inv = rsqrtf(rx * rx + ry * ry + 1.0f);
    const float cosang = (rx * s_dir[k][0] + ry * s_dir[k][1] + s_dir[k][2]) * inv;
    if (cosang < s_dir[k][3]) continue;
    const int v = v0 + k;
    const int64_t tile = (int64_t)E.tile_base + (int64_t)ty * E.tiles_x + tx;
    atomicOr(&A.tile_masks[tile * A.mask_words + (v >> 5)], 1u << (v & 31));
  }
}

cudaError_t launch_view_setup(const FrameArgs& a, const InlineEyes& eyes, cudaStream_t s) {
  dim3 grid((a.n_views + kViewsPerSetupBlock - 1) / kViewsPerSetupBlock, a.n_eyes, kViewSetupSlices);
  view_setup_kernel<<<grid, kViewSetupThreads, 0, s>>>(a, eyes);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ cluster depth bounds

// Per view and cluster of kClusterCells^2 mesh cells: the smallest and largest
// depth of its vertices, once per mesh build.  A warp per cluster.
__global__ void cluster_bounds_kernel(const void* __restrict__ depth, int mesh_format,
                                      const ViewStatic* __restrict__ views, int G, int ncl, int64_t n_clusters,
                                      float2* __restrict__ out) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_clusters) return;
  const int64_t v = w / (ncl * ncl);
  const int c = (int)(w - v * ncl * ncl), cy = c / ncl, cx = c - cy * ncl;
  float lo = INFINITY, hi = -INFINITY;
  if (lane < 25) {
    const int k = min(cy * kClusterCells + lane / 5, G - 1), j = min(cx * kClusterCells + lane % 5, G - 1);
    const int64_t gi = (v * G + k) * G + j;
    const float z = mesh_format == LF_MESH_F16_OFFSET
                        ? __fadd_rn(views[v].depth_origin, __half2float(reinterpret_cast<const __half*>(depth)[gi]))
                        : reinterpret_cast<const float*>(depth)[gi];
    lo = hi = z;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) out[w] = make_float2(lo, hi);
}

cudaError_t launch_cluster_bounds(const void* depth, int mesh_format, const ViewStatic* views, int n_views, int G,
                                  float2* out, cudaStream_t s) {
  const int ncl = clusters_per_side(G);
  const int64_t n = (int64_t)n_views * ncl * ncl;
  cluster_bounds_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(depth, mesh_format, views, G, ncl, n, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ triangle set-up

constexpr uint32_t kOcBehind = 16;  // outcode: bit0..3 left/right/above/below the padded footprint, bit4 behind z_near
constexpr uint32_t kOcFar = 32;     // in front of it, but its snapped coordinates leave the 32-bit range: its triangles are dropped

struct SetupCtx {
  float fx, fy, cx, cy, zn;
  int bb0, bb1, bb2, bb3;
};

// Orient, classify and bound one snapped sub-triangle; false if culled.  The
// coordinates are below kSnapLimit, so differences and boxes are 32-bit; only the
// area needs 64.
__device__ __forceinline__ bool setup_sub(const int32_t* sx, const int32_t* sy, const SetupCtx& C, TriRec& t,
                                          int32_t& tl) {
  static_assert((int64_t)kSnapLimit + 256 < (int64_t)1 << 30, "differences of snapped coordinates fit 32 bits");
  const int32_t X0 = sx[0], Y0 = sy[0];
  const int64_t area = (int64_t)(sx[1] - X0) * (sy[2] - Y0) - (int64_t)(sy[1] - Y0) * (sx[2] - X0);
  if (area == 0) return false;
  const bool turn = area < 0;
  const int32_t X1 = turn ? sx[2] : sx[1], Y1 = turn ? sy[2] : sy[1];
  const int32_t X2 = turn ? sx[1] : sx[2], Y2 = turn ? sy[1] : sy[2];
  // the pixel centres of its box: the first at or after the least coordinate, the last at or before the greatest
  const int32_t i0 = max((min(X0, min(X1, X2)) + 127) >> 8, C.bb0), i1 = min((max(X0, max(X1, X2)) - 128) >> 8, C.bb2);
  const int32_t j0 = max((min(Y0, min(Y1, Y2)) + 127) >> 8, C.bb1), j1 = min((max(Y0, max(Y1, Y2)) - 128) >> 8, C.bb3);
  if (i0 > i1 || j0 > j1) return false;
  t.bx0 = (int16_t)i0; t.by0 = (int16_t)j0; t.bx1 = (int16_t)i1; t.by1 = (int16_t)j1;
  t.x[0] = X0; t.y[0] = Y0;
  t.x[1] = X1; t.y[1] = Y1;
  t.x[2] = X2; t.y[2] = Y2;
  const int32_t X[3] = {X0, X1, X2}, Y[3] = {Y0, Y1, Y2};
  tl = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3;
    const bool f = (Y[k] == Y[k1] && X[k1] > X[k]) || (Y[k1] < Y[k]);
    tl |= (int)f << k;
  }
  return true;
}

// A vertex in eye space.
struct EyeVtx {
  float x, y, z;
};

// A parent's FP32 inverse-depth plane (original vertex order, fixed order); false if it has none.
__device__ __forceinline__ bool setup_plane(const EyeVtx& v0, const EyeVtx& v1, const EyeVtx& v2, TriRec& t) {
  const float e1x = __fsub_rn(v1.x, v0.x), e1y = __fsub_rn(v1.y, v0.y), e1z = __fsub_rn(v1.z, v0.z);
  const float e2x = __fsub_rn(v2.x, v0.x), e2y = __fsub_rn(v2.y, v0.y), e2z = __fsub_rn(v2.z, v0.z);
  const float nx = __fsub_rn(__fmul_rn(e1y, e2z), __fmul_rn(e1z, e2y));
  const float ny = __fsub_rn(__fmul_rn(e1z, e2x), __fmul_rn(e1x, e2z));
  const float nz = __fsub_rn(__fmul_rn(e1x, e2y), __fmul_rn(e1y, e2x));
  const float dd = dot3_rn(nx, ny, nz, v0.x, v0.y, v0.z);
  t.ia = __fdiv_rn(nx, dd); t.ib = __fdiv_rn(ny, dd); t.ic = __fdiv_rn(nz, dd);
  return dd != 0.0f && isfinite(t.ia) && isfinite(t.ib) && isfinite(t.ic);
}

// The snapped polygon of a parent triangle that crosses the near plane: np
// vertices (0: dropped, 3, or 4: two sub-triangles, a fan from the first kept
// vertex).  The decisions (snap, clip) are taken exactly as the oracle takes them.
struct SetupPoly {
  int32_t px[4], py[4];
  int np;
};

__device__ __forceinline__ void clip_poly(const EyeVtx& v0, const EyeVtx& v1, const EyeVtx& v2, uint32_t o0,
                                          uint32_t o1, uint32_t o2, const SetupCtx& C, SetupPoly& P) {
  P.np = 0;
  // Sutherland-Hodgman against z >= z_near, walking v0 -> v1 -> v2 -> v0.
  const float vx[3] = {v0.x, v1.x, v2.x}, vy[3] = {v0.y, v1.y, v2.y}, vz[3] = {v0.z, v1.z, v2.z};
  const bool in[3] = {(o0 & kOcBehind) == 0, (o1 & kOcBehind) == 0, (o2 & kOcBehind) == 0};
  int np = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3;
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // the vertex if it is in front, then the crossing of the edge
      float ix = vx[k], iy = vy[k], iz = vz[k];
      if (h == 0 ? !in[k] : in[k] == in[k1]) continue;
      if (h == 1) {
        const float tt = __fdiv_rn(__fsub_rn(C.zn, vz[k]), __fsub_rn(vz[k1], vz[k]));
        ix = __fmaf_rn(tt, __fsub_rn(vx[k1], vx[k]), vx[k]);
        iy = __fmaf_rn(tt, __fsub_rn(vy[k1], vy[k]), vy[k]);
        iz = C.zn;
      }
      int32_t sx, sy;
      if (!snap_rn(ix, iy, iz, C.fx, C.fy, C.cx, C.cy, sx, sy)) return;
#pragma unroll
      for (int i = 0; i < 4; ++i)  // static indexes keep the polygon in registers
        if (i == np) { P.px[i] = sx; P.py[i] = sy; }
      ++np;
    }
  }
  P.np = np;
}

// Block-wide exclusive scan of small non-negative counts (blockDim.x multiple of 32).
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  int base = 0;
  total = 0;
  for (int w = 0; w < nw; ++w) {
    int c = s_warp[w];
    if (w < warp) base += c;
    total += c;
  }
  __syncthreads();
  return base + x - v;
}

// ------------------------------------------------------------------ binning

// A view's set-up triangles are binned into the screen tiles of its footprint
// box: per tile the bin holds the pool indices of the triangles whose pixel box
// overlaps it, in no particular order (the per-view depth decision does not
// depend on order).  Offsets and cursors live in the offset pool: [ntiles + 1
// absolute entry offsets][ntiles cursors].

struct TileBox {
  int tx0, ty0, ntx, nty;
  int sw, sh;  // log2 of the tile's width and height (8, 16 or 32)
};

__device__ __forceinline__ TileBox footprint_tiles(const int32_t* bb, int tw, int th) {
  TileBox b;
  b.sw = __ffs(tw) - 1;
  b.sh = __ffs(th) - 1;
  b.tx0 = bb[0] >> b.sw;
  b.ty0 = bb[1] >> b.sh;
  b.ntx = (bb[2] >> b.sw) - b.tx0 + 1;
  b.nty = (bb[3] >> b.sh) - b.ty0 + 1;
  return b;
}

// The tiles of the box (relative to it) that a record's pixel box overlaps.
// Shifts, not divisions: set-up of the stereo rig 25 -> 22 us.
struct RecordTiles {
  int x0, y0, x1, y1;
};
__device__ __forceinline__ RecordTiles record_tiles(int2 bb, const TileBox& b) {
  return {max(((int)(int16_t)(bb.x & 0xffff) >> b.sw) - b.tx0, 0), max((bb.x >> (16 + b.sh)) - b.ty0, 0),
          min(((int)(int16_t)(bb.y & 0xffff) >> b.sw) - b.tx0, b.ntx - 1), min((bb.y >> (16 + b.sh)) - b.ty0, b.nty - 1)};
}
// f(tile) for each of them; returns false, without calling f, when they are more than max_tiles.
template <typename F>
__device__ __forceinline__ bool for_record_tiles(int2 bb, const TileBox& b, int max_tiles, F&& f) {
  const RecordTiles t = record_tiles(bb, b);
  if (t.x0 > t.x1 || t.y0 > t.y1) return true;
  if ((t.x1 - t.x0 + 1) * (t.y1 - t.y0 + 1) > max_tiles) return false;
  for (int y = t.y0; y <= t.y1; ++y)
    for (int x = t.x0; x <= t.x1; ++x) f(y * b.ntx + x);
  return true;
}

// One thread: room for a view's offsets and cursors; -1 (and the error bit) when there is none.
__device__ long long take_offsets(const FrameArgs& A, int nt) {
  const unsigned long long o = atomicAdd(A.bin_offsets_counter, (unsigned long long)(2 * nt + 1));
  if ((long long)o + 2 * nt + 1 <= A.bin_offsets_capacity) return (long long)o;
  atomicOr(A.error_word, kErrPoolOverflow);
  return -1;
}

__device__ long long take_entries(const FrameArgs& A, int need) {
  const unsigned long long b = atomicAdd(A.bin_entries_counter, (unsigned long long)need);
  if ((long long)b + need <= A.bin_entries_capacity) return (long long)b;
  atomicOr(A.error_word, kErrPoolOverflow);
  return -1;
}

// Counts -> absolute offsets (offs, nt + 1 of them) and cursors (cnt, in place)
// by one block; `extra` entries follow the bins.  Returns the first entry, or -1
// when the entry pool is full.
template <int BLOCK>
__device__ long long scan_bins(const FrameArgs& A, int* cnt, int* offs, int nt, int extra, int* s_warp, int& total) {
  __shared__ long long s_ent;
  const int per = (nt + BLOCK - 1) / BLOCK;  // each thread owns a contiguous run
  const int r0 = threadIdx.x * per, r1 = min(r0 + per, nt);
  int run = 0;
  for (int k = r0; k < r1; ++k) run += cnt[k];
  int o = block_exclusive_scan(run, s_warp, total);
  if (threadIdx.x == 0) s_ent = take_entries(A, total + extra);
  __syncthreads();
  const long long ent = s_ent;
  if (ent < 0) return -1;
  for (int k = r0; k < r1; ++k) {
    const int c = cnt[k];
    offs[k] = (int)(ent + o);
    cnt[k] = (int)(ent + o);
    o += c;
  }
  if (threadIdx.x == 0) offs[nt] = (int)(ent + total);
  return ent;
}

// Bins one view's records, the n_ranges ranges (first pool index, count <= 32)
// its block has just written; a warp takes a range.  Triangles whose box spans
// more than A.bin_max_tiles tiles go to the view's list of big ones, which every
// tile of the view scans (only the static-scratch render caps it).  The per-tile
// counts and cursors use `cnt` (cnt_cap ints of shared memory) when the
// footprint fits, else the pool's cursor half.
template <int BLOCK>
__device__ void bin_view(const FrameArgs& A, ViewRec& R, const int2* ranges, int n_ranges, int* cnt_smem, int cnt_cap,
                         int* s_warp) {
  __shared__ long long s_off;
  __shared__ int s_big;
  constexpr int NW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tw = A.tile_w, th = A.tile_h;
  const TileBox tb = footprint_tiles(R.bb, tw, th);
  const int nt = tb.ntx * tb.nty;
  if (threadIdx.x == 0) {
    s_off = take_offsets(A, nt);
    s_big = 0;
  }
  __syncthreads();
  if (s_off < 0) return;
  int* offs = A.bin_offsets + s_off;
  int* curs = offs + nt + 1;
  int* cnt = nt <= cnt_cap ? cnt_smem : curs;  // counts, then cursors
  for (int k = threadIdx.x; k < nt; k += BLOCK) cnt[k] = 0;
  __syncthreads();
  int my_big = 0;
  for (int r = warp; r < n_ranges; r += NW) {
    if (lane >= ranges[r].y) continue;
    const int2 bb = *reinterpret_cast<const int2*>(A.pool + ranges[r].x + lane);
    if (!for_record_tiles(bb, tb, A.bin_max_tiles, [&](int tile) { atomicAdd(&cnt[tile], 1); })) ++my_big;
  }
  if (my_big) atomicAdd(&s_big, my_big);
  __syncthreads();
  int total;
  const long long ent = scan_bins<BLOCK>(A, cnt, offs, nt, s_big, s_warp, total);
  if (ent < 0) return;
  __syncthreads();
  if (threadIdx.x == 0) s_big = 0;
  __syncthreads();
  const int big_base = (int)(ent + total);
  for (int r = warp; r < n_ranges; r += NW) {
    if (lane >= ranges[r].y) continue;
    const int idx = ranges[r].x + lane;
    const int2 bb = *reinterpret_cast<const int2*>(A.pool + idx);
    if (!for_record_tiles(bb, tb, A.bin_max_tiles, [&](int tile) { A.bin_entries[atomicAdd(&cnt[tile], 1)] = idx; }))
      A.bin_entries[big_base + atomicAdd(&s_big, 1)] = idx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    R.bin_off = (int32_t)s_off;
    R.btx0 = (int16_t)tb.tx0; R.bty0 = (int16_t)tb.ty0;
    R.bntx = (int16_t)tb.ntx; R.bnty = (int16_t)tb.nty;
    R.big_base = big_base;
    R.big_count = s_big;
  }
}

constexpr int kSetupBlock = 256;
constexpr int kPartClusters = kSetupPartClusters;
static_assert(kPartClusters <= kSetupBlock, "one thread per cluster in the first cull");
// A view of one part takes 512 threads where its list of clusters is long: the grid has at least 64 of them and few
// enough views share the sphere (a footprint holds about a view's share of it).  Microseconds, 256 / 512 threads
// (1024 in brackets): a batch of 64 eyes, 16 views of 32^2, 200 / 150; ovals, 256 views of 64^2, 50 / 42 (40); 512
// views 31.5 / 26.6; 640 views 32 / 27.5; a 256^2 eye 18.5 / 17.5 (16.8), 731x517 17.6 / 16.5 (17.7).  Shorter lists
// leave the second half idle: 1024 views of 64^2 28.2 / 29.8, 26 views of 23^2 14.6 / 15.2.
constexpr int kWideBlock = 512;
static bool long_lists(int n_views, int n_clusters) { return n_clusters >= 64 && n_views <= 3 * n_clusters; }

// One block per (eye, view, part) whose disk footprint reaches the eye; a part
// is kPartClusters clusters of 4x4 cells, the whole view for grids up to 65^2.
// (1) A thread per cluster: the eight corners of the frustum piece that holds
//     the cluster (its ray rectangle between its nearest and farthest depth)
//     against the padded footprint; a cluster wholly beyond one side, or behind
//     the near plane, is dropped without touching its vertices.  On the rig all
//     but a few per cent go here: a view's footprint holds tens of its cells.
// (2) A warp per listed cluster: 25 lanes transform its vertices, and each of
//     the 32 lanes takes a triangle from their registers (shuffles), culls it by
//     outcodes, sets it up (snap, clip, orientation, fill rule) and the warp
//     appends the kept records to the pool.
// (3) MULTI = false (one part): the block bins the view's records.  MULTI = true:
//     every record notes its (eye, view) and its box once more (A.pool_owner, A.pool_box), the last part of a view
//     to finish reserves and clears its tile counts, and the bin_* kernels below
//     count and scatter all records of the call, a thread each.
// Bound by the latency of its phases (dependent loads, the pool's atomic, the
// divisions of a triangle), not by bytes (about 40 KB per view).  Against blocks
// that staged and transformed every vertex of a view (in bands, twice, where the
// grid did not fit shared memory), launches serialised: stereo rig 34 -> 22 us;
// grids of 129^2 and 200^2 (256 views, a 400^2 eye, count and scatter included)
// 208 -> 51 us and 458 -> 62 us; a prefilter's 64 renders of 256^2 meshes 5.7 ->
// 2.3 ms.  One-part grids keep the binning in the block: with a view's blocks as a
// cluster that counts in the leader's shared memory (distributed shared memory
// atomics), 256 views and a 400^2 eye took 20 us instead of 29, but the stereo rig
// 30 to 128 us instead of 22 (1 to 8 blocks per view).
template <bool MULTI, int BLOCK>
__global__ void __launch_bounds__(BLOCK, BLOCK > kSetupBlock ? 1024 / BLOCK : MULTI ? 4 : 3) tri_setup_kernel(FrameArgs A, int cnt_cap) {
  constexpr int NW = BLOCK / 32;
  const int v = blockIdx.x, e = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the view set-up has completed (it wrote the view records read below); the
  // raster may then launch, and waits for this grid before it reads the bins
  griddep_wait();
  griddep_release();
  ViewRec& R = A.vrecs[(int64_t)e * A.n_views + v];
  SetupCtx C;
  C.bb0 = R.bb[0]; C.bb1 = R.bb[1]; C.bb2 = R.bb[2]; C.bb3 = R.bb[3];
  if (C.bb0 > C.bb2 || C.bb1 > C.bb3) return;  // disk footprint misses the eye
  // a two-level frame sets up only the views the eye draws
  if (A.enable_bits && !((A.enable_bits[(int64_t)e * A.mask_words + (v >> 5)] >> (v & 31)) & 1u)) return;
  const EyeFloat& EF = A.eyes_f[e];
  const int G = A.G, n_cell = G - 1, ncl = clusters_per_side(G);
  extern __shared__ __align__(16) unsigned char smem[];  // the binning's per-tile counts
  __shared__ int s_warp[NW];
  __shared__ uint16_t s_list[kPartClusters];
  __shared__ int2 s_range[2 * kPartClusters];  // records written: a range per cluster, a second one after a near clip
  __shared__ int s_nlist, s_nrange, s_total;
  if (threadIdx.x == 0) s_nlist = s_nrange = s_total = 0;
  C.fx = EF.fx; C.fy = EF.fy; C.cx = EF.cx; C.cy = EF.cy;
  C.zn = A.z_near;
  // outcode planes in the form fx*x <op> (edge - cx) * z, padded by 2 pixels
  const float oxl = (float)C.bb0 - 2.0f - C.cx, oxr = (float)C.bb2 + 3.0f - C.cx;
  const float oyt = (float)C.bb1 - 2.0f - C.cy, oyb = (float)C.bb3 + 3.0f - C.cy;
  float Mf[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) Mf[k] = R.Mf[k];
  const float* ta = A.tables.a + (int64_t)v * G;
  const float* tb = A.tables.b + (int64_t)v * G;
  auto to_eye = [&](float a, float b, float z) {  // grid point z (a, b, 1), fixed order
    const float X = __fmul_rn(z, a), Y = __fmul_rn(z, b);
    EyeVtx q;
    q.x = __fmaf_rn(Mf[0], X, __fmaf_rn(Mf[1], Y, __fmaf_rn(Mf[2], z, Mf[9])));
    q.y = __fmaf_rn(Mf[3], X, __fmaf_rn(Mf[4], Y, __fmaf_rn(Mf[5], z, Mf[10])));
    q.z = __fmaf_rn(Mf[6], X, __fmaf_rn(Mf[7], Y, __fmaf_rn(Mf[8], z, Mf[11])));
    return q;
  };
  auto side_bits = [&](const EyeVtx& q, float mx, float my) -> uint32_t {  // beyond a side by more than a margin
    const float ux = C.fx * q.x, uy = C.fy * q.y;
    return (ux < oxl * q.z - mx ? 1u : 0u) | (ux > oxr * q.z + mx ? 2u : 0u) | (uy < oyt * q.z - my ? 4u : 0u) |
           (uy > oyb * q.z + my ? 8u : 0u);
  };
  __syncthreads();

  // ---- (1) clusters that can reach the footprint.  The half-spaces are linear, so
  // what holds at the eight corners holds for every point between them - but for the
  // roundings: to_eye is within four of them, 2^-22 of the sum of its terms' sizes,
  // at a corner and at a vertex, and the crossing of an edge with the near plane and
  // the sides' products are within ten more.  The corners must be beyond a plane by
  // 2^-19 of those sums, so that no cluster is dropped of which (2) would keep a triangle.
  // (Without the margin, clusters whose vertices lie on the near plane within rounding were lost.)
  {
    const int c = blockIdx.z * kPartClusters + threadIdx.x;
    bool keep = false;
    if (threadIdx.x < kPartClusters && c < ncl * ncl) {
      const int cl_y = c / ncl, cl_x = c - cl_y * ncl;
      const float2 zr = __ldg(A.cluster_z + (int64_t)v * ncl * ncl + c);
      const int j = cl_x * kClusterCells, k = cl_y * kClusterCells;
      const float a[2] = {__ldg(ta + j), __ldg(ta + min(j + kClusterCells, n_cell))};
      const float b[2] = {__ldg(tb + k), __ldg(tb + min(k + kClusterCells, n_cell))};
      const float am = fmaxf(fabsf(a[0]), fabsf(a[1])), bm = fmaxf(fabsf(b[0]), fabsf(b[1]));
      const float zm = fmaxf(fabsf(zr.x), fabsf(zr.y));
      float sum[3];  // per eye axis, the size of to_eye's terms
#pragma unroll
      for (int r = 0; r < 3; ++r)
        sum[r] = zm * (fabsf(Mf[3 * r]) * am + fabsf(Mf[3 * r + 1]) * bm + fabsf(Mf[3 * r + 2])) + fabsf(Mf[9 + r]);
      constexpr float kRound = 1.0f / (1 << 19);
      const float mx = kRound * (C.fx * sum[0] + fmaxf(fabsf(oxl), fabsf(oxr)) * sum[2]);
      const float my = kRound * (C.fy * sum[1] + fmaxf(fabsf(oyt), fabsf(oyb)) * sum[2]);
      const float near = C.zn - kRound * sum[2];
      uint32_t oc = 31u;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const EyeVtx q = to_eye(a[i & 1], b[(i >> 1) & 1], i < 4 ? zr.x : zr.y);
        oc &= side_bits(q, mx, my) | (q.z < near ? kOcBehind : 0u);
      }
      keep = oc == 0u;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(&s_nlist, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (keep) s_list[base + __popc(m & ((1u << lane) - 1u))] = (uint16_t)threadIdx.x;
  }
  __syncthreads();

  // ---- (2) the listed clusters' triangles
  const int n_list = s_nlist;
  const float z0 = A.mesh_format == LF_MESH_F16_OFFSET ? A.views[v].depth_origin : 0.0f;
  const int cell = lane >> 1, half = lane & 1;
  const int tcx = cell & 3, tcy = cell >> 2;  // this lane's cell in the cluster
  // its vertices among the cluster's 5 x 5: (j,k)(j+1,k)(j,k+1) or (j+1,k)(j+1,k+1)(j,k+1)
  const int l0 = tcy * 5 + tcx + half, l1 = half ? l0 + 5 : l0 + 1, l2 = (tcy + 1) * 5 + tcx;
  const uint32_t below = (1u << lane) - 1u;
  for (int i = warp; i < n_list; i += NW) {
    const int c = blockIdx.z * kPartClusters + s_list[i];
    const int cl_y = c / ncl, cl_x = c - cl_y * ncl;
    const int vk = min(cl_y * kClusterCells + min(lane / 5, 4), n_cell), vj = min(cl_x * kClusterCells + lane % 5, n_cell);
    const int64_t gi = ((int64_t)v * G + vk) * G + vj;
    const float z = A.mesh_format == LF_MESH_F16_OFFSET
                        ? __fadd_rn(z0, __half2float(reinterpret_cast<const __half*>(A.depth)[gi]))
                        : __ldg(reinterpret_cast<const float*>(A.depth) + gi);
    const EyeVtx q = to_eye(__ldg(ta + vj), __ldg(tb + vk), z);
    // snapped here, once per vertex, instead of by the up to six triangles around it (with 32-bit boxes and the
    // plane's divisions for kept triangles only: stereo rig 29.2 -> 27.8 us, ovals 52 -> 50, a 256^2 eye 19.7 -> 18.2)
    int32_t qx = 0, qy = 0;
    uint32_t oc = kOcBehind;
    if (q.z >= C.zn) oc = side_bits(q, 0.0f, 0.0f) | (snap_rn(q.x, q.y, q.z, C.fx, C.fy, C.cx, C.cy, qx, qy) ? 0u : kOcFar);
    EyeVtx p0, p1, p2;
    p0.x = __shfl_sync(0xffffffffu, q.x, l0); p0.y = __shfl_sync(0xffffffffu, q.y, l0); p0.z = __shfl_sync(0xffffffffu, q.z, l0);
    p1.x = __shfl_sync(0xffffffffu, q.x, l1); p1.y = __shfl_sync(0xffffffffu, q.y, l1); p1.z = __shfl_sync(0xffffffffu, q.z, l1);
    p2.x = __shfl_sync(0xffffffffu, q.x, l2); p2.y = __shfl_sync(0xffffffffu, q.y, l2); p2.z = __shfl_sync(0xffffffffu, q.z, l2);
    const uint32_t o0 = __shfl_sync(0xffffffffu, oc, l0), o1 = __shfl_sync(0xffffffffu, oc, l1);
    const uint32_t o2 = __shfl_sync(0xffffffffu, oc, l2);
    const int j = cl_x * kClusterCells + tcx, k = cl_y * kClusterCells + tcy;
    SetupPoly P;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int l = i == 0 ? l0 : i == 1 ? l1 : l2;
      P.px[i] = __shfl_sync(0xffffffffu, qx, l);
      P.py[i] = __shfl_sync(0xffffffffu, qy, l);
    }
    P.px[3] = P.px[2]; P.py[3] = P.py[2];
    // the outcodes only drop triangles that lie wholly behind the near plane or outside
    // the padded disk footprint, whose pixels never see this view
    P.np = j < n_cell && k < n_cell && (o0 & o1 & o2) == 0 && ((o0 | o1 | o2) & kOcFar) == 0 ? 3 : 0;
    if (P.np && ((o0 | o1 | o2) & kOcBehind)) clip_poly(p0, p1, p2, o0, o1, o2, C, P);
    const int id = 2 * (k * n_cell + j) + half;
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      if (f == 1 && !__any_sync(0xffffffffu, P.np == 4)) break;
      TriRec t;
      int32_t tl = 0;
      bool kept = false;
      if (P.np >= f + 3) {
        const int32_t sx[3] = {P.px[0], P.px[f + 1], P.px[f + 2]}, sy[3] = {P.py[0], P.py[f + 1], P.py[f + 2]};
        kept = setup_sub(sx, sy, C, t, tl) && setup_plane(p0, p1, p2, t);
      }
      const uint32_t m = __ballot_sync(0xffffffffu, kept);
      if (m == 0) continue;
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(A.pool_counter, (unsigned long long)__popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      const int n = __popc(m);
      const bool fits = (int64_t)base + n <= A.pool_capacity;
      const int64_t at = (int64_t)base + __popc(m & below);
      if (kept && at < A.pool_capacity) {
        t.id_tl = (id << 3) | tl;
        A.pool[at] = t;
        if constexpr (MULTI) {
          A.pool_owner[at] = e * A.n_views + v;
          A.pool_box[at] = *reinterpret_cast<const int2*>(&t);
        }
      }
      if (lane == 0) {
        if (!fits) atomicOr(A.error_word, kErrPoolOverflow);
        if (MULTI) atomicAdd(&s_total, n);
        if (!MULTI && fits) s_range[atomicAdd(&s_nrange, 1)] = make_int2((int)base, n);
      }
    }
  }
  __syncthreads();  // the block's records and ranges are visible to all its threads

  // ---- (3) bins
  if constexpr (!MULTI) {
    if (s_nrange > 0) bin_view<BLOCK>(A, R, s_range, s_nrange, reinterpret_cast<int*>(smem), cnt_cap, s_warp);
  } else {
    __shared__ int s_last;
    __shared__ long long s_off;
    if (threadIdx.x == 0) {
      if (s_total) atomicAdd(&R.tri_count, s_total);
      __threadfence();
      s_last = atomicAdd(&R.parts_done, 1) == (int)gridDim.z - 1;
      s_off = -1;
      if (s_last && atomicAdd(&R.tri_count, 0) > 0) {
        const TileBox t = footprint_tiles(R.bb, A.tile_w, A.tile_h);
        s_off = take_offsets(A, t.ntx * t.nty);
        if (s_off >= 0) {
          R.bin_off = (int32_t)s_off;
          R.btx0 = (int16_t)t.tx0; R.bty0 = (int16_t)t.ty0;
          R.bntx = (int16_t)t.ntx; R.bnty = (int16_t)t.nty;
        }
      }
    }
    __syncthreads();
    if (s_off < 0) return;
    const TileBox t = footprint_tiles(R.bb, A.tile_w, A.tile_h);
    const int nt = t.ntx * t.nty;
    int* curs = A.bin_offsets + s_off + nt + 1;
    for (int k = threadIdx.x; k < nt; k += BLOCK) curs[k] = 0;
  }
}

// Records of the call, a thread each (four at a time, their loads together): pass
// 0 counts the bins' entries, pass 1 (after bin_scan_kernel) scatters the pool
// indices through the cursors.  The boxes lie in an array of their own, 12 bytes
// per record with the owner instead of a sector of the record and the owner: 64
// renders of 256^2 meshes (36 M records) count 465 -> 340 us, scatter 695 -> 553,
// their writing adds 50 us to the set-up.  SHARE: lanes whose records enter the same
// bin share one addition and write neighbouring entries - for fine meshes, whose
// neighbours meet in one tile: scatter 553 -> 455 us; counting, whose additions
// return nothing, 340 -> 373 (kept apart), and triangles of several tiles, which the
// warp then walks in step, count 35 -> 45 us at 128^2 meshes of a 256^2 eye.
// Triangles of many tiles (a telephoto eye over a dense mesh: up to 15,625 of a 2000^2 image each) are
// walked by all lanes of a warp, and by several warps where the records are no more than the warps.
// Whole passes of such an eye (focal length 20,000 pixels, 1400x1200; 100,000, 2000^2), the older set-up's
// blocks / a thread each / so: 64 views of 66^2 meshes 223 / 1,219 / 108 us and 626 / 5,538 / 198; of 129^2
// 251 / 510 / 110 and 996 / 4,915 / 199.  A prefilter's 36 M records as before (count 340, scatter 445).
constexpr int kWideTiles = 32;
constexpr int kBinThreads = 256, kBinBlocks = 152 * 8;

template <int PASS, bool SHARE>
__global__ void __launch_bounds__(kBinThreads) bin_records_kernel(FrameArgs A) {
  static_assert(PASS == 1 || !SHARE, "only the scatter shares additions");
  constexpr int U = 4;
  griddep_wait();
  griddep_release();
  const int64_t n = min((int64_t)*A.pool_counter, A.pool_capacity), step = (int64_t)gridDim.x * blockDim.x;
  const int sw = __ffs(A.tile_w) - 1, sh = __ffs(A.tile_h) - 1;
  const int lane = threadIdx.x & 31;
  auto tiles_of = [&](int2 bb, int4 bins, RecordTiles& T, int& ntx, int& curs) {  // bins: bin_off, btx0 | bty0, bntx | bnty
    const TileBox b = {(int16_t)(bins.y & 0xffff), bins.y >> 16, (int16_t)(bins.z & 0xffff), bins.z >> 16, sw, sh};
    T = record_tiles(bb, b);
    ntx = b.ntx;
    curs = bins.x + b.ntx * b.nty + 1;
  };
  auto enter = [&](int bin, int record) {
    const int at = atomicAdd(&A.bin_offsets[bin], 1);
    if (PASS == 1) A.bin_entries[at] = record;
  };
  // tiles first, first + stride, .. of a record's box
  auto walk = [&](const RecordTiles& T, int ntx, int curs, int record, int first, int stride) {
    const int w = T.x1 - T.x0 + 1, count = w * (T.y1 - T.y0 + 1);
#pragma unroll 4
    for (int t = first; t < count; t += stride) enter(curs + (T.y0 + t / w) * ntx + T.x0 + t % w, record);
  };
  const int64_t warps = step >> 5;
  if (n <= warps) {  // a warp or more per record
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int parts = n > 0 ? (int)min(warps / n, (int64_t)64) : 0;
    if (w >= n * parts) return;
    const int64_t i = w % n;
    const int4 bins = *reinterpret_cast<const int4*>(&A.vrecs[A.pool_owner[i]].bin_off);
    if (bins.x < 0) return;
    RecordTiles T;
    int ntx, curs;
    tiles_of(A.pool_box[i], bins, T, ntx, curs);
    if (T.x0 <= T.x1 && T.y0 <= T.y1) walk(T, ntx, curs, (int)i, (int)(w / n) * 32 + lane, parts * 32);
    return;
  }
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 - lane < n; i0 += U * step) {
    int2 bb[U];
    int4 bins[U];  // bin_off, btx0 | bty0, bntx | bnty, big_base
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * step;
      bins[u].x = -1;
      if (i >= n) continue;
      bb[u] = A.pool_box[i];
      bins[u] = *reinterpret_cast<const int4*>(&A.vrecs[A.pool_owner[i]].bin_off);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      RecordTiles T = {0, 0, -1, -1};
      int ntx = 0, curs = 0;
      if (bins[u].x >= 0) tiles_of(bb[u], bins[u], T, ntx, curs);
      const int record = (int)(i0 + u * step);
      for (uint32_t m = __ballot_sync(0xffffffffu, T.x0 <= T.x1 && T.y0 <= T.y1 && (T.x1 - T.x0 + 1) * (T.y1 - T.y0 + 1) > kWideTiles);
           m; m &= m - 1) {  // the warp's wide records, one after the other
        const int l = __ffs(m) - 1;
        const RecordTiles W = {__shfl_sync(0xffffffffu, T.x0, l), __shfl_sync(0xffffffffu, T.y0, l),
                               __shfl_sync(0xffffffffu, T.x1, l), __shfl_sync(0xffffffffu, T.y1, l)};
        walk(W, __shfl_sync(0xffffffffu, ntx, l), __shfl_sync(0xffffffffu, curs, l), __shfl_sync(0xffffffffu, record, l), lane, 32);
        if (lane == l) T.x1 = T.x0 - 1;
      }
      if constexpr (!SHARE) {
        for (int y = T.y0; y <= T.y1; ++y)
          for (int x = T.x0; x <= T.x1; ++x) enter(curs + y * ntx + x, record);
        continue;
      }
      int x = T.x0, y = T.y0;
      bool has = T.x0 <= T.x1 && T.y0 <= T.y1;
      while (__any_sync(0xffffffffu, has)) {
        // lanes whose records enter the same bin here share one addition
        const int key = has ? curs + y * ntx + x : -1 - lane;
        const uint32_t same = __match_any_sync(0xffffffffu, key);
        const int first = __ffs(same) - 1;
        int at = 0;
        if (has && lane == first) at = atomicAdd(&A.bin_offsets[key], __popc(same));
        at = __shfl_sync(0xffffffffu, at, first);
        if (has) A.bin_entries[at + __popc(same & ((1u << lane) - 1u))] = record;
        if (has && ++x > T.x1) {
          x = T.x0;
          has = ++y <= T.y1;
        }
      }
    }
  }
}

// A block per (eye, view) with records: its counts become offsets and cursors.
__global__ void __launch_bounds__(kSetupBlock) bin_scan_kernel(FrameArgs A) {
  __shared__ int s_warp[kSetupBlock / 32];
  griddep_wait();
  griddep_release();
  ViewRec& R = A.vrecs[(int64_t)blockIdx.y * A.n_views + blockIdx.x];
  if (R.bin_off < 0) return;
  const int nt = (int)R.bntx * R.bnty;
  int* offs = A.bin_offsets + R.bin_off;
  int total;
  const long long ent = scan_bins<kSetupBlock>(A, offs + nt + 1, offs, nt, 0, s_warp, total);
  if (ent < 0 && threadIdx.x == 0) R.bin_off = -1;  // no room: the view has no bins (its offsets were not written)
}

cudaError_t launch_tri_setup(const FrameArgs& a, cudaStream_t s, bool pdl) {
  const size_t bytes = sizeof(int) * (size_t)kBinSmemTiles;
  const int ncl = clusters_per_side(a.G);
  const int parts = (ncl * ncl + kPartClusters - 1) / kPartClusters;
  const dim3 grid(a.n_views, a.n_eyes, parts), block(kSetupBlock);
  if (parts == 1 && long_lists(a.n_views, ncl * ncl))
    return launch_kernel(tri_setup_kernel<false, kWideBlock>, grid, dim3(kWideBlock), bytes, s, pdl, a, kBinSmemTiles);
  if (parts == 1) return launch_kernel(tri_setup_kernel<false, kSetupBlock>, grid, block, bytes, s, pdl, a, kBinSmemTiles);
  cudaError_t e = launch_kernel(tri_setup_kernel<true, kSetupBlock>, grid, block, 0, s, pdl, a, 0);
  const dim3 all(kBinBlocks), threads(kBinThreads);
  if (e == cudaSuccess) e = launch_kernel(bin_records_kernel<0, false>, all, threads, 0, s, pdl, a);
  if (e == cudaSuccess) e = launch_kernel(bin_scan_kernel, dim3(a.n_views, a.n_eyes), block, 0, s, pdl, a);
  auto scatter = a.fine_most ? bin_records_kernel<1, true> : bin_records_kernel<1, false>;
  if (e == cudaSuccess) e = launch_kernel(scatter, all, threads, 0, s, pdl, a);
  return e;
}

}  // namespace lfk
