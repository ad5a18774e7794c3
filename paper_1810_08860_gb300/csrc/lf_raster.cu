// lf_raster.cu - the raster's dispatch over texture formats (lf_raster_impl.h holds its
// kernels), and the view selection of two-level frames (Sec. 7.2).
#include "lf_raster_impl.h"

namespace lfk {

// The exact view selection of a two-level frame: a warp per tile tests the
// tile's pixels against the disks of its mask's views that no tile has marked
// in A.visible yet (a stale flag only costs the test), 32 pixels at a time
// until every view of the round has been seen.
template <bool OVAL>
__global__ void __launch_bounds__(kRasterWarps * 32) select_kernel(FrameArgs A) {
  __shared__ float4 s_disk[kRasterWarps][kViewsPerRound][OVAL ? 4 : 1];
  __shared__ int s_views[kRasterWarps][kViewsPerRound];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = blockIdx.x * kRasterWarps + warp;
  if (item >= A.total_tiles) return;
  const int e = eye_of_tile<true>(A, item);
  const EyeParams& E = A.eyes[e];
  const float4 ray = A.eyes_f[e].ray, centre = A.eyes_f[e].centre;
  const int tile = item - E.tile_base;
  const int ty = tile / E.tiles_x, tx = tile - ty * E.tiles_x;
  const uint32_t* mask = A.tile_masks + (int64_t)item * A.mask_words;
  const int64_t vbase = (int64_t)e * A.n_views;
  int* views = s_views[warp];
  int cur_word = 0;
  bool partial = false;
  uint32_t pbits = 0;
  while (cur_word < A.mask_words) {
    const int nv = collect_views(mask, A.mask_words, views, cur_word, partial, pbits);
    if (nv == 0) break;
    const int v = lane < nv ? views[lane] : 0;
    const bool open = lane < nv && A.visible[vbase + v] == 0;
    uint32_t todo = __ballot_sync(0xffffffffu, open), found = 0;
    if (open) {
      if constexpr (OVAL) {
        for (int k = 0; k < 4; ++k) s_disk[warp][lane][k] = reinterpret_cast<const float4*>(A.vrecs[vbase + v].ov)[k];
      } else {
        s_disk[warp][lane][0] = *reinterpret_cast<const float4*>(A.vrecs[vbase + v].cc);
      }
    }
    __syncwarp();
    for (int c = lane; todo != 0 && c - lane < A.tile_w * A.tile_h; c += 32) {
      const int pi = tx * A.tile_w + c % A.tile_w, pj = ty * A.tile_h + c / A.tile_w;
      const bool has = pi < E.W && pj < E.H;
      const float ex = A.ray_cols[4 * (int64_t)E.line_base + min(pi, E.W - 1)];
      const float4 row = A.ray_rows[(int64_t)E.line_base + min(pj, E.H - 1)];
      float p[3];
      if constexpr (!OVAL) sphere_crossing(ray, centre, ex, row, p);
      for (uint32_t m = todo; m; m &= m - 1) {
        const int sl = __ffs(m) - 1;
        bool in;
        if constexpr (OVAL) in = has && oval_rho2(s_disk[warp][sl], ex, row.x) < 1.0f;
        else in = has && disk_d2(s_disk[warp][sl][0], p) < s_disk[warp][sl][0].w;
        if (__any_sync(0xffffffffu, in)) found |= 1u << sl;
      }
      todo &= ~found;
    }
    if ((found >> lane) & 1u) A.visible[vbase + v] = 1;
    __syncwarp();  // the view table is rewritten by the next round
  }
}

cudaError_t launch_select(const FrameArgs& a, cudaStream_t s) {
  if (a.total_tiles <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((a.total_tiles + kRasterWarps - 1) / kRasterWarps);
  if (a.disk_mode == 1) select_kernel<true><<<blocks, kRasterWarps * 32, 0, s>>>(a);
  else select_kernel<false><<<blocks, kRasterWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

// The views each eye draws in a two-level frame (Sec. 7.2): a fine view that it
// selects and whose image is resident; a coarse view that it selects and whose
// disk overlaps a selected fine view whose image is missing.
// A warp per view: its lanes share the overlaps.
__global__ void drawn_kernel(FrameArgs A) {
  const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, e = blockIdx.y, lane = threadIdx.x & 31;
  if (v >= A.n_views) return;
  const uint8_t* vis = A.visible + (int64_t)e * A.n_views;
  if (!vis[v]) return;
  bool on = false;
  if (v < A.n_fine) {
    on = A.page_of_view[v] >= 0;
  } else {
    const int c = v - A.n_fine;
    for (int k = A.overlap_off[c] + lane; k < A.overlap_off[c + 1] && !on; k += 32) {
      const int f = A.overlap_ids[k];
      on = vis[f] && A.page_of_view[f] < 0;
    }
  }
  if (__any_sync(0xffffffffu, on) && lane == 0)
    atomicOr(A.enable_bits + (int64_t)e * A.mask_words + (v >> 5), 1u << (v & 31));
}

// Only the drawn views stay in the tile masks: one thread per (tile, mask word).
__global__ void enable_masks_kernel(FrameArgs A) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)A.total_tiles * A.mask_words) return;
  const int tile = (int)(idx / A.mask_words), w = (int)(idx % A.mask_words);
  int e = 0;
  for (int lo = 0, hi = A.n_eyes; hi - lo > 1;) {  // the last eye whose first tile is <= tile
    const int mid = (lo + hi) >> 1;
    if (A.eyes[mid].tile_base <= tile) lo = mid;
    else hi = mid;
    e = lo;
  }
  A.tile_masks[idx] &= A.enable_bits[(int64_t)e * A.mask_words + w];
}

cudaError_t launch_drawn(const FrameArgs& a, cudaStream_t s) {
  dim3 grid((a.n_views + 3) / 4, a.n_eyes);
  drawn_kernel<<<grid, 128, 0, s>>>(a);
  const int64_t n = (int64_t)a.total_tiles * a.mask_words;
  if (n > 0) enable_masks_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_raster(const FrameArgs& a, bool inspect, bool persistent, int pblocks, cudaStream_t s, bool pdl) {
  if (a.total_tiles <= 0) return cudaSuccess;
  switch (a.tex_format) {
    case LF_TEX_F32: return launch_raster_fmt<LF_TEX_F32>(a, inspect, persistent, pblocks, s, pdl);
    case LF_TEX_U8: return launch_raster_fmt<LF_TEX_U8>(a, inspect, persistent, pblocks, s, pdl);
    case LF_TEX_BF16: return launch_raster_fmt<LF_TEX_BF16>(a, inspect, persistent, pblocks, s, pdl);
    case LF_TEX_FP8E4M3: return launch_raster_fmt<LF_TEX_FP8E4M3>(a, inspect, persistent, pblocks, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t raster_occupancy(int tile_w, int tile_h, int fmt, int disk_mode, int* n) {
  switch (fmt) {
    case LF_TEX_F32: return raster_occupancy_fmt<LF_TEX_F32>(tile_w, tile_h, disk_mode, n);
    case LF_TEX_U8: return raster_occupancy_fmt<LF_TEX_U8>(tile_w, tile_h, disk_mode, n);
    case LF_TEX_BF16: return raster_occupancy_fmt<LF_TEX_BF16>(tile_w, tile_h, disk_mode, n);
    default: return raster_occupancy_fmt<LF_TEX_FP8E4M3>(tile_w, tile_h, disk_mode, n);
  }
}

}  // namespace lfk
