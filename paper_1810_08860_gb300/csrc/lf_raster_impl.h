// lf_raster_impl.h - the fragment stage: rasterise, depth test within each view,
// fetch, weight, accumulate and normalise (Eq. 2, Sec. 4.2 and 4.2.2).
//
// A warp owns a screen tile (or one strip of it when a call has fewer tiles) and
// draws it by itself, without block barriers, strip by strip: a strip is TW x
// (kPx * 32 / TW) pixels, kPx (two or four) vertically adjacent pixels per lane, whose FP32
// accumulators of Eq. 2's numerator and denominator stay in registers (the
// paper's accumulation framebuffer becomes registers, and its second pass
// becomes the epilogue).
//
// What the strips of a tile share is done once per tile, lanes in parallel:
// the views of the tile's mask are listed (32 per round), their records copied
// to shared memory, this tile's bin entries gathered (64 per window) and their
// edge functions re-based to the tile origin, with one bit per (triangle,
// strip) that says whether the strip can be covered.  Then per strip, for each
// view in view order:
//   1. each pixel tests its sphere crossing against the view's disk (views no
//      pixel of the strip sees are skipped);
//   2. every pixel tests the view's triangles that reach the strip with three
//      int32 multiply-adds (the int64 edge function divided by 256, exact
//      because pixel centres step by 256 subpixels) and keeps the nearest
//      fragment by FP32 1/z, ties to the lower id;
//   3. the winner is projected into the source view and sampled bilinearly,
//      weighted, and accumulated, all pixels of a lane in one go: the view's
//      constants are warp-uniform, and their texel loads are in flight together.
//
// Bound by instruction issue (DRAM traffic is a few per cent of the peak), so
// what counts is instructions per pixel and view.  Against one warp per strip
// that listed, gathered and buffered winners by itself: 217 M -> 142 M warp
// instructions on the stereo rig frame (1,024 views, 2 x 1440x1600, FP32), the raster
// alone 293 -> 205 us; 3,772 -> 1,898 us for a batch of 64 eyes of the cap rig; 144 ->
// 82 us for a 1921x1083 eye with oval disks and FP8 texels.  Of that, reading a
// column's slope and a row's terms from tables instead of dividing per pixel gives
// 2,100 -> 2,011 us on the batch, and five blocks per SM at 96 registers instead of
// six at 80 2,011 -> 1,901.  With four pixels per lane 96 registers are too few as well
// (110 bytes of spills stored and 168 loaded per thread, round disks; 118 and 176 with the
// batch's work counter; two pixels 8 and 12).
//
// Included by the lf_raster_<format>.cu files, a texture format each (compiled side by
// side), and by lf_raster.cu for what the view selection shares.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <type_traits>

#include "lf_internal.h"
#include "lf_launch.h"
#include "lf_ray.h"

namespace lfk {

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16; x *= 0x85EBCA6Bu;
  x ^= x >> 13; x *= 0xC2B2AE35u;
  x ^= x >> 16;
  return x;
}

constexpr float kTwo23 = 8388608.0f;

// One texel as stored, and its decoded colour.
template <int FMT> struct Texel;
template <> struct Texel<LF_TEX_F32> {
  using T = float4;
  __device__ static float3 rgb(T c, float) { return make_float3(c.x, c.y, c.z); }
};
template <> struct Texel<LF_TEX_U8> {
  using T = uint32_t;
  // A byte under the exponent of 2^23, less 2^23, is its value exactly.  Twelve integer conversions per pixel and view
  // instead bound the kernel by the conversion unit: u8 stereo rig, raster alone 234 -> 194 us; 48 eyes of 25 views
  // 1,782 -> 1,546; ovals 1921x1083 124 -> 111; 64 prefilter renders 2,456 -> 2,285.
  __device__ static float3 rgb(T p, float) {
    const auto value = [&](uint32_t s) {
      return __fmul_rn(__fsub_rn(__uint_as_float(__byte_perm(p, 0x4b000000u, s)), kTwo23), 1.0f / 255.0f);
    };
    return make_float3(value(0x7440u), value(0x7441u), value(0x7442u));
  }
};
template <> struct Texel<LF_TEX_BF16> {
  using T = uint2;
  __device__ static float3 rgb(T p, float) {
    return make_float3(__uint_as_float(p.x << 16), __uint_as_float(p.x & 0xffff0000u), __uint_as_float(p.y << 16));
  }
};
template <> struct Texel<LF_TEX_FP8E4M3> {
  using T = uint32_t;
  __device__ static float3 rgb(T p, float scale) {
    __nv_fp8x2_e4m3 lo, hi;
    lo.__x = (__nv_fp8x2_storage_t)(p & 0xffffu);
    hi.__x = (__nv_fp8x2_storage_t)(p >> 16);
    float2 a = static_cast<float2>(lo);
    float2 b = static_cast<float2>(hi);
    return make_float3(__fmul_rn(a.x, scale), __fmul_rn(a.y, scale), __fmul_rn(b.x, scale));
  }
};

constexpr int kViewsPerRound = 32;  // views a warp handles per round (one per lane)
constexpr int kWindow = 64;         // gathered triangles a warp holds at a time
// Vertically adjacent pixels per lane: two, or four where a call has many tiles of 256
// pixels (FrameArgs::raster_form) - a view's list, disk, triangles and constants are then
// read half as often.  Whole tiles, raster alone, two / four: BF16 stereo 1081x1203 119 /
// 109 us, FP8 ovals 1921x1083 91 / 82, u8 stereo rig 214 / 194, FP32 stereo rig 217 / 215
// (its texels' registers take most of the gain), 640 views of 512^2 in FP32 234 / 220, 256
// views 204 / 195, the batch of 64 eyes 1,898 / 1,898.
template <int TW, int TH>
constexpr int tile_px() { return TW * TH == 256 ? 4 : 2; }
constexpr int kPxMax = 4;
constexpr int kRasterWarps = 4;     // warps per block, each on its own work item
// An eye of few tiles near its axis (kEyeFew, lf_api.cu) has few warps, which wait for each
// view's record, disk test and vote in turn.  Of full rounds of views (a rig of a thousand
// in an image of 48^2) they test all disks first and keep the views that a pixel sees.
// Whole passes, without / with: 4,096 views, one pixel 432 / 185 us, 32^2 430 / 351;
// 1,024 views, 48^2 168 / 142.

// A warp's private shared memory: its view table and its window of triangles.
// The triangle arrays are 16-byte columns, so the 32 lanes that store one
// triangle each and the uniform loads that read one are both conflict-free.
struct TriWindow {
  int4 tq[kWindow];                              // q0 q1 q2 id (bit 31: int64 edges, then q0 is the pool index)
  int4 ta[kWindow];                              // a0 b0 a1 b1
  int4 tb[kWindow];                              // a2 b2 ia ib
  float tc[kWindow];                             // ic
  uint32_t smask[kWindow / 32][8];               // per half window and strip: the triangles that reach it
};
// What a strip needs instead when a lane takes a triangle (fine meshes).
struct FineScratch {
  uint32_t depth[32 * kPxMax];                   // the view's nearest 1/z per pixel of the strip (bits), 0: none
  int queue[64];                                 // pool indices of triangles that reach the strip
  float ex[32], ey[32];                          // the strip's ray slopes by column and by row
};
struct WarpSmem {
  float4 rec[kViewsPerRound][kViewShadeQuads];   // ViewRec::cc .. tex
  union {
    TriWindow win;
    FineScratch fine;
  };
  int2 range[kViewsPerRound];                    // the view's entries in the round's concatenated bins
  int bstart[kViewsPerRound], bcount[kViewsPerRound], gbase[kViewsPerRound];
  int views[kViewsPerRound];
};

// With oval disks (Sec. 4.4) a warp also holds each view's oval constants:
// n (3), x (3), y (3), k, u0, v0, 1/e_u+, 1/e_u-, 1/e_v+, 1/e_v-.
struct WarpSmemOval : WarpSmem {
  float4 ov[kViewsPerRound][4];
};

// Oval membership, the FP32 decision (fixed order, as the oracle takes it):
// the ray (ex, ey, 1) meets the disk plane at t = k / (n.e) >= 0; inside where
// (u / e_u)^2 + (v / e_v)^2 < 1, the extents chosen by the signs of u and v.
// Returns rho^2 (the weight is 1 - sqrt(rho^2)), or 2 when outside.
__device__ __forceinline__ float oval_rho2(const float4* o4, float ex, float ey) {
  const float4 o0 = o4[0], o1 = o4[1], o2 = o4[2], o3 = o4[3];
  const float den = __fmaf_rn(o0.x, ex, __fmaf_rn(o0.y, ey, o0.z));
  if (den == 0.0f) return 2.0f;
  const float t = __fdiv_rn(o2.y, den);
  if (!(t >= 0.0f)) return 2.0f;
  const float ue = __fmaf_rn(o0.w, ex, __fmaf_rn(o1.x, ey, o1.y));
  const float ve = __fmaf_rn(o1.z, ex, __fmaf_rn(o1.w, ey, o2.x));
  const float u = __fmaf_rn(t, ue, -o2.z), v = __fmaf_rn(t, ve, -o2.w);
  const float a = __fmul_rn(u, u >= 0.0f ? o3.x : o3.y);
  const float b = __fmul_rn(v, v >= 0.0f ? o3.z : o3.w);
  const float r2 = __fmaf_rn(a, a, __fmul_rn(b, b));
  return r2 < 1.0f ? r2 : 2.0f;
}

// The next (up to 32) views of the tile's mask in increasing order, resuming
// at (cur_word, cur_bits) when the previous round stopped inside a word.
__device__ __forceinline__ int collect_views(const uint32_t* mask, int mask_words, int* views, int& cur_word,
                                             bool& partial, uint32_t& pbits) {
  const int lane = threadIdx.x & 31;
  int n = 0;
  while (cur_word < mask_words) {
    const int wl = cur_word + lane;
    uint32_t b = 0;
    if (wl < mask_words) b = (lane == 0 && partial) ? pbits : __ldg(mask + wl);
    const int c = __popc(b);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int excl = incl - c;
    const int room = kViewsPerRound - n;
    const int take = min(max(room - excl, 0), c);
    uint32_t bb = b;
    for (int k = 0; k < take; ++k) {
      const int bp = __ffs(bb) - 1;
      bb &= bb - 1;
      views[n + excl + k] = wl * 32 + bp;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total <= room) {
      n += total;
      cur_word += 32;
      partial = false;
      continue;
    }
    const unsigned over = __ballot_sync(0xffffffffu, incl > room);
    const int L = __ffs(over) - 1;
    pbits = __shfl_sync(0xffffffffu, bb, L);
    n = kViewsPerRound;
    cur_word += L;
    partial = true;
    break;
  }
  __syncwarp();
  return n;
}

// The eye holding a tile: the last one whose first tile is <= item (a binary
// search where a call may hold up to 128 eyes, a scan for the usual one or two).
template <bool MANY_EYES>
__device__ __forceinline__ int eye_of_tile(const FrameArgs& A, int item) {
  int e = 0;
  if constexpr (MANY_EYES) {
    for (int lo = 0, hi = A.n_eyes; hi - lo > 1;) {
      const int mid = (lo + hi) >> 1;
      if (A.eyes[mid].tile_base <= item) lo = mid;
      else hi = mid;
      e = lo;
    }
  } else {
    while (e + 1 < A.n_eyes && A.eyes[e + 1].tile_base <= item) ++e;
  }
  return e;
}

// The edge functions of a triangle whose deltas exceed the int32 path, at one
// pixel centre in 256ths, from its pool record.
__device__ __forceinline__ bool covers_wide(const TriRec* tr, int64_t Px, int64_t Py) {
  bool in = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3;
    const int64_t DX = (int64_t)tr->x[k1] - tr->x[k], DY = (int64_t)tr->y[k1] - tr->y[k];
    in &= DX * (Py - tr->y[k]) - DY * (Px - tr->x[k]) + ((tr->id_tl >> k) & 1) - 1 >= 0;
  }
  return in;
}

// One warp's work item: strips s0 .. s1 - 1 of tile `item`.  EYE_FINE: the eyes may differ in
// EyeParams::fine (the look-up costs a batch of 64 like eyes 0.7 per cent of its raster).
template <int TW, int TH, int FMT, bool INSPECT, bool MANY_EYES, bool OVAL, int kPx, bool EYE_FINE, typename Smem>
__device__ __forceinline__ void raster_item(const FrameArgs& A, const int item, const int s0, const int s1, Smem& S) {
  constexpr int ROWS = (32 / TW) * kPx;
  constexpr int STRIPS = TH / ROWS;
  const int lane = threadIdx.x & 31;
  const uint32_t* mask = A.tile_masks + (int64_t)item * A.mask_words;
  const int e = eye_of_tile<MANY_EYES>(A, item);
  const EyeParams& E = A.eyes[e];
  const int tile = item - E.tile_base;
  const int ty = tile / E.tiles_x, tx = tile - ty * E.tiles_x;
  const int i0 = tx * TW, j0 = ty * TH;
  const int W = E.W, H = E.H;
  const int di = lane % TW;
  const int pi = i0 + di;
  const float4* rows = A.ray_rows + E.line_base;
  const float ex = A.ray_cols[4 * (int64_t)E.line_base + min(pi, W - 1)];
  const float px = (float)pi + 0.5f;
  const int64_t vbase = (int64_t)e * A.n_views;

  // (a flag held in a register over the loops below made the stereo rig's frame 234 -> 250 us)
  auto fine = [&]() { return !INSPECT && A.fine_mesh && (!EYE_FINE || A.fine_mesh == 1 || E.fine); };

  int nv = 0, T = 0;          // the round's views, and their bin entries
  int w0 = 0, w1 = 0;         // the window: entries [w0, w1) are in shared memory
  bool resident = false;      // the tile's only round is in shared memory
  uint32_t stored = 0;        // views of the round whose active flag this warp has set

  // ---- the next round of views: their records and this tile's bin ranges
  // (`sees`: whether the lane's pixels see the view of a slot whose disk is in shared memory)
  auto load_round = [&](int& cur_word, bool& partial, uint32_t& pbits, auto&& sees) {
    __syncwarp();
    nv = collect_views(mask, A.mask_words, S.views, cur_word, partial, pbits);
    w0 = w1 = T = 0;
    stored = 0;
    if constexpr (kPx == 2) {
      if (nv == kViewsPerRound && (E.form & kEyeFew)) {  // drop the views that no pixel sees
        const int v = S.views[lane];
        if constexpr (OVAL) {
          for (int k = 0; k < 4; ++k) S.ov[lane][k] = reinterpret_cast<const float4*>(A.vrecs[vbase + v].ov)[k];
        } else {
          S.rec[lane][0] = *reinterpret_cast<const float4*>(A.vrecs[vbase + v].cc);
        }
        __syncwarp();
        uint32_t m = 0;
#pragma unroll 8
        for (int sl = 0; sl < kViewsPerRound; ++sl) m |= (uint32_t)sees(sl) << sl;
        m = __reduce_or_sync(0xffffffffu, m);
        if ((m >> lane) & 1u) S.views[__popc(m & ((1u << lane) - 1u))] = v;
        nv = __popc(m);
        __syncwarp();
      }
    }
    if (nv == 0) return;
    int c = 0;
    if (lane < nv) {
      const ViewRec& VR = A.vrecs[vbase + S.views[lane]];
      const int4 b = *reinterpret_cast<const int4*>(&VR.bin_off);  // bin_off, btx0 | bty0, bntx | bnty, big_base
      int bs = 0, bn = 0;
      if (b.x >= 0) {
        const int lx = tx - (int16_t)(b.y & 0xffff), ly = ty - (b.y >> 16), bw = (int16_t)(b.z & 0xffff);
        if (lx >= 0 && lx < bw && ly >= 0 && ly < (b.z >> 16)) {
          const int* offs = A.bin_offsets + b.x + ly * bw + lx;
          bs = offs[0];
          bn = offs[1] - bs;
        }
        c = VR.big_count;
      }
      S.bstart[lane] = bs;
      S.bcount[lane] = bn;
      S.gbase[lane] = b.w;
      c += bn;
    }
    // the records, 16 bytes per lane
    for (int i = lane; i < nv * kViewShadeQuads; i += 32) {
      const int v = i / kViewShadeQuads, k = i - v * kViewShadeQuads;
      S.rec[v][k] = reinterpret_cast<const float4*>(A.vrecs + vbase + S.views[v])[k];
    }
    if constexpr (OVAL) {
      for (int i = lane; i < nv * 4; i += 32)
        S.ov[i >> 2][i & 3] = reinterpret_cast<const float4*>(A.vrecs[vbase + S.views[i >> 2]].ov)[i & 3];
    }
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    S.range[lane] = make_int2(incl - c, incl);
    T = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
  };

  // ---- a window of bin entries from f0 on: re-based edges, strip bits
  auto gather = [&](int f0) {
    __syncwarp();
    w0 = f0;
    w1 = min(T, f0 + kWindow);
    const int64_t P0x = 256 * (int64_t)i0 + 128, P0y = 256 * (int64_t)j0 + 128;
    for (int h = 0; h < kWindow / 32; ++h) {
      const int f = f0 + h * 32 + lane;
      uint32_t reach = 0;
      if (f < T) {
        int lo = 0, hi = nv;
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (S.range[mid].x <= f) lo = mid;
          else hi = mid;
        }
        const int k = f - S.range[lo].x;
        const int idx = k < S.bcount[lo] ? __ldg(A.bin_entries + S.bstart[lo] + k)
                                         : __ldg(A.bin_entries + S.gbase[lo] + (k - S.bcount[lo]));
        const TriRec* tr = A.pool + idx;
        const int4 ra = __ldg(reinterpret_cast<const int4*>(tr));       // bbox, x0, x1
        const int4 rb = __ldg(reinterpret_cast<const int4*>(tr) + 1);   // x2, y0, y1, y2
        const int4 rc = __ldg(reinterpret_cast<const int4*>(tr) + 2);   // ia, ib, ic, id_tl
        const int bx0 = (int16_t)(ra.x & 0xffff), by0 = ra.x >> 16;
        const int bx1 = (int16_t)(ra.y & 0xffff), by1 = ra.y >> 16;
        const int32_t X[3] = {ra.z, ra.w, rb.x};
        const int32_t Y[3] = {rb.y, rb.z, rb.w};
        int32_t q[3], a[3], b[3];
        bool big = false;
#pragma unroll
        for (int k2 = 0; k2 < 3; ++k2) {
          const int k1 = (k2 + 1) % 3;
          const int64_t DX = (int64_t)X[k1] - X[k2], DY = (int64_t)Y[k1] - Y[k2];
          const int64_t q64 = (DX * (P0y - Y[k2]) - DY * (P0x - X[k2]) + ((rc.w >> k2) & 1) - 1) >> 8;  // floor
          q[k2] = (int32_t)max(min(q64, (int64_t)kQClamp), -(int64_t)kQClamp);
          a[k2] = (int32_t)-DY;
          b[k2] = (int32_t)DX;
          big |= (DX >= kBigEdge || DX <= -kBigEdge || DY >= kBigEdge || DY <= -kBigEdge);
        }
        if (bx0 <= i0 + TW - 1 && bx1 >= i0) {
#pragma unroll
          for (int s = 0; s < STRIPS; ++s) {
            const int r0 = s * ROWS, r1 = r0 + ROWS - 1;
            bool ok = by0 <= j0 + r1 && by1 >= j0 + r0;
            if (!big) {  // the largest value of each edge over the strip's pixel centres; < 0 rejects it
#pragma unroll
              for (int k2 = 0; k2 < 3; ++k2)
                ok &= q[k2] + max(0, a[k2] * (TW - 1)) + max(b[k2] * r0, b[k2] * r1) >= 0;
            }
            reach |= (uint32_t)ok << s;
          }
        }
        const int at = h * 32 + lane;
        const int id = rc.w >> 3;
        S.win.tq[at] = big ? make_int4(idx, 0, 0, id | (int32_t)0x80000000) : make_int4(q[0], q[1], q[2], id);
        S.win.ta[at] = make_int4(a[0], b[0], a[1], b[1]);
        S.win.tb[at] = make_int4(a[2], b[2], rc.x, rc.y);
        S.win.tc[at] = __int_as_float(rc.z);
      }
#pragma unroll
      for (int s = 0; s < STRIPS; ++s) {
        const uint32_t m = __ballot_sync(0xffffffffu, (reach >> s) & 1u);
        if (lane == 0) S.win.smask[h][s] = m;
      }
    }
    __syncwarp();
  };

  // ---- fine meshes: the nearest 1/z of view slot sl for every pixel of strip s.
  // Triangles of a few pixels leave most lanes of a pixel-parallel test idle, so a
  // lane takes a triangle and walks the pixels of its box inside the strip; the
  // depths meet in shared memory (unsigned maximum of the bits of 1/z > 0).  The
  // edge functions and 1/z are the ones of the pixel-parallel form.
  auto fine_depth = [&](FineScratch& F, int sl, int s) {
    const int r0 = j0 + s * ROWS, r1 = r0 + ROWS - 1;
    const int64_t P0x = 256 * (int64_t)i0 + 128, P0y = 256 * (int64_t)r0 + 128;
#pragma unroll
    for (int q = 0; q < kPx; ++q) F.depth[q * 32 + lane] = 0u;
    __syncwarp();
    auto walk = [&](int cnt) {
      if (lane >= cnt) return;
      const TriRec* tr = A.pool + F.queue[lane];
      const int4 ra = __ldg(reinterpret_cast<const int4*>(tr));
      const int4 rb = __ldg(reinterpret_cast<const int4*>(tr) + 1);
      const int4 rc = __ldg(reinterpret_cast<const int4*>(tr) + 2);
      const int x0 = max((int)(int16_t)(ra.x & 0xffff), i0), y0 = max(ra.x >> 16, r0);
      const int x1 = min((int)(int16_t)(ra.y & 0xffff), i0 + TW - 1), y1 = min(ra.y >> 16, r1);
      const int32_t X[3] = {ra.z, ra.w, rb.x};
      const int32_t Y[3] = {rb.y, rb.z, rb.w};
      const float ia = __int_as_float(rc.x), ib = __int_as_float(rc.y), ic = __int_as_float(rc.z);
      int32_t k[3], a[3], b[3];  // the edges at the box's first pixel, and their steps per column and row
      bool big = false;
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) {
        const int k1 = (k2 + 1) % 3;
        const int64_t DX = (int64_t)X[k1] - X[k2], DY = (int64_t)Y[k1] - Y[k2];
        const int64_t q64 = (DX * (P0y - Y[k2]) - DY * (P0x - X[k2]) + ((rc.w >> k2) & 1) - 1) >> 8;
        a[k2] = (int32_t)-DY;
        b[k2] = (int32_t)DX;
        big |= (DX >= kBigEdge || DX <= -kBigEdge || DY >= kBigEdge || DY <= -kBigEdge);
        k[k2] = (int32_t)max(min(q64, (int64_t)kQClamp), -(int64_t)kQClamp) + (big ? 0 : a[k2] * (x0 - i0) + b[k2] * (y0 - r0));
      }
      for (int y = y0; y <= y1; ++y) {
        int32_t e0 = k[0], e1 = k[1], e2 = k[2];
        const float zr = __fmaf_rn(ib, F.ey[y - r0], ic);
        for (int x = x0; x <= x1; ++x) {
          const bool cov = big ? covers_wide(tr, 256 * (int64_t)x + 128, 256 * (int64_t)y + 128) : (e0 | e1 | e2) >= 0;
          const float iz = __fmaf_rn(ia, F.ex[x - i0], zr);
          if (cov && iz > 0.0f) atomicMax(&F.depth[(y - r0) * TW + x - i0], __float_as_uint(iz));
          e0 += a[0]; e1 += a[1]; e2 += a[2];
        }
        k[0] += b[0]; k[1] += b[1]; k[2] += b[2];
      }
    };
    const int n = S.range[sl].y - S.range[sl].x, nb = S.bcount[sl];
    int qn = 0;
    for (int f0 = 0; f0 < n; f0 += 32) {
      const int f = f0 + lane;
      bool reach = false;
      int idx = 0;
      if (f < n) {
        idx = f < nb ? __ldg(A.bin_entries + S.bstart[sl] + f) : __ldg(A.bin_entries + S.gbase[sl] + (f - nb));
        const int2 bb = __ldg(reinterpret_cast<const int2*>(A.pool + idx));
        reach = (int16_t)(bb.x & 0xffff) <= i0 + TW - 1 && (int16_t)(bb.y & 0xffff) >= i0 && (bb.x >> 16) <= r1 &&
                (bb.y >> 16) >= r0;
      }
      const uint32_t m = __ballot_sync(0xffffffffu, reach);
      if (reach) F.queue[qn + __popc(m & ((1u << lane) - 1u))] = idx;
      qn += __popc(m);
      __syncwarp();
      if (qn >= 32) {
        walk(32);
        __syncwarp();
        const int rest = F.queue[32 + lane];
        __syncwarp();
        F.queue[lane] = rest;
        qn -= 32;
        __syncwarp();
      }
    }
    walk(qn);
    __syncwarp();
  };

  for (int s = s0; s < s1; ++s) {
    if (j0 + s * ROWS >= H) break;  // the image ends above this strip
    const int dj = s * ROWS + (lane / TW) * kPx;  // this lane's first row, tile-relative
    const float4 ray = A.eyes_f[e].ray, centre = A.eyes_f[e].centre;
    bool valid[kPx];
    float ey[kPx], py[kPx], p[kPx][3];
    float acc_r[kPx], acc_g[kPx], acc_b[kPx], acc_w[kPx];
    int n_rec[kPx];
#pragma unroll
    for (int q = 0; q < kPx; ++q) {
      const int pj = j0 + dj + q;
      valid[q] = pi < W && pj < H;
      const float4 row = rows[min(pj, H - 1)];
      ey[q] = row.x;
      py[q] = (float)pj + 0.5f;
      // ovals are met in their own planes, not at the sphere
      if constexpr (!OVAL) sphere_crossing(ray, centre, ex, row, p[q]);
      if (!valid[q]) p[q][0] = __int_as_float(0x7fffffff);  // NaN: in no disk
      acc_r[q] = acc_g[q] = acc_b[q] = acc_w[q] = 0.0f;
      n_rec[q] = 0;
    }
    if (fine()) {
      if (lane < TW) S.fine.ex[lane] = ex;
#pragma unroll
      for (int q = 0; q < kPx; ++q)
        if (di == 0) S.fine.ey[dj - s * ROWS + q] = ey[q];
      __syncwarp();
    }
    // whether pixel q of the lane sees the view in slot sl; its squared distance from the disk's centre (ovals: rho^2)
    auto member = [&](int sl, int q, float& dd) -> bool {
      if constexpr (OVAL) {
        dd = valid[q] ? oval_rho2(S.ov[sl], ex, ey[q]) : 2.0f;
        return dd < 1.0f;
      } else {
        const float4 cc = S.rec[sl][0];
        dd = disk_d2(cc, p[q]);
        return dd < cc.w;
      }
    };
    auto sees = [&](int sl) {
      bool any = false;
      float dd;
#pragma unroll
      for (int q = 0; q < kPx; ++q) any |= member(sl, q, dd);
      return any;
    };
    int cur_word = 0;
    bool partial = false;
    uint32_t pbits = 0;
    for (int round = 0;; ++round) {
      if (!resident) load_round(cur_word, partial, pbits, sees);
      uint32_t seen = 0;  // views some pixel of the strip sees
      for (int sl = 0; sl < nv; ++sl) {
        // ---- disk membership of each pixel's sphere crossing
        float d2[kPx];
        bool in[kPx];
#pragma unroll
        for (int q = 0; q < kPx; ++q) in[q] = member(sl, q, d2[q]);
        bool any_in = false;
#pragma unroll
        for (int q = 0; q < kPx; ++q) any_in |= in[q];
        if (!__any_sync(0xffffffffu, any_in)) continue;
        seen |= 1u << sl;

        // ---- the view's triangles: the depth winner is the largest 1/z > 0 of the
        // covering triangles.  Which of two equal depths wins (the lower id) does not
        // show in the image, which only takes the depth; the inspection form, which
        // reports the winner, keeps both in one key: the bits of 1/z (positive, so
        // they order as unsigned integers) above 0x7fffffff - id.
        float best[kPx];
        uint64_t best_key[kPx];
        int n_cover[kPx], min_id[kPx], max_id[kPx];
        uint32_t hash[kPx];
#pragma unroll
        for (int q = 0; q < kPx; ++q) {
          best[q] = 0.0f;
          best_key[q] = 0;
          n_cover[q] = 0; min_id[q] = 0x7fffffff; max_id[q] = -1; hash[q] = 0u;
        }
        if (fine()) {
          fine_depth(S.fine, sl, s);
#pragma unroll
          for (int q = 0; q < kPx; ++q) best[q] = __uint_as_float(S.fine.depth[(dj - s * ROWS + q) * TW + di]);
          __syncwarp();  // the depths are reset by the next view
        } else {
          const int2 range = S.range[sl];
          for (int f = range.x; f < range.y;) {
            if (f < w0 || f >= w1) gather(f);
            const int n = min(min(range.y, w1) - f, 32), base = f - w0;
            uint32_t m = (uint32_t)((((uint64_t)S.win.smask[1][s] << 32) | S.win.smask[0][s]) >> base);
            if (n < 32) m &= (1u << n) - 1u;
            f += n;
            while (m) {
              const int t = base + __ffs(m) - 1;
              m &= m - 1;
              const int4 tq = S.win.tq[t], ta = S.win.ta[t], tb = S.win.tb[t];
              bool cov[kPx];
              if (tq.w >= 0) {
                int k0 = tq.x + ta.x * di + ta.y * dj;
                int k1 = tq.y + ta.z * di + ta.w * dj;
                int k2 = tq.z + tb.x * di + tb.y * dj;
  #pragma unroll
                for (int q = 0; q < kPx; ++q) {
                  cov[q] = (k0 | k1 | k2) >= 0;
                  k0 += ta.y; k1 += ta.w; k2 += tb.y;
                }
              } else {
  #pragma unroll
                for (int q = 0; q < kPx; ++q)
                  cov[q] = covers_wide(A.pool + tq.x, 256 * (int64_t)pi + 128, 256 * (int64_t)(j0 + dj + q) + 128);
              }
              const float ia = __int_as_float(tb.z), ib = __int_as_float(tb.w), ic = S.win.tc[t];
  #pragma unroll
              for (int q = 0; q < kPx; ++q) {
                const float iz = __fmaf_rn(ia, ex, __fmaf_rn(ib, ey[q], ic));
                if constexpr (INSPECT) {
                  if (!cov[q]) continue;
                  const int id = tq.w & 0x7fffffff;
                  ++n_cover[q];
                  min_id[q] = min(min_id[q], id);
                  max_id[q] = max(max_id[q], id);
                  hash[q] ^= mix32((uint32_t)id);
                  if (iz > 0.0f) {
                    const uint64_t key = ((uint64_t)__float_as_uint(iz) << 32) | (uint32_t)(0x7fffffff - id);
                    if (key > best_key[q]) best_key[q] = key;
                    best[q] = __uint_as_float((uint32_t)(best_key[q] >> 32));
                  }
                } else {
                  if (cov[q]) best[q] = fmaxf(best[q], iz);
                }
              }
            }
          }
        }
        if constexpr (INSPECT) {
#pragma unroll
          for (int q = 0; q < kPx; ++q) {
            if (!in[q]) continue;
            if (n_rec[q] < A.max_records) {
              lf_frag_record r;
              r.view = S.views[sl];
              r.n_cover = n_cover[q];
              r.winner = best_key[q] ? 0x7fffffff - (int)(uint32_t)best_key[q] : -1;
              r.min_id = n_cover[q] ? min_id[q] : -1;
              r.max_id = n_cover[q] ? max_id[q] : -1;
              r.id_hash = hash[q];
              const int64_t pix = (int64_t)(j0 + dj + q) * W + pi;
              A.records[pix * A.max_records + n_rec[q]] = r;
            }
            ++n_rec[q];
          }
        }
        bool hit[kPx];
#pragma unroll
        for (int q = 0; q < kPx; ++q) hit[q] = in[q] && best[q] > 0.0f;
        bool any_hit = false;
#pragma unroll
        for (int q = 0; q < kPx; ++q) any_hit |= hit[q];
        if (!__any_sync(0xffffffffu, any_hit)) continue;

        // ---- shade: project the winner into the view, bilinear texels, weight, accumulate.
        // The bilinear coordinates (s - 1/2, t - 1/2) are clamped to the texel
        // centres' range and the footprint's corner to the last but one texel, which
        // is clamp to edge with one address: the outer texel of an edge sample then
        // has weight 0 or 1.  Explicit roundings: the same image for every tile
        // shape, and for the inspection form.
        using T4 = typename Texel<FMT>::T;
        const float4 h0 = S.rec[sl][1], h1 = S.rec[sl][2], h2 = S.rec[sl][3], ms = S.rec[sl][4];
        const T4* tex = reinterpret_cast<const T4*>(((uint64_t)__float_as_uint(ms.w) << 32) | __float_as_uint(ms.z));
        const int sw = A.src_w, sh = A.src_h;
        T4 c00[kPx], c10[kPx], c01[kPx], c11[kPx];
        float al[kPx], be[kPx], wt[kPx];
#pragma unroll
        for (int q = 0; q < kPx; ++q) {
          const float iz = best[q];
          const float hx = fmaf(h0.x, px, fmaf(h0.y, py[q], fmaf(h0.w, iz, h0.z)));
          const float hy = fmaf(h1.x, px, fmaf(h1.y, py[q], fmaf(h1.w, iz, h1.z)));
          const float hz = fmaf(h2.x, px, fmaf(h2.y, py[q], fmaf(h2.w, iz, h2.z)));
          const bool ok = hit[q] && hz > 0.0f;
          const float rz = __fdividef(1.0f, hz);
          const float u = fminf(fmaxf(__fmul_rn(hx, rz), 0.0f), (float)(sw - 1));
          const float v = fminf(fmaxf(__fmul_rn(hy, rz), 0.0f), (float)(sh - 1));
          // floor by adding 2^23 rounded down (0 <= u, v < 2^23): the integer is in the
          // low bits and the conversion unit is not needed
          const float tu = fminf(__fadd_rd(u, kTwo23), kTwo23 + (float)(sw - 2));
          const float tv = fminf(__fadd_rd(v, kTwo23), kTwo23 + (float)(sh - 2));
          al[q] = __fsub_rn(u, __fsub_rn(tu, kTwo23));
          be[q] = __fsub_rn(v, __fsub_rn(tv, kTwo23));
          const int iu = __float_as_int(tu) - __float_as_int(kTwo23), jv = __float_as_int(tv) - __float_as_int(kTwo23);
          // the weight is a value, not a decision: fast square root
          const float dist = d2[q] > 0.0f ? __fmul_rn(d2[q], rsqrtf(d2[q])) : 0.0f;
          wt[q] = ok ? fmaxf(0.0f, OVAL ? 1.0f - dist : __fmaf_rn(-dist, ms.x, 1.0f)) : 0.0f;
          c00[q] = c10[q] = c01[q] = c11[q] = T4{};
          if (ok) {
            const T4* t0 = tex + (jv * sw + iu);
            const T4* t1 = t0 + sw;
            c00[q] = __ldg(t0); c10[q] = __ldg(t0 + 1);
            c01[q] = __ldg(t1); c11[q] = __ldg(t1 + 1);
            if constexpr (INSPECT) {
              if (A.texel_bits) {  // the texels of the footprint, clamped to the edge
                const float ub = fminf(fmaxf(__fmul_rn(hx, rz), -1.0f), (float)sw);
                const float vb = fminf(fmaxf(__fmul_rn(hy, rz), -1.0f), (float)sh);
                const int ib0 = (int)floorf(ub), jb0 = (int)floorf(vb);
                const int i[2] = {min(max(ib0, 0), sw - 1), min(max(ib0 + 1, 0), sw - 1)};
                const int j[2] = {min(max(jb0, 0), sh - 1), min(max(jb0 + 1, 0), sh - 1)};
                for (int k = 0; k < 4; ++k) {
                  const int64_t bit = ((int64_t)S.views[sl] * sh + j[k >> 1]) * sw + i[k & 1];
                  atomicOr(&A.texel_bits[bit >> 5], 1u << (bit & 31));
                }
              }
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kPx; ++q) {
          const float3 a = Texel<FMT>::rgb(c00[q], ms.y), b = Texel<FMT>::rgb(c10[q], ms.y);
          const float3 c = Texel<FMT>::rgb(c01[q], ms.y), d = Texel<FMT>::rgb(c11[q], ms.y);
          const float nal = __fsub_rn(1.0f, al[q]), nbe = __fsub_rn(1.0f, be[q]);
          const float w00 = __fmul_rn(nal, nbe), w10 = __fmul_rn(al[q], nbe), w01 = __fmul_rn(nal, be[q]),
                      w11 = __fmul_rn(al[q], be[q]);
          acc_r[q] = __fmaf_rn(wt[q], __fmaf_rn(w11, d.x, __fmaf_rn(w01, c.x, __fmaf_rn(w10, b.x, __fmul_rn(w00, a.x)))), acc_r[q]);
          acc_g[q] = __fmaf_rn(wt[q], __fmaf_rn(w11, d.y, __fmaf_rn(w01, c.y, __fmaf_rn(w10, b.y, __fmul_rn(w00, a.y)))), acc_g[q]);
          acc_b[q] = __fmaf_rn(wt[q], __fmaf_rn(w11, d.z, __fmaf_rn(w01, c.z, __fmaf_rn(w10, b.z, __fmul_rn(w00, a.z)))), acc_b[q]);
          acc_w[q] = __fadd_rn(acc_w[q], wt[q]);
        }
      }
      // the views' active flags (view selection), each set once per work item
      if (lane < nv && (((seen & ~stored) >> lane) & 1u)) A.active[vbase + S.views[lane]] = 1;
      stored |= seen;
      const bool more = cur_word < A.mask_words;
      if (resident || !more) {
        // one round and one window hold the whole tile: the next strips reuse them
        resident = resident || (round == 0 && (T <= kWindow || fine()));
        break;
      }
    }
#pragma unroll
    for (int q = 0; q < kPx; ++q) {
      if (!valid[q]) continue;
      const int64_t pix = (int64_t)(j0 + dj + q) * W + pi;
      float4 out;
      if (acc_w[q] > 0.0f) {
        const float inv = __frcp_rn(acc_w[q]);
        out = make_float4(__fmul_rn(acc_r[q], inv), __fmul_rn(acc_g[q], inv), __fmul_rn(acc_b[q], inv), 1.0f);
      } else {
        out = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      reinterpret_cast<float4*>(E.out)[pix] = out;
      if constexpr (INSPECT) {
        A.counts[pix] = n_rec[q];
        if (n_rec[q] > A.max_records) atomicOr(A.error_word, kErrRecordOverflow);
      }
    }
  }
}

// The warps of the grid take work items (a tile's strips, A.strips_per_item at
// a time): their own in a plain launch, the next one from the device counter
// in a persistent launch.
template <int TW, int TH, int FMT, bool INSPECT, bool PERSISTENT, bool OVAL, int PX>
__global__ void __launch_bounds__(kRasterWarps * 32, 5) raster_kernel(FrameArgs A) {
  constexpr int STRIPS = TH / ((32 / TW) * PX);
  using Smem = typename std::conditional<OVAL, WarpSmemOval, WarpSmem>::type;
  __shared__ Smem S[kRasterWarps];
  const int warp = threadIdx.x >> 5;
  const int per = A.strips_per_item, groups = STRIPS / per;
  const int n_items = A.total_tiles * groups;
  // Launched early (programmatic dependent launch), the blocks wait here until
  // the set-up grid before this one has completed: everything read below (eye
  // constants, tile masks, view records, bins, the work counter) is written by
  // the kernels of the frame before this one.
  griddep_wait();
  for (int turn = 0;; ++turn) {
    int item = 0;
    if constexpr (PERSISTENT) {
      if ((threadIdx.x & 31) == 0) item = atomicAdd(A.work_counter, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
    } else {
      if (turn) break;
      item = blockIdx.x * kRasterWarps + warp;
    }
    if (item >= n_items) break;
    const int tile = item / groups, s0 = (item - tile * groups) * per;
    raster_item<TW, TH, FMT, INSPECT, PERSISTENT, OVAL, PX, tile_px<TW, TH>() == 2>(A, tile, s0, s0 + per, S[warp]);
  }
}

// Where the eyes of a call differ, in what a warp should take of their tiles (EyeParams::form) or in
// being fine, both raster_item forms in one kernel, an eye's items from its item_base on.
template <int TW, int TH, int FMT, bool PERSISTENT, bool OVAL>
__global__ void __launch_bounds__(kRasterWarps * 32, 5) raster_mixed_kernel(FrameArgs A) {
  using Smem = typename std::conditional<OVAL, WarpSmemOval, WarpSmem>::type;
  __shared__ Smem S[kRasterWarps];
  constexpr int STRIPS2 = TH / ((32 / TW) * 2), STRIPS4 = STRIPS2 / 2;
  const int warp = threadIdx.x >> 5;
  griddep_wait();
  for (int turn = 0;; ++turn) {
    int item = 0;
    if constexpr (PERSISTENT) {
      if ((threadIdx.x & 31) == 0) item = atomicAdd(A.work_counter, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
    } else {
      if (turn) break;
      item = blockIdx.x * kRasterWarps + warp;
    }
    if (item >= A.mixed_items) break;
    int e = 0;  // the last eye whose first item is <= item
    for (int hi = A.n_eyes; hi - e > 1;) {
      const int mid = (e + hi) >> 1;
      if (A.eyes[mid].item_base <= item) e = mid;
      else hi = mid;
    }
    const EyeParams& E = A.eyes[e];
    const int i = item - E.item_base, form = E.form & 3;
    if (form == kRasterStrips) {
      raster_item<TW, TH, FMT, false, PERSISTENT, OVAL, 2, true>(A, E.tile_base + i / STRIPS2, i % STRIPS2, i % STRIPS2 + 1, S[warp]);
    } else {
      const int per = form == kRasterWhole ? STRIPS4 : 1, groups = STRIPS4 / per, s0 = i % groups * per;
      raster_item<TW, TH, FMT, false, PERSISTENT, OVAL, 4, true>(A, E.tile_base + i / groups, s0, s0 + per, S[warp]);
    }
  }
}

template <int TW, int TH, int FMT, bool OVAL, int PX>
static cudaError_t launch_px(FrameArgs a, bool inspect, bool persistent, int pblocks, cudaStream_t s, bool pdl) {
  constexpr int STRIPS = TH / ((32 / TW) * PX);
  a.strips_per_item = a.raster_form == kRasterWhole ? STRIPS : 1;
  const int64_t items = (int64_t)a.total_tiles * (STRIPS / a.strips_per_item);
  const dim3 block(kRasterWarps * 32), grid((unsigned)((items + kRasterWarps - 1) / kRasterWarps));
  if constexpr (PX == 2)  // the inspection form: two pixels per lane only
    if (inspect) return launch_kernel(raster_kernel<TW, TH, FMT, true, false, OVAL, PX>, grid, block, 0, s, pdl, a);
  if (persistent) return launch_kernel(raster_kernel<TW, TH, FMT, false, true, OVAL, PX>, dim3(pblocks), block, 0, s, pdl, a);
  return launch_kernel(raster_kernel<TW, TH, FMT, false, false, OVAL, PX>, grid, block, 0, s, pdl, a);
}

template <int TW, int TH, int FMT, bool OVAL>
static cudaError_t launch_disk(const FrameArgs& a, bool inspect, bool persistent, int pblocks, cudaStream_t s,
                               bool pdl) {
  if constexpr (tile_px<TW, TH>() == 4) {
    if (a.raster_form == kRasterMixed) {
      const dim3 block(kRasterWarps * 32), grid((unsigned)((a.mixed_items + kRasterWarps - 1) / kRasterWarps));
      if (persistent) return launch_kernel(raster_mixed_kernel<TW, TH, FMT, true, OVAL>, dim3(pblocks), block, 0, s, pdl, a);
      return launch_kernel(raster_mixed_kernel<TW, TH, FMT, false, OVAL>, grid, block, 0, s, pdl, a);
    }
    if (a.raster_form != kRasterStrips && !inspect) return launch_px<TW, TH, FMT, OVAL, 4>(a, false, persistent, pblocks, s, pdl);
  }
  return launch_px<TW, TH, FMT, OVAL, 2>(a, inspect, persistent, pblocks, s, pdl);
}

template <int TW, int TH, int FMT>
static cudaError_t launch_fmt(const FrameArgs& a, bool inspect, bool persistent, int pblocks, cudaStream_t s,
                              bool pdl) {
  if (a.disk_mode == 1) return launch_disk<TW, TH, FMT, true>(a, inspect, persistent, pblocks, s, pdl);
  return launch_disk<TW, TH, FMT, false>(a, inspect, persistent, pblocks, s, pdl);
}

// What a texture format's file defines (LF_RASTER_FORMAT).
template <int FMT>
cudaError_t launch_raster_fmt(const FrameArgs& a, bool inspect, bool persistent, int pblocks, cudaStream_t s, bool pdl);
template <int FMT>
cudaError_t raster_occupancy_fmt(int tile_w, int tile_h, int disk_mode, int* n);

#ifdef LF_RASTER_FORMAT
template <>
cudaError_t launch_raster_fmt<LF_RASTER_FORMAT>(const FrameArgs& a, bool inspect, bool persistent, int pblocks,
                                                cudaStream_t s, bool pdl) {
  constexpr int F = LF_RASTER_FORMAT;
  if (a.tile_w == 16 && a.tile_h == 16) return launch_fmt<16, 16, F>(a, inspect, persistent, pblocks, s, pdl);
  if (a.tile_w == 32 && a.tile_h == 8) return launch_fmt<32, 8, F>(a, inspect, persistent, pblocks, s, pdl);
  if (a.tile_w == 8 && a.tile_h == 8) return launch_fmt<8, 8, F>(a, inspect, persistent, pblocks, s, pdl);
  return cudaErrorInvalidValue;
}

// Both forms of a tile (two and four pixels per lane) have the same launch bounds, 96 registers and the same shared
// memory, so one answers for the other: five blocks per SM.
template <int TW, int TH, int FMT>
static cudaError_t occupancy_tile(int disk_mode, int* n) {
  constexpr int kThreads = kRasterWarps * 32;
  return disk_mode == 1
             ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, raster_kernel<TW, TH, FMT, false, true, true, 2>, kThreads, 0)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, raster_kernel<TW, TH, FMT, false, true, false, 2>, kThreads, 0);
}

template <>
cudaError_t raster_occupancy_fmt<LF_RASTER_FORMAT>(int tile_w, int tile_h, int disk_mode, int* n) {
  if (tile_w == 16 && tile_h == 16) return occupancy_tile<16, 16, LF_RASTER_FORMAT>(disk_mode, n);
  if (tile_w == 32 && tile_h == 8) return occupancy_tile<32, 8, LF_RASTER_FORMAT>(disk_mode, n);
  return occupancy_tile<8, 8, LF_RASTER_FORMAT>(disk_mode, n);
}
#endif

}  // namespace lfk
