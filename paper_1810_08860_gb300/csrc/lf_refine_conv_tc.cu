// lf_refine_conv_tc.cu - the refinement's training GEMMs on the fifth-
// generation tensor cores (tcgen05.mma from shared memory into TMEM): the
// single-layer convolutions (forward layers of training and of the per-layer
// inference path, the backward pass through a layer's input as the same
// correlation with flipped, transposed weights, the fused residual / loss
// epilogues) and the weight and bias gradients (wgrad_tc_kernel, below).  The network
// is the learned stand-in for the offline projection of Sec. 5, Eq. 4-5:
// y = x + conv3x3(32->3) . ReLU . conv3x3(32->32) . ReLU . conv3x3(3->32) (x).
//
// out[p][o] = sum_{tap, c} W[tap][o][c] * in[p + off(tap)][c], tap = 3 ky + kx
// reading (y + ky - 1, x + kx - 1), zero outside the image.
//
// Persistent CTAs of four warps; output tiles of 30 x 16 pixels over a halo
// of 32 positions x 18 rows, positions q = 32 hy + hx, so a halo row is one
// TMEM lane quadrant and a tap is an A operand shifted by 32 (ky - 1) + kx - 1
// positions (a descriptor start 16 bytes per position on).  Four M-tiles of
// 128 positions (4 halo rows each) per tile, N = the output channels (32, or
// 16 for the 3-output layer).  32-channel BF16 inputs: two K = 16 MMAs per tap,
// 18 per M-tile.  3-channel FP32 RGBA inputs are staged pair-packed (position
// s holds x[s] and x[s+1] as R, G, B, 0 twice) and the A descriptor puts the
// second K group two positions on, so one MMA covers kernel columns -1..+2 of
// a kernel row: 3 MMAs per M-tile.  Output columns 0 and 31 of the halo see a
// wrapped neighbour and are never stored.
//
// Per tile: the halo is staged (zeros outside the image), one thread issues
// the tile's MMAs and commits to an mbarrier, every warp waits (bounded by
// wait_ns, an error word on give-up), reads its lane quadrant of each M-tile's
// accumulators with tcgen05.ld and runs the epilogue.  Halos arrive by TMA: a
// 32-channel BF16 halo by one tiled copy per group of 8 channels straight into
// the MMA operand layout, the next tile's copy issued as soon as the current
// tile's MMAs have read the buffer (it lands during the epilogue); a 3-channel
// FP32 RGBA halo into a staging buffer that the four warps convert to BF16
// pairs, the next tile's copy issued as soon as they have read it (it lands
// during the MMAs and the epilogue).  Four CTAs share an SM, so one CTA's MMAs
// overlap another's staging and epilogue.
//
// Shared-memory operands use the K-major layout without swizzling: a position
// (row) holds 8 channels in 16 contiguous bytes, rows follow every 16 bytes
// (8-row core matrices 128 bytes apart), and each further group of 8 channels
// starts kCGroupB bytes later.  The weights arrive in the packed layouts of
// pack_weights_kernel (rows of 32 K values per output) and are rearranged into
// core-matrix blocks when a CTA loads them.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "lf_internal.h"
#include "lf_launch.h"

namespace lfk {

namespace {

constexpr int kCTW = 30, kCTH = 16;              // output tile
constexpr int kCHW = 32, kCHH = kCTH + 2;         // halo: 32 positions x 18 rows
constexpr int kCMT = kCTH / 4;                    // M-tiles of 128 positions per tile
constexpr int kCPos = kCHH * kCHW;                // 576 positions
constexpr int kCGuard = 2;                        // positions before and after (reads reach one beyond)
constexpr int kCGroupB = ((kCPos + 2 * kCGuard) * 16 + 127) / 128 * 128;  // bytes per group of 8 channels
constexpr int kCXOff = 128 - kCGuard * 16;        // halo position 0 of each group starts 128-byte aligned
constexpr int kCHaloTx = 4 * kCPos * 16;          // bytes of a tile's four TMA copies (32-channel halo)
constexpr int kCXsB = kCPos * 16;                 // a tile's FP32 RGBA halo (3-channel input), one TMA copy
constexpr int kCThreads = 128;
constexpr int kCPerSM = 4;                        // CTAs per SM: 4 x 128 TMEM columns
constexpr uint32_t kCTmemCols = 128;
constexpr uint64_t kCDrainNs = 2000000000ull;     // the teardown's wait for issued MMAs

__device__ __forceinline__ uint32_t c_su32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t c_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// kind::f16, FP32 accumulator, BF16 A and B, both K-major.
__host__ __device__ constexpr uint32_t c_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void c_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void c_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(c_su32(bar))
               : "memory");
}

// 0 once the phase of `bar` with this parity completed, 2 after limit_ns of
// %globaltimer without it.
__device__ __forceinline__ int c_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  uint32_t done;
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(c_su32(bar)), "r"(parity)
        : "memory");
    if (done) return 0;
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (it == 0) t0 = t;
    else if (t - t0 >= limit_ns) return 2;
  }
}

__device__ __forceinline__ void c_tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Tile `tile`'s 32-channel BF16 halo by TMA: one tiled copy per group g of 8
// channels (a box of 8 channels x 32 positions x 18 rows of the 5-D tensor map
// {8, 4, W, H, n} over the map; zeros where the box leaves the image) into the
// group's operand rows, completing on `bar` with the copies' byte count.
__device__ __forceinline__ void c_load_halo(const CUtensorMap* tmap, uint32_t sx0, uint64_t* bar, int img, int x0,
                                            int y0) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(c_su32(bar)), "r"(kCHaloTx) : "memory");
#pragma unroll
  for (int g = 0; g < 4; ++g)
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
        "[%7];" ::"r"(sx0 + g * kCGroupB),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(0), "r"(g), "r"(x0 - 1), "r"(y0 - 1), "r"(img), "r"(c_su32(bar))
        : "memory");
}

// Tile `tile`'s FP32 RGBA halo by TMA: one tiled copy (4 channels x 32
// positions x 18 rows of the 4-D tensor map {4, W, H, n}; zeros outside the
// image) into the staging buffer xs, completing on `bar`.  Earlier reads of xs
// by this CTA's threads are ordered before the copy by a barrier and the
// proxy fence.
__device__ __forceinline__ void c_load_rgba(const CUtensorMap* tmap, uint32_t xs, uint64_t* bar, int img, int x0,
                                            int y0) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(c_su32(bar)), "r"(kCXsB) : "memory");
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::
          "r"(xs), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(0), "r"(x0 - 1), "r"(y0 - 1), "r"(img),
      "r"(c_su32(bar))
      : "memory");
}

__device__ __forceinline__ uint32_t c_pack(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

}  // namespace

template <int IN, int COUT, int EPI>
__global__ void __launch_bounds__(kCThreads, kCPerSM)
    conv_tc_kernel(RefineConvArgs A, const __grid_constant__ CUtensorMap tmap) {
  constexpr int N = COUT < 16 ? 16 : COUT;                 // MMA N (the 3-output layer pads to 16)
  constexpr int NB = IN == kConvInBF16 ? 18 : 3;           // B blocks: (tap, half) or kernel row
  constexpr int kBlkB = 2 * N * 16;
  constexpr int kWBytes = NB * kBlkB;
  constexpr int G = IN == kConvInBF16 ? 4 : 1;             // channel groups in the halo
  extern __shared__ __align__(128) unsigned char sm[];
  unsigned char* sw = sm;
  unsigned char* sx = sm + kWBytes + kCXOff;  // group g, position p: sx + g * kCGroupB + (p + kCGuard) * 16
  constexpr int kXsOff = (kWBytes + kCXOff + G * kCGroupB + 127) / 128 * 128;
  unsigned char* xs = sm + kXsOff;             // 3-channel input: the FP32 RGBA halo as it landed
  constexpr int kBarOff = IN == kConvInBF16 ? kWBytes + kCXOff + G * kCGroupB : kXsOff + kCXsB;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kBarOff);     // the tile's MMAs completed
  uint64_t* xbar = bar + 1;                                         // the tile's TMA halo landed
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  __shared__ float s_bias[32];
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = A.H, W = A.W;

  // Weights into core-matrix blocks: block b, K group g, row n at sw + b * kBlkB + (g * N + n) * 16.
  for (int i = tid; i < NB * 2 * N; i += kCThreads) {
    const int b = i / (2 * N), g = (i / N) & 1, n = i % N;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (n < COUT) {
      if (IN == kConvInBF16) {  // packed [tap][n][32]: block b = 2 tap + half
        v = *reinterpret_cast<const uint4*>(A.wt + ((size_t)(b >> 1) * COUT + n) * 32 + 16 * (b & 1) + 8 * g);
      } else {  // packed [n][32], k = tap * 3 + c; block b = ky, element e: kx = 2g + e / 4, c = e % 4
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t half2 = 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int e = 2 * j + h, kx = 2 * g + (e >> 2), c = e & 3;
            uint32_t bits = 0;
            if (kx < 3 && c < 3) bits = *reinterpret_cast<const uint16_t*>(A.wt + n * 32 + (b * 3 + kx) * 3 + c);
            half2 |= bits << (16 * h);
          }
          w[j] = half2;
        }
        v = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    *reinterpret_cast<uint4*>(sw + b * kBlkB + (g * N + n) * 16) = v;
  }
  for (int i = tid; i < G * kCGroupB / 16; i += kCThreads)  // the guard rows stay zero
    reinterpret_cast<uint4*>(sx)[i] = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the zeros, to the tensor core and TMA
  if (tid < 32) s_bias[tid] = (EPI == kEpiRelu || (EPI != kEpiMask && tid < 3)) ? A.bias[tid] : 0.f;
  if (tid == 0) {
    s_abort = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c_su32(bar)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c_su32(xbar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c_su32(tslot)),
                 "r"(kCTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  float loss_scale = 0.f;
  if (EPI == kEpiLoss) {
    const int cnt = *A.count;
    loss_scale = cnt > 0 ? 1.0f / (3.0f * (float)cnt) : 0.f;
  }
  const int tiles_x = (W + kCTW - 1) / kCTW, tiles_y = (H + kCTH - 1) / kCTH;
  const int n_tiles = tiles_x * tiles_y * A.n;
  // tile -> image and output origin (the halo starts one row and one column before)
  auto origin = [&](int tile, int& img, int& x0, int& y0) {
    img = tile / (tiles_x * tiles_y);
    const int rem = tile - img * tiles_x * tiles_y;
    y0 = (rem / tiles_x) * kCTH;
    x0 = (rem % tiles_x) * kCTW;
  };
  const uint32_t sx0 = c_su32(sx) + kCGuard * 16;  // halo position 0 of group 0 (128-byte aligned)
  uint32_t phase = 0, xphase = 0;
  bool issued = false;        // an MMA commit of this CTA may still be outstanding
  bool halo_pending = false;  // thread 0: a TMA halo copy may still be landing
  if (tid == 0 && (int)blockIdx.x < n_tiles) {
    int img, x0, y0;
    origin(blockIdx.x, img, x0, y0);
    if (IN == kConvInBF16) c_load_halo(&tmap, sx0, xbar, img, x0, y0);
    else c_load_rgba(&tmap, c_su32(xs), xbar, img, x0, y0);
    halo_pending = true;
  }
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    int img, x0, y0;
    origin(tile, img, x0, y0);

    // ---- stage the halo
    if (IN == kConvInBF16) {  // issued before this tile (above, or during the previous epilogue)
      if (tid == 0) {
        if (c_wait(xbar, xphase, A.wait_ns) != 0) {
          atomicOr(A.error, 1024);
          s_abort = 1;
        } else {
          xphase ^= 1u;
          halo_pending = false;
        }
      }
    } else {  // every thread waits for the staged FP32 halo, then converts its positions
      if (c_wait(xbar, xphase, A.wait_ns) != 0) {
        atomicOr(A.error, 1024);
        s_abort = 1;
      } else {
        xphase ^= 1u;
        if (tid == 0) halo_pending = false;
      }
      __syncthreads();
      if (!s_abort) {
        const float4* xf = reinterpret_cast<const float4*>(xs);
        for (int p = tid; p < kCPos; p += kCThreads) {
          const float4 v0 = xf[p], v1 = p + 1 < kCPos ? xf[p + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
          *reinterpret_cast<uint4*>(sx + (p + kCGuard) * 16) =
              make_uint4(c_pack(v0.x, v0.y), c_pack(v0.z, 0.f), c_pack(v1.x, v1.y), c_pack(v1.z, 0.f));
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (s_abort) break;  // the halo copy's wait gave up
    // the warps have read the staged FP32 halo: the next tile's copy lands during the MMAs
    if (IN == kConvInRGBA && tid == 0 && tile + (int)gridDim.x < n_tiles) {
      int nimg, nx0, ny0;
      origin(tile + gridDim.x, nimg, nx0, ny0);
      c_load_rgba(&tmap, c_su32(xs), xbar, nimg, nx0, ny0);
      halo_pending = true;
    }

    // ---- the tile's MMAs: M-tile m holds output positions 32 (4m + 1) + r, r < 128
    if (tid == 0) {
      const uint32_t sxa = c_su32(sx) + kCGuard * 16;  // position 0
      const uint64_t ad = c_desc(sxa, IN == kConvInBF16 ? kCGroupB : 32, 128);
      const uint64_t bd = c_desc(c_su32(sw), N * 16, 128);
      constexpr uint32_t id = c_idesc(128, N);
      for (int m = 0; m < kCMT; ++m) {
        const uint32_t d = tmem + (uint32_t)(m * N);
        if (IN == kConvInBF16) {
#pragma unroll
          for (int t = 0; t < 9; ++t) {  // tap t = 3 ky + kx starts at 32 (4m + ky) + kx - 1
#pragma unroll
            for (int h = 0; h < 2; ++h)
              c_mma(d, ad + (uint64_t)(int64_t)(32 * (4 * m + t / 3) + t % 3 - 1) + (uint64_t)(h * (2 * kCGroupB / 16)),
                    bd + (uint64_t)((2 * t + h) * (kBlkB / 16)), id, t > 0 || h > 0);
          }
        } else {
#pragma unroll
          for (int ky = 0; ky < 3; ++ky)  // kernel row ky: pairs from 32 (4m + ky) - 1
            c_mma(d, ad + (uint64_t)(int64_t)(32 * (4 * m + ky) - 1), bd + (uint64_t)(ky * (kBlkB / 16)), id, ky > 0);
        }
      }
      c_commit(bar);
    }
    issued = true;
    if (lane == 0 && c_wait(bar, phase, A.wait_ns) != 0) {
      atomicOr(A.error, 64);
      s_abort = 1;
    }
    __syncthreads();  // every warp has waited: the abort decision is the same for the whole CTA
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (s_abort) break;
    issued = false;
    phase ^= 1u;
    // the MMAs have read the halo: the next tile's copy lands during this epilogue
    if (IN == kConvInBF16 && tid == 0 && tile + (int)gridDim.x < n_tiles) {
      int nimg, nx0, ny0;
      origin(tile + gridDim.x, nimg, nx0, ny0);
      c_load_halo(&tmap, sx0, xbar, nimg, nx0, ny0);
      halo_pending = true;
    }

    // ---- epilogue: warp w reads lanes 32w.. (halo row 4m + 1 + w, column lane) of each M-tile
    const uint32_t lane_base = (uint32_t)(32 * warp) << 16;
    const int gx = x0 + lane - 1;
    float lsum = 0.f;
    for (int m = 0; m < kCMT; ++m) {
      const int gy = y0 + 4 * m + warp;
      const bool store = lane >= 1 && lane <= kCTW && gy < H && gx < W;
      const size_t pix = ((size_t)img * H + (store ? gy : 0)) * W + (store ? gx : 0);
      const uint32_t t = tmem + lane_base + (uint32_t)(m * N);
      if (EPI == kEpiRelu || EPI == kEpiMask) {
        float v0[16], v1[16];
        c_tmem_ld16(t, v0);
        c_tmem_ld16(t + 16, v1);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (!store) continue;
        float v[32];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          v[k] = v0[k];
          v[16 + k] = v1[k];
        }
        uint32_t w[16];
        if (EPI == kEpiRelu) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            w[j] = c_pack(fmaxf(v[2 * j] + s_bias[2 * j], 0.f), fmaxf(v[2 * j + 1] + s_bias[2 * j + 1], 0.f));
        } else {
          const uint4* mk = reinterpret_cast<const uint4*>(A.mask + pix * 32);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 mq = mk[q];
            const uint32_t mw[4] = {mq.x, mq.y, mq.z, mq.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const __nv_bfloat162 mm = *reinterpret_cast<const __nv_bfloat162*>(&mw[j]);
              const int k = 8 * q + 2 * j;
              w[4 * q + j] = c_pack(__bfloat162float(mm.x) > 0.f ? v[k] : 0.f, __bfloat162float(mm.y) > 0.f ? v[k + 1] : 0.f);
            }
          }
        }
        uint4* dst = reinterpret_cast<uint4*>(A.out_h + pix * 32);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
      } else {  // kEpiResid / kEpiLoss: outputs 0..2
        float v[16];
        c_tmem_ld16(t, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (!store) continue;
        const float4 x = reinterpret_cast<const float4*>(A.x)[pix];
        const float r0 = v[0] + s_bias[0], r1 = v[1] + s_bias[1], r2 = v[2] + s_bias[2];
        if (EPI == kEpiResid) {
          const bool valid = x.w > 0.f;
          reinterpret_cast<float4*>(A.out_f)[pix] =
              valid ? make_float4(x.x + r0, x.y + r1, x.z + r2, 1.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
          const float4 tg = reinterpret_cast<const float4*>(A.target)[pix];
          const bool valid = x.w > 0.f && tg.w > 0.f;
          const float d0 = valid ? (x.x + r0) - tg.x : 0.f;
          const float d1 = valid ? (x.y + r1) - tg.y : 0.f;
          const float d2 = valid ? (x.z + r2) - tg.z : 0.f;
          lsum += d0 * d0 + d1 * d1 + d2 * d2;
          reinterpret_cast<float4*>(A.out_f)[pix] =
              make_float4(2.f * loss_scale * d0, 2.f * loss_scale * d1, 2.f * loss_scale * d2, 0.f);
        }
      }
    }
    if (EPI == kEpiLoss) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
      if (lane == 0 && lsum != 0.f) atomicAdd(A.loss, lsum * loss_scale);
    }
    // every warp has read the accumulators and the halo before the next tile overwrites them
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }

  // A wait that gave up may leave MMAs running: wait for them before the tensor memory is freed.
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && issued && s_abort && c_wait(bar, phase, kCDrainNs) != 0) atomicOr(A.error, 128);
  // and for a halo copy still landing (a wait that gave up) before the shared memory is released
  if (tid == 0 && halo_pending && c_wait(xbar, xphase, kCDrainNs) != 0) atomicOr(A.error, 2048);
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCTmemCols));
  }
}

namespace {

template <int IN, int COUT, int EPI>
cudaError_t launch_conv_tc_t(const RefineConvArgs& a, cudaStream_t s) {
  constexpr int N = COUT < 16 ? 16 : COUT;
  constexpr int kW = (IN == kConvInBF16 ? 18 : 3) * 2 * N * 16;
  constexpr int used = IN == kConvInBF16 ? kW + kCXOff + 4 * kCGroupB + 24
                                         : (kW + kCXOff + kCGroupB + 127) / 128 * 128 + kCXsB + 24;
  // At least 54 KB: no more than kCPerSM CTAs share an SM, so their tensor memory (128 columns each)
  // always fits and no CTA waits in tcgen05.alloc for another persistent CTA to finish.
  constexpr int smem = used < 54 * 1024 ? 54 * 1024 : used;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(conv_tc_kernel<IN, COUT, EPI>), smem);
  if (e != cudaSuccess) return e;
  const int n_tiles = ((a.W + kCTW - 1) / kCTW) * ((a.H + kCTH - 1) / kCTH) * a.n;
  if (n_tiles == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  // The halo copies' tensor map, over a 16-byte aligned base.  32-channel input: a 5-D tensor
  // {8 channels, 4 groups, W, H, n} of BF16, with group, position, row and image strides of 16,
  // 64, W * 64 and W * H * 64 bytes.  3-channel input: a 4-D tensor {4 channels, W, H, n} of FP32
  // RGBA, strides 16, W * 16 and W * H * 16 bytes.
  CUtensorMap tmap;
  std::memset(&tmap, 0, sizeof(tmap));
  const EncodeTiled enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  if (IN == kConvInBF16) {
    if ((reinterpret_cast<uintptr_t>(a.src_h) & 15u) != 0) return cudaErrorInvalidValue;
    const cuuint64_t dims[5] = {8, 4, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.n};
    const cuuint64_t strides[4] = {16, 64, (cuuint64_t)a.W * 64, (cuuint64_t)a.W * a.H * 64};
    const cuuint32_t box[5] = {8, 1, (cuuint32_t)kCHW, (cuuint32_t)kCHH, 1};
    const cuuint32_t step[5] = {1, 1, 1, 1, 1};
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16*>(a.src_h), dims, strides, box,
            step, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  } else {
    if ((reinterpret_cast<uintptr_t>(a.src_f) & 15u) != 0) return cudaErrorInvalidValue;
    const cuuint64_t dims[4] = {4, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.n};
    const cuuint64_t strides[3] = {16, (cuuint64_t)a.W * 16, (cuuint64_t)a.W * a.H * 16};
    const cuuint32_t box[4] = {4, (cuuint32_t)kCHW, (cuuint32_t)kCHH, 1};
    const cuuint32_t step[4] = {1, 1, 1, 1};
    if (enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(a.src_f), dims, strides, box, step,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const int grid = n_tiles < sms * kCPerSM ? n_tiles : sms * kCPerSM;
  conv_tc_kernel<IN, COUT, EPI><<<grid, kCThreads, smem, s>>>(a, tmap);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_refine_conv(int in_mode, int cout, int epi, const RefineConvArgs& a, cudaStream_t s) {
  if (in_mode == kConvInRGBA && cout == 32 && epi == kEpiRelu) return launch_conv_tc_t<kConvInRGBA, 32, kEpiRelu>(a, s);
  if (in_mode == kConvInRGBA && cout == 32 && epi == kEpiMask) return launch_conv_tc_t<kConvInRGBA, 32, kEpiMask>(a, s);
  if (in_mode == kConvInBF16 && cout == 32 && epi == kEpiRelu) return launch_conv_tc_t<kConvInBF16, 32, kEpiRelu>(a, s);
  if (in_mode == kConvInBF16 && cout == 32 && epi == kEpiMask) return launch_conv_tc_t<kConvInBF16, 32, kEpiMask>(a, s);
  if (in_mode == kConvInBF16 && cout == 8 && epi == kEpiResid) return launch_conv_tc_t<kConvInBF16, 8, kEpiResid>(a, s);
  if (in_mode == kConvInBF16 && cout == 8 && epi == kEpiLoss) return launch_conv_tc_t<kConvInBF16, 8, kEpiLoss>(a, s);
  return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ weight gradients
//
// dW[o][c][ky][kx] = sum_p g[p][o] a[p + (ky - 1, kx - 1)][c], db[o] = sum_p g[p][o]
// (g = dL/dz of the layer's output, a = the layer's input), as one GEMM over
// K = pixels whose operands are the maps as they lie in memory: both are read
// MN-major (channels contiguous), so nothing is transposed.  A tile is 32 x 8
// positions of a; per image row r of g
//   D[(i, c)][(kx, o)] += sum_x a[r - 1 + i][x][c] g[r][x + 1 - kx][o]
// with M = 128: four consecutive rows i of a (ky = i; the fourth is not used) of
// 32 channels, and N = 96: three copies of g, each loaded by TMA with its own shift
// (zeros outside the image).  A 32-channel map lies as [row][position][32 channels]
// under the 64-byte swizzle, so M steps from row to row of a and N from copy to copy
// of g.  The 3-channel maps (the network input, dL/dr) land as FP32 RGBA and two
// warps round them to BF16 rows of 8 channels, the last five zero, without swizzle:
// M then covers sixteen rows (three used), N = 32 four copies (three used).  The
// same two warps sum g for the bias gradient.
//   MODE 1: g = dL/dz1 (BF16, 32), a = the network input (FP32 RGBA, 3).  W1, b1.
//   MODE 2: g = dL/dz2 (BF16, 32), a = a1 (BF16, 32).                        W2, b2.
//   MODE 3: g = dL/dr  (FP32 RGBA, 3), a = a2 (BF16, 32).                    W3, b3.
//
// One CTA per SM, a ring of stages between a TMA warp, an MMA warp and the two
// warps above; the accumulators stay in TMEM over all tiles of a CTA, which then
// writes one partial row; the rows are summed in a fixed order afterwards
// (deterministic).  Bound by the operands' way through shared memory (an MMA reads
// 4 KB of A and 3 KB of B, 62 cycles against the 53 of its arithmetic) and by the
// three copies of g from L2.  Against kernels that transposed chunks of 64 pixels
// with ldmatrix and wrote every input nine times for its taps, 16 crops of 256^2:
// 109, 67 and 93 us for W2, W1 and W3 -> 33, 32 and 23 us (training step 564 -> 370).

namespace {

constexpr int kGTW = 32, kGTH = 8;               // tile: 32 x 8 positions
constexpr int kG32Row = kGTW * 64;               // a row of 32 channels
constexpr int kG8Row = kGTW * 16;                // a row of 8 channels
constexpr int kGThreads = 128;

template <int MODE>
struct WgradShape {
  static constexpr int OC = MODE == 3 ? 8 : 32;          // channels of g as held
  static constexpr int KX = MODE == 3 ? 4 : 3;           // copies of g held (three loaded)
  static constexpr int N = KX * OC;
  static constexpr int COUT = MODE == 3 ? 3 : 32, CIN = MODE == 1 ? 3 : 32;
  static constexpr int kARow = MODE == 1 ? kG8Row : kG32Row, kAB = (kGTH + 2) * kARow;
  static constexpr int kGRow = MODE == 3 ? kG8Row : kG32Row, kGCopy = kGTH * kGRow, kGB = KX * kGCopy;
  static constexpr int FW = MODE == 1 ? kGTW : kGTW + 2, FH = MODE == 1 ? kGTH + 2 : kGTH;  // FP32 RGBA positions
  static constexpr int kFB = MODE == 2 ? 0 : (FW * FH * 16 + 511) / 512 * 512;
  static constexpr int kStageB = kAB + kGB + kFB;
  static constexpr int kTx = MODE == 1 ? kGB + FW * FH * 16 : MODE == 2 ? kAB + kGB : kAB + FW * FH * 16;
  static constexpr int kStages = MODE == 3 ? 5 : 3;
  // The unused accumulator rows take what lies behind a tile's rows of a: the stage's g
  static_assert((kGTH - 1) * kARow + (MODE == 1 ? 16 : 4) * kARow <= kStageB, "MMAs read within the stage");
  static_assert(kStageB % 512 == 0, "stages start on a swizzle atom");
  static constexpr int kBarOff = kStages * kStageB;
  static constexpr int kSmem = 1024 + kBarOff + (3 * kStages + 1) * 8 + 16;  // 1024: the base is rounded up
  static_assert(kSmem <= 224 * 1024, "fits one CTA's shared memory");
};

// kind::f16, FP32 accumulator, BF16 A and B, both MN-major.
__host__ __device__ constexpr uint32_t g_idesc(int M, int N) { return c_idesc(M, N) | (1u << 15) | (1u << 16); }

__device__ __forceinline__ void g_tma4(const CUtensorMap* m, uint32_t dst, uint64_t* bar, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::
          "r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c_su32(bar))
      : "memory");
}
// MN-major operands: 32-channel rows under the 64-byte swizzle (next 32 elements of M or N `mn` bytes on, 8
// positions 512 bytes), and 8-channel rows without (next 8 elements `mn` bytes on, 8 positions 128 bytes).
__device__ __forceinline__ uint64_t g_desc32(uint32_t addr, uint32_t mn) { return c_desc(addr, mn, 512) | (4ull << 61); }
__device__ __forceinline__ uint64_t g_desc8(uint32_t addr, uint32_t mn) { return c_desc(addr, 128, mn); }

__device__ __forceinline__ void g_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(c_su32(bar)) : "memory");
}

}  // namespace

template <int MODE>
__global__ void __launch_bounds__(kGThreads) wgrad_tc_kernel(RefineWgradArgs A, const __grid_constant__ CUtensorMap amap,
                                                             const __grid_constant__ CUtensorMap gmap) {
  using S = WgradShape<MODE>;
  extern __shared__ __align__(128) unsigned char sm_raw[];
  unsigned char* sm = sm_raw + ((1024u - (c_su32(sm_raw) & 1023u)) & 1023u);  // stages start on a swizzle atom
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + S::kBarOff);  // a stage's copies landed
  uint64_t* ready = full + S::kStages;                             // its FP32 map is rounded (modes 1, 3)
  uint64_t* empty = ready + S::kStages;                            // its MMAs and its readers are done
  uint64_t* done = empty + S::kStages;                             // all MMAs of the CTA are complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  __shared__ volatile int s_abort;
  __shared__ float s_bias[64][8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_tiles = A.n_tiles;

  if (tid == 0) {
    s_abort = 0;
    for (int k = 0; k < S::kStages; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c_su32(full + k)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(c_su32(ready + k)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 3;" ::"r"(c_su32(empty + k)));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c_su32(done)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c_su32(tslot)),
                 "r"(kCTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int n_own = (int)blockIdx.x < n_tiles ? (n_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

  // A wait for use j of stage j % kStages; on give-up sets the error bit and the CTA's abort flag.
  auto wait_use = [&](uint64_t* bar, int j, int err) -> bool {
    if (s_abort) return false;
    if (c_wait(bar + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, A.wait_ns) == 0) return true;
    atomicOr(A.error, err);
    s_abort = 1;
    return false;
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- copies
    if (lane == 0) {
      int issued = 0;
      for (int j = 0; j < n_own; ++j) {
        if (j >= S::kStages && !wait_use(empty, j - S::kStages, 256)) break;
        const int tile = blockIdx.x + j * gridDim.x, img = tile / (A.tiles_x * A.tiles_y);
        const int rem = tile - img * A.tiles_x * A.tiles_y;
        const int y0 = rem / A.tiles_x * kGTH, x0 = rem % A.tiles_x * kGTW;
        const uint32_t st = c_su32(sm) + (j % S::kStages) * S::kStageB, sg = st + S::kAB, sf = sg + S::kGB;
        uint64_t* bar = full + j % S::kStages;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(c_su32(bar)), "r"(S::kTx) : "memory");
        g_tma4(&amap, MODE == 1 ? sf : st, bar, 0, x0, y0 - 1, img);
        if (MODE == 3) {
          g_tma4(&gmap, sf, bar, 0, x0 - 1, y0, img);
        } else {
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) g_tma4(&gmap, sg + kx * S::kGCopy, bar, 0, x0 + 1 - kx, y0, img);
        }
        issued = j + 1;
      }
      // the last copies land before the CTA can leave (earlier ones have been waited for by their readers or are
      // waited for here, after an abort)
      for (int j = issued > S::kStages ? issued - S::kStages : 0; j < issued; ++j)
        if (c_wait(full + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, kCDrainNs) != 0) atomicOr(A.error, 2048);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMAs
    if (lane == 0) {
      constexpr uint32_t id = g_idesc(128, S::N);
      for (int j = 0; j < n_own; ++j) {
        if (!wait_use(full, j, 256)) break;
        if (MODE != 2 && !wait_use(ready, j, 256)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st = c_su32(sm) + (j % S::kStages) * S::kStageB;
        constexpr int kAK = MODE == 1 ? 256 : 1024, kGK = MODE == 3 ? 256 : 1024;  // 16 positions
        const uint64_t ad = MODE == 1 ? g_desc8(st, kG8Row) : g_desc32(st, kG32Row);
        const uint64_t bd = MODE == 3 ? g_desc8(st + S::kAB, S::kGCopy) : g_desc32(st + S::kAB, S::kGCopy);
        for (int r = 0; r < kGTH; ++r)
#pragma unroll
          for (int k = 0; k < 2; ++k)
            c_mma(tmem, ad + (uint64_t)((r * S::kARow + k * kAK) / 16), bd + (uint64_t)((r * S::kGRow + k * kGK) / 16), id,
                  j > 0 || r > 0 || k > 0);
        c_commit(empty + j % S::kStages);
      }
      // completes once every MMA issued has: also after an abort, so the tensor memory is never freed under one
      c_commit(done);
      if (c_wait(done, 0u, A.wait_ns > kCDrainNs ? A.wait_ns : kCDrainNs) != 0) atomicOr(A.error, 512);
    }
  } else {
    // ---------------------------------------------------------------- rounding of FP32 maps, bias sums
    const int t = tid - 64;  // 0 .. 63
    float acc[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = 0.f;
    for (int j = 0; j < n_own; ++j) {
      int ok = 1;
      if (lane == 0) ok = wait_use(full, j, 1024);
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      // (a lane that did not poll sees the copies through the shuffle's warp: every lane tests the phase once)
      if (c_wait(full + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, kCDrainNs) != 0) break;
      unsigned char* st = sm + (j % S::kStages) * S::kStageB;
      unsigned char* sg = st + S::kAB;
      if (MODE != 2) {
        const float4* f = reinterpret_cast<const float4*>(sg + S::kGB);
        for (int i = t; i < S::FW * S::FH; i += 64) {
          const float4 v = f[i];
          const uint4 w = make_uint4(c_pack(v.x, v.y), c_pack(v.z, 0.f), 0u, 0u);
          if (MODE == 1) {
            reinterpret_cast<uint4*>(st)[i] = w;  // [row][position]
          } else {
            const int r = i / S::FW, x = i - r * S::FW;  // image column x0 - 1 + x
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) {  // copy kx holds column x0 + 1 - kx first
              const int q = x - 2 + kx;
              if (q >= 0 && q < kGTW) *reinterpret_cast<uint4*>(sg + kx * S::kGCopy + r * kG8Row + q * 16) = w;
            }
            if (x >= 1 && x <= kGTW) {  // the tile's own pixels, as rounded for the MMAs
              acc[0] += __uint_as_float(w.x << 16);
              acc[1] += __uint_as_float(w.x & 0xffff0000u);
              acc[2] += __uint_as_float(w.y << 16);
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core
        __syncwarp();
        if (lane == 0) g_arrive(ready + j % S::kStages);
      }
      if (MODE != 3) {  // thread t: channels 8 (t & 3) .., positions t / 4 and t / 4 + 16 of the unshifted copy
        for (int r = 0; r < kGTH; ++r) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int q = (t >> 2) + 16 * h;  // the swizzle moves a 16-byte chunk by the position's bits 1 and 2
            const uint4 v = *reinterpret_cast<const uint4*>(sg + S::kGCopy + r * kG32Row + q * 64 + (((t & 3) ^ ((q >> 1) & 3)) << 4));
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              acc[2 * k] += __uint_as_float(w[k] << 16);
              acc[2 * k + 1] += __uint_as_float(w[k] & 0xffff0000u);
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) g_arrive(empty + j % S::kStages);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) s_bias[t][k] = acc[k];
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();  // the MMAs are complete (the issuing thread has waited for them)
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // ---- this CTA's partial row, [ky][kx][o][c] then the biases: warp w reads accumulator rows 32w ..
  float* out = A.partial + (size_t)blockIdx.x * A.seg;
  if (!s_abort && n_own > 0) {
    if (warp < (MODE == 1 ? 1 : 3)) {
      const int ky = MODE == 1 ? lane >> 3 : warp, c = MODE == 1 ? lane & 7 : lane;
      const bool keep = c < S::CIN && ky < 3;
#pragma unroll
      for (int h = 0; h < S::N / 16; ++h) {
        float v[16];
        c_tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + 16 * h, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (keep) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            const int col = 16 * h + k, kx = col / S::OC, o = col % S::OC;
            if (kx < 3 && o < S::COUT) out[((ky * 3 + kx) * S::COUT + o) * S::CIN + c] = v[k];
          }
        }
      }
    }
    if (tid < S::COUT) {  // bias gradient: the threads' sums in a fixed order
      float b = 0.f;
      if (MODE == 3) for (int k = 0; k < 64; ++k) b += s_bias[k][tid];
      else for (int k = 0; k < 16; ++k) b += s_bias[4 * k + (tid >> 3)][tid & 7];
      out[9 * S::COUT * S::CIN + tid] = b;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCTmemCols));
  }
}

namespace {

// Tensor maps over an NHWC map: 32 BF16 channels as {32, W, H, n} under the 64-byte swizzle, or FP32 RGBA as
// {4, W, H, n}.  (As {8, W, 4 groups, H, n}, 16 bytes at a time, the copies bounded the kernel: 75 us instead of 33 for 32 channels against 32.)
bool encode_map32(EncodeTiled enc, CUtensorMap* m, const void* p, int n, int H, int W, int box_w, int box_h) {
  const cuuint64_t dims[4] = {32, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)n};
  const cuuint64_t strides[3] = {64, (cuuint64_t)W * 64, (cuuint64_t)W * H * 64};
  const cuuint32_t box[4] = {32, (cuuint32_t)box_w, (cuuint32_t)box_h, 1}, step[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p), dims, strides, box, step,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool encode_rgba(EncodeTiled enc, CUtensorMap* m, const void* p, int n, int H, int W, int box_w, int box_h) {
  const cuuint64_t dims[4] = {4, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)n};
  const cuuint64_t strides[3] = {16, (cuuint64_t)W * 16, (cuuint64_t)W * H * 16};
  const cuuint32_t box[4] = {4, (cuuint32_t)box_w, (cuuint32_t)box_h, 1}, step[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(p), dims, strides, box, step,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE>
cudaError_t launch_wgrad_tc_t(const RefineWgradArgs& a, cudaStream_t s) {
  using S = WgradShape<MODE>;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(wgrad_tc_kernel<MODE>), S::kSmem);
  if (e != cudaSuccess) return e;
  const EncodeTiled enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  CUtensorMap am, gm;
  std::memset(&am, 0, sizeof(am));
  std::memset(&gm, 0, sizeof(gm));
  const bool ok = (MODE == 1 ? encode_rgba(enc, &am, a.x, a.n, a.H, a.W, S::FW, S::FH)
                             : encode_map32(enc, &am, a.a_h, a.n, a.H, a.W, kGTW, kGTH + 2)) &&
                  (MODE == 3 ? encode_rgba(enc, &gm, a.g_f, a.n, a.H, a.W, S::FW, S::FH)
                             : encode_map32(enc, &gm, a.g_h, a.n, a.H, a.W, kGTW, kGTH));
  if (!ok) return cudaErrorInvalidValue;
  wgrad_tc_kernel<MODE><<<a.n_ctas, kGThreads, S::kSmem, s>>>(a, am, gm);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_refine_wgrad(int mode, const RefineWgradArgs& a, cudaStream_t s) {
  if (mode == 1) return launch_wgrad_tc_t<1>(a, s);
  if (mode == 2) return launch_wgrad_tc_t<2>(a, s);
  if (mode == 3) return launch_wgrad_tc_t<3>(a, s);
  return cudaErrorInvalidValue;
}

int refine_wgrad_tiles(int n, int H, int W, int* tiles_x, int* tiles_y) {
  *tiles_x = (W + kGTW - 1) / kGTW;
  *tiles_y = (H + kGTH - 1) / kGTH;
  return *tiles_x * *tiles_y * n;
}

}  // namespace lfk
