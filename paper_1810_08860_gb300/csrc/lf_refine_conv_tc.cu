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
// 32-channel BF16 halo by one tiled copy straight into the MMA operand layout, the next tile's copy issued as soon as the current
// tile's MMAs have read the buffer (it lands during the epilogue); a 3-channel
// FP32 RGBA halo into a staging buffer that the four warps convert to BF16
// pairs, the next tile's copy issued as soon as they have read it (it lands
// during the MMAs and the epilogue).  Four CTAs share an SM, so one CTA's MMAs
// overlap another's staging and epilogue.
//
// A 32-channel halo lies K-major under the 64-byte swizzle, a position's 32 channels
// in 64 bytes; pair-packed rows and the weights use the layout without swizzling:
// a row holds 8 channels in 16 contiguous bytes, rows follow every 16 bytes (8-row
// core matrices 128 bytes apart).  (As four groups of 8 channels, 16 bytes at a time,
// the halo copies alone took half as long as the MMAs.)  The weights arrive in the packed layouts of
// pack_weights_kernel (rows of 32 K values per output) and are rearranged into
// core-matrix blocks when a CTA loads them.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
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
constexpr int kCPairB = (kCPos + 2 * kCGuard) * 16;  // 3-channel input: the pair-packed halo
constexpr int kCXOff = 128 - kCGuard * 16;        // its position 0 starts 128-byte aligned
constexpr int kCHaloTx = kCPos * 64;              // 32-channel input: a tile's halo, one TMA copy
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

// Tile `tile`'s 32-channel BF16 halo by TMA: one tiled copy (32 channels x 32
// positions x 18 rows of the 4-D tensor map {32, W, H, n}; zeros where the box
// leaves the image) under the 64-byte swizzle, completing on `bar`.
__device__ __forceinline__ void c_load_halo(const CUtensorMap* tmap, uint32_t sx0, uint64_t* bar, int img, int x0,
                                            int y0) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(c_su32(bar)), "r"(kCHaloTx) : "memory");
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::
          "r"(sx0), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(0), "r"(x0 - 1), "r"(y0 - 1), "r"(img), "r"(c_su32(bar))
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

// 32-channel inputs, inference (STACK): one MMA per kernel row and 16 channels, the
// three kernel columns stacked along N (32 outputs: N = 96, one M-tile of accumulators
// at a time; 3 outputs: N = 16, four columns each).  An MMA of N = 32 or less costs
// about 45 cycles, of N = 96 about 62, so six take 372 cycles an M-tile where eighteen
// take 810; the epilogue adds two shuffles per output.  517 x 731 pixels: the last
// layer 14.7 -> 9.3 us; 2 x 1440x1600: 32 -> 32 128 -> 126, 32 -> 3 151 -> 97 us.
// Training keeps a tap an MMA (N = 32, 16), for 21 us of a step more: the sum of three
// accumulators rounds differently from one, some hidden values then round to another
// BF16 neighbour, and Adam carries that on (gradients up to 7e-4 apart after sixteen
// steps).  3-channel inputs: see above.
template <int IN, int COUT, bool STACK>
struct ConvShape {
  static constexpr bool kStacked = IN == kConvInBF16 && STACK;
  static constexpr int kOutStep = COUT == 8 ? 4 : 32;                    // stacked: rows of a kernel column along N
  static constexpr int N = kStacked && COUT == 32 ? 96 : COUT == 8 ? 16 : 32;
  static constexpr int NB = IN != kConvInBF16 ? 3 : kStacked ? 6 : 18;   // B blocks: kernel row, (row, half) or (tap, half)
  static constexpr int kMB = N == 96 ? 1 : kCMT;                         // M-tiles per batch of MMAs (128 TMEM columns)
  static constexpr int kBlkB = 2 * N * 16, kWBytes = NB * kBlkB;
};

// Four lanes (4 i .. 4 i + 3) hold a pixel each, as four 16-byte pieces; afterwards
// lane 4 i + r holds piece r of the four pixels, so that a warp's store writes whole
// pixels (64 contiguous bytes).  Stored a pixel per lane, 16 bytes at a 64-byte
// stride, every 32-byte sector was written in two halves: on 16 x 256^2 pixels the
// 3 -> 32 layer took 29 us instead of 22, the 32 -> 32 one 52 instead of 45.
__device__ __forceinline__ void c_transpose4(uint4 (&c)[4]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int b = 1; b <= 2; b <<= 1) {
    const bool up = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int k = b == 1 ? 2 * i : i, k2 = k + b;
      const uint4 give = up ? c[k] : c[k2];
      uint4 got;
      got.x = __shfl_xor_sync(0xffffffffu, give.x, b);
      got.y = __shfl_xor_sync(0xffffffffu, give.y, b);
      got.z = __shfl_xor_sync(0xffffffffu, give.z, b);
      got.w = __shfl_xor_sync(0xffffffffu, give.w, b);
      if (up) c[k] = got;
      else c[k2] = got;
    }
  }
}

// A word of two BF16 values where the same half of `gate` is > 0, else 0.
__device__ __forceinline__ uint32_t c_gate(uint32_t v, uint32_t gate) {
  const uint32_t lo = (int32_t)(gate << 16) > 0 ? 0x0000ffffu : 0u, hi = (int32_t)(gate & 0xffff0000u) > 0 ? 0xffff0000u : 0u;
  return v & (lo | hi);
}

}  // namespace

template <int IN, int COUT, int EPI, bool STACK>
__global__ void __launch_bounds__(kCThreads, kCPerSM)
    conv_tc_kernel(RefineConvArgs A, const __grid_constant__ CUtensorMap tmap) {
  using S = ConvShape<IN, COUT, STACK>;
  constexpr int N = S::N, NB = S::NB, kBlkB = S::kBlkB, kWBytes = S::kWBytes;
  constexpr bool kStacked = S::kStacked;
  extern __shared__ __align__(128) unsigned char sm_raw[];
  unsigned char* sm = sm_raw + ((1024u - (c_su32(sm_raw) & 1023u)) & 1023u);  // the 32-channel halo starts on a swizzle atom
  unsigned char* sw = sm;
  static_assert(IN != kConvInBF16 || kWBytes % 512 == 0, "a swizzle atom is 512 bytes");
  // 32 channels: position p in the 64 bytes at sx + 64 p (swizzled); windows of one tap reach one position before, into the
  // weights, and one after (output columns that are never used).  3 channels: pairs, 16 bytes at sx + (p + kCGuard) * 16.
  unsigned char* sx = sm + kWBytes + (IN == kConvInBF16 ? 0 : kCXOff);
  constexpr int kXsOff = (kWBytes + kCXOff + kCPairB + 127) / 128 * 128;
  unsigned char* xs = sm + kXsOff;             // 3-channel input: the FP32 RGBA halo as it landed
  constexpr int kBarOff = IN == kConvInBF16 ? kWBytes + kCHaloTx + 128 : kXsOff + kCXsB;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + kBarOff);     // the tile's MMAs completed
  uint64_t* xbar = bar + 1;                                         // the tile's TMA halo landed
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
  __shared__ float s_bias[32];
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = A.H, W = A.W;

  if (IN == kConvInRGBA)
    for (int i = tid; i < kCPairB / 16; i += kCThreads)  // the guard rows stay zero
      reinterpret_cast<uint4*>(sx)[i] = make_uint4(0u, 0u, 0u, 0u);
  else if (tid < 8)
    reinterpret_cast<uint4*>(sx + kCHaloTx)[tid] = make_uint4(0u, 0u, 0u, 0u);
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
  // Launched as a programmatic dependent, what is above overlaps the end of the kernel before; everything read below
  // is written by it or by earlier ones.  The next kernel launches as this one's CTAs leave: released at the start,
  // its CTAs slow this grid down (a training step 389 -> 371 us without), and they would have to wait until every CTA
  // here holds its tensor memory.
  griddep_wait();
  // Weights into core-matrix blocks: block b, K group g, row n at sw + b * kBlkB + (g * N + n) * 16.
  for (int i = tid; i < NB * 2 * N; i += kCThreads) {
    const int b = i / (2 * N), g = (i / N) & 1, n = i % N;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (IN == kConvInBF16 && !kStacked) {  // packed [tap][o][32]: block b = 2 tap + half, row n = o
      if (n < COUT) v = *reinterpret_cast<const uint4*>(A.wt + ((size_t)(b >> 1) * COUT + n) * 32 + 16 * (b & 1) + 8 * g);
    } else if (IN == kConvInBF16) {  // block b = 2 ky + half, row n = kx * S::kOutStep + o
      const int kx = n / S::kOutStep, o = n % S::kOutStep;
      if (kx < 3) v = *reinterpret_cast<const uint4*>(A.wt + ((size_t)(3 * (b >> 1) + kx) * COUT + o) * 32 + 16 * (b & 1) + 8 * g);
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
    *reinterpret_cast<uint4*>(sw + b * kBlkB + (g * N + n) * 16) = v;
  }
  if (tid < 32) s_bias[tid] = (EPI == kEpiRelu || (EPI != kEpiMask && tid < 3)) ? A.bias[tid] : 0.f;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // weights and zeros, to the tensor core and TMA
  __syncthreads();

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
  const uint32_t sx0 = c_su32(sx);  // 32 channels: halo position 0
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

    // ---- the tile's MMAs, a batch of kMB M-tiles at a time: M-tile m holds output positions 32 (4m + 1) + r, r < 128
    // (one thread issues them)
    auto issue = [&](int m0) {
      // A, 32 channels: positions (rows) of 64 bytes under the 64-byte swizzle, 8 of them 512 bytes on; the swizzle
      // goes by address, so a window's shift by whole positions and the second 16 channels only move the start.
      const uint64_t ad = IN == kConvInBF16 ? c_desc(sx0, 16, 512) | (4ull << 61)
                                            : c_desc(c_su32(sx) + kCGuard * 16, 32, 128);
      const uint64_t bd = c_desc(c_su32(sw), N * 16, 128);
      constexpr uint32_t id = c_idesc(128, N);
#pragma unroll (S::kMB == kCMT ? kCMT : 1)
      for (int m = m0; m < m0 + S::kMB; ++m) {
        const uint32_t d = tmem + (uint32_t)((m - m0) * N);
        if (IN == kConvInBF16 && !kStacked) {
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {  // tap 3 ky + kx reads positions 32 (4m + ky) + kx - 1 + r
#pragma unroll
            for (int h = 0; h < 2; ++h)
              c_mma(d, ad + (uint64_t)(int64_t)(4 * (32 * (4 * m + tap / 3) + tap % 3 - 1) + 2 * h),
                    bd + (uint64_t)((2 * tap + h) * (kBlkB / 16)), id, tap > 0 || h > 0);
          }
        }
#pragma unroll
        for (int ky = 0; ky < (IN == kConvInBF16 && !kStacked ? 0 : 3); ++ky) {
          if (IN == kConvInBF16) {  // kernel row ky reads positions 32 (4m + ky) + r, its columns lie along N
#pragma unroll
            for (int h = 0; h < 2; ++h)
              c_mma(d, ad + (uint64_t)(4 * 32 * (4 * m + ky) + 2 * h), bd + (uint64_t)((2 * ky + h) * (kBlkB / 16)), id,
                    ky > 0 || h > 0);
          } else {  // pairs from 32 (4m + ky) - 1
            c_mma(d, ad + (uint64_t)(int64_t)(32 * (4 * m + ky) - 1), bd + (uint64_t)(ky * (kBlkB / 16)), id, ky > 0);
          }
        }
      }
      c_commit(bar);
    };
    // every warp waits for the batch; false when a wait of the CTA gave up (the same for the whole CTA)
    auto landed = [&]() -> bool {
      if (lane == 0 && c_wait(bar, phase, A.wait_ns) != 0) {
        atomicOr(A.error, 64);
        s_abort = 1;
      }
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (s_abort) return false;
      issued = false;
      phase ^= 1u;
      return true;
    };
    // the accumulators of M-tile m are in registers in every warp: the next batch may overwrite them
    auto next_batch = [&](int m) {
      if (S::kMB == kCMT || m + 1 == kCMT) return;
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) issue(m + 1);
      issued = true;
    };
    if (tid == 0) issue(0);
    issued = true;

    // ---- epilogue: warp w reads lanes 32w.. (halo row 4m + 1 + w, column lane) of each M-tile.  Stacked, an
    // output is D[q-1][kx = 0] + D[q][1] + D[q+1][2]; the neighbours' parts come from the
    // neighbouring lanes (columns 0 and 31 get a wrong one and are never used).
    const uint32_t lane_base = (uint32_t)(32 * warp) << 16;
    const int gx = x0 + lane - 1;
    float lsum = 0.f;
    bool ok = true;
#pragma unroll (S::kMB == kCMT ? kCMT : 1)
    for (int m = 0; m < kCMT; ++m) {
      if (m % S::kMB == 0 && !landed()) {
        ok = false;
        break;
      }
      // the MMAs have read the halo: the next tile's copy lands during this epilogue
      if (IN == kConvInBF16 && tid == 0 && m == kCMT - S::kMB && tile + (int)gridDim.x < n_tiles) {
        int nimg, nx0, ny0;
        origin(tile + gridDim.x, nimg, nx0, ny0);
        c_load_halo(&tmap, sx0, xbar, nimg, nx0, ny0);
        halo_pending = true;
      }
      const int gy = y0 + 4 * m + warp;
      const bool store = lane >= 1 && lane <= kCTW && gy < H && gx < W;
      const uint32_t t = tmem + lane_base + (uint32_t)((m % S::kMB) * N);
      if (EPI == kEpiRelu || EPI == kEpiMask) {
        // after the transpose this lane holds piece lane % 4 of the pixels in columns (lane & ~3) + j
        const int col0 = lane & ~3;
        const size_t at0 = (((size_t)img * H + gy) * W + x0 + col0 - 1) * 32 + 8 * (lane & 3);
        bool keep[4];
        uint4 gate[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          keep[j] = col0 + j >= 1 && col0 + j <= kCTW && gy < H && x0 + col0 + j - 1 < W;
          gate[j] = make_uint4(0u, 0u, 0u, 0u);
          if (EPI == kEpiMask && keep[j]) gate[j] = *reinterpret_cast<const uint4*>(A.mask + at0 + 32 * j);
        }
        uint4 w[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // output channels 16 h .. 16 h + 15
          float v[16];
          if (kStacked) {
            float d0[16], d2[16];
            c_tmem_ld16(t + 16 * h, d0);
            c_tmem_ld16(t + 32 + 16 * h, v);
            c_tmem_ld16(t + 64 + 16 * h, d2);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (h == 1) next_batch(m);
#pragma unroll
            for (int k = 0; k < 16; ++k)
              v[k] += __shfl_up_sync(0xffffffffu, d0[k], 1) + __shfl_down_sync(0xffffffffu, d2[k], 1);
          } else {
            c_tmem_ld16(t + 16 * h, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          }
          uint32_t p[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float lo = v[2 * j], hi = v[2 * j + 1];
            if (EPI == kEpiRelu) {
              lo = fmaxf(lo + s_bias[16 * h + 2 * j], 0.f);
              hi = fmaxf(hi + s_bias[16 * h + 2 * j + 1], 0.f);
            }
            p[j] = c_pack(lo, hi);
          }
          w[2 * h] = make_uint4(p[0], p[1], p[2], p[3]);
          w[2 * h + 1] = make_uint4(p[4], p[5], p[6], p[7]);
        }
        c_transpose4(w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (!keep[j]) continue;
          if (EPI == kEpiMask)
            w[j] = make_uint4(c_gate(w[j].x, gate[j].x), c_gate(w[j].y, gate[j].y), c_gate(w[j].z, gate[j].z),
                              c_gate(w[j].w, gate[j].w));
          *reinterpret_cast<uint4*>(A.out_h + at0 + 32 * j) = w[j];
        }
      } else {  // kEpiResid / kEpiLoss: outputs 0..2; stacked, column kx in 4 kx ..
        const size_t pix = ((size_t)img * H + (store ? gy : 0)) * W + (store ? gx : 0);
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), tg = x;
        if (store) {
          x = reinterpret_cast<const float4*>(A.x)[pix];
          if (EPI == kEpiLoss) tg = reinterpret_cast<const float4*>(A.target)[pix];
        }
        float v[16], r[3];
        c_tmem_ld16(t, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int o = 0; o < 3; ++o)
          r[o] = (kStacked ? __shfl_up_sync(0xffffffffu, v[o], 1) + v[4 + o] + __shfl_down_sync(0xffffffffu, v[8 + o], 1)
                           : v[o]) + s_bias[o];
        if (!store) continue;
        if (EPI == kEpiResid) {
          const bool valid = x.w > 0.f;
          reinterpret_cast<float4*>(A.out_f)[pix] =
              valid ? make_float4(x.x + r[0], x.y + r[1], x.z + r[2], 1.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
          const bool valid = x.w > 0.f && tg.w > 0.f;
          const float d0 = valid ? (x.x + r[0]) - tg.x : 0.f;
          const float d1 = valid ? (x.y + r[1]) - tg.y : 0.f;
          const float d2 = valid ? (x.z + r[2]) - tg.z : 0.f;
          lsum += d0 * d0 + d1 * d1 + d2 * d2;
          reinterpret_cast<float4*>(A.out_f)[pix] =
              make_float4(2.f * loss_scale * d0, 2.f * loss_scale * d1, 2.f * loss_scale * d2, 0.f);
        }
      }
    }
    if (!ok) break;
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

// Tensor maps over an NHWC map: 32 BF16 channels as {32, W, H, n} under the 64-byte swizzle, or FP32 RGBA as
// {4, W, H, n}.
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

template <int IN, int COUT, int EPI, bool STACK = false>
cudaError_t launch_conv_tc_t(const RefineConvArgs& a, cudaStream_t s, bool pdl) {
  constexpr int kW = ConvShape<IN, COUT, STACK>::kWBytes;
  constexpr int used = 1024 + (IN == kConvInBF16 ? kW + kCHaloTx + 128 + 24
                                                 : (kW + kCXOff + kCPairB + 127) / 128 * 128 + kCXsB + 24);
  // At least 54 KB: no more than kCPerSM CTAs share an SM, so their tensor memory (128 columns each)
  // always fits and no CTA waits in tcgen05.alloc for another persistent CTA to finish.
  constexpr int smem = used < 54 * 1024 ? 54 * 1024 : used;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(conv_tc_kernel<IN, COUT, EPI, STACK>), smem);
  if (e != cudaSuccess) return e;
  const int n_tiles = ((a.W + kCTW - 1) / kCTW) * ((a.H + kCTH - 1) / kCTH) * a.n;
  if (n_tiles == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  // the halo copies' tensor map, over a 16-byte aligned base
  CUtensorMap tmap;
  std::memset(&tmap, 0, sizeof(tmap));
  const EncodeTiled enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const void* src = IN == kConvInBF16 ? static_cast<const void*>(a.src_h) : a.src_f;
  if ((reinterpret_cast<uintptr_t>(src) & 15u) != 0) return cudaErrorInvalidValue;
  if (!(IN == kConvInBF16 ? encode_map32(enc, &tmap, src, a.n, a.H, a.W, kCHW, kCHH)
                          : encode_rgba(enc, &tmap, src, a.n, a.H, a.W, kCHW, kCHH)))
    return cudaErrorInvalidValue;
  const int grid = n_tiles < sms * kCPerSM ? n_tiles : sms * kCPerSM;
  return launch_kernel(conv_tc_kernel<IN, COUT, EPI, STACK>, dim3(grid), dim3(kCThreads), smem, s, pdl, a, tmap);
}

}  // namespace

cudaError_t launch_refine_conv(int in_mode, int cout, int epi, const RefineConvArgs& a, cudaStream_t s, bool pdl,
                               bool inference) {
  const bool rgba = in_mode == kConvInRGBA, wide = cout == 32;
  if (rgba && wide && epi == kEpiRelu) return launch_conv_tc_t<kConvInRGBA, 32, kEpiRelu>(a, s, pdl);
  if (rgba && wide && epi == kEpiMask) return launch_conv_tc_t<kConvInRGBA, 32, kEpiMask>(a, s, pdl);
  if (!rgba && wide && epi == kEpiRelu)
    return inference ? launch_conv_tc_t<kConvInBF16, 32, kEpiRelu, true>(a, s, pdl)
                     : launch_conv_tc_t<kConvInBF16, 32, kEpiRelu>(a, s, pdl);
  if (!rgba && wide && epi == kEpiMask) return launch_conv_tc_t<kConvInBF16, 32, kEpiMask>(a, s, pdl);
  if (!rgba && cout == 8 && epi == kEpiResid) return launch_conv_tc_t<kConvInBF16, 8, kEpiResid, true>(a, s, pdl);
  if (!rgba && cout == 8 && epi == kEpiLoss) return launch_conv_tc_t<kConvInBF16, 8, kEpiLoss>(a, s, pdl);
  return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ weight gradients
//
// dW[o][c][ky][kx] = sum_p g[p][o] a[p + (ky - 1, kx - 1)][c], db[o] = sum_p g[p][o]
// (g = dL/dz of the layer's output, a = the layer's input), as one GEMM over
// K = pixels whose operands are the maps as they lie in memory: both are read
// MN-major (channels contiguous), so nothing is transposed.  Per image row r of a
// chunk of 32 x 2 pixels, and per kernel column kx,
//   D[kx][(i, c)][o] += sum_x a[r - 1 + i][x - 1 + kx][c] g[r][x][o]
// with M = 128: three rows i of a (ky = i) of 32 channels and, as the fourth, a row of
// ones, whose product with g is the bias gradient; N = the output channels.  A chunk's
// a lands by TMA as three rows of 34 positions (zeros outside the image) for each of
// its two pixel rows, each time in front of a constant row of ones.  A 32-channel map
// lies as [row][position][32 channels] under the 64-byte swizzle, which goes by
// address, so that a column's start one position on reads it correctly.  The
// 3-channel maps (the network input, dL/dr) land as FP32 RGBA and two warps round
// them to BF16 rows of 8 channels, the last five zero, without swizzle.
//   MODE 1: g = dL/dz1 (BF16, 32), a = the network input (FP32 RGBA, 3).  W1, b1.
//   MODE 2: g = dL/dz2 (BF16, 32), a = a1 (BF16, 32).                        W2, b2.
//   MODE 3: g = dL/dr  (FP32 RGBA, 3), a = a2 (BF16, 32).                    W3, b3.
//
// Order of the sums.  An MMA adds 16 neighbouring pixels of a row to an accumulator,
// the tensor core truncates as it adds, and Adam turns gradients that differ by 1e-6
// into weights that round to another BF16 neighbour a few steps later, so the order is
// part of the result: a chain of accumulation is one of A.n_rows (three per SM) that
// takes every n_rows-th chunk, row by row, and the chains are added in a fixed order
// (reduce_partials_kernel).  A CTA, one per SM, runs up to three chains in turn, each
// with accumulators of its own that stay in TMEM to the end.
//
// A ring of stages runs between a copying and an issuing warp per chain and two
// rounding warps.
// Bound by the MMAs (six per pixel row of 32, about 45 cycles each at N = 32: 28 us at
// 16 x 256^2), next to reading the maps (134 and 84 MB: 20 and 12 us) and some 10 us
// of start and end.  One thread issues an MMA per 59 cycles and a chunk's copies in
// some 600, hence the warps per chain (one of each: 57 us for W2).  Against kernels
// that transposed chunks of 64 pixels with ldmatrix and wrote every input nine times
// for its taps, 16 crops of 256^2, the same sums bit for bit: 109, 67 and 93 us for
// W2, W1 and W3 -> 43, 52 and 42 us.  (All nine taps in one MMA of N = 96, over positions of a
// instead of g, took 31, 25 and 23 us, but groups the pixels differently: gradients
// 1.5e-6 apart, 2e-4 after sixteen steps.)

namespace {

constexpr int kGTW = 32, kGTH = 2;               // chunk: 32 x 2 pixels
constexpr int kGHW = kGTW + 2, kGHR = 3;         // a: three rows of 34 positions per pixel row
constexpr int kGChains = 3;                      // accumulation chains per CTA, each with a copying and an issuing warp
constexpr int kGRoundWarp = 2 * kGChains;         // the first of two rounding warps
constexpr int kGThreads = 32 * (kGRoundWarp + 2);

template <int MODE>
struct WgradShape {
  static constexpr int N = MODE == 3 ? 16 : 32;
  static constexpr int COUT = MODE == 3 ? 3 : 32, CIN = MODE == 1 ? 3 : 32;
  static constexpr int kAPos = MODE == 1 ? 16 : 64, kARow = kGHW * kAPos;               // bytes per position, per row
  static constexpr int kAGrp = (kGHR + 1) * kARow;                                      // three rows and the ones
  static constexpr int kAB = (kGTH * kAGrp + 511) / 512 * 512;
  static constexpr int kGRow = kGTW * (MODE == 3 ? 16 : 64), kGB = kGTH * kGRow + (MODE == 3 ? 512 : 0);
  static constexpr int FW = MODE == 1 ? kGHW : kGTW, FH = MODE == 1 ? kGTH + 2 : kGTH;  // FP32 RGBA positions
  static constexpr int kFB = MODE == 2 ? 0 : FW * FH * 16;
  static constexpr int kStageB = (kAB + kGB + kFB + 511) / 512 * 512;
  static constexpr int kTx = (MODE == 1 ? 0 : kGTH * kGHR * kARow) + (MODE == 3 ? 0 : kGTH * kGRow) + kFB;
  static constexpr int kStages = 6;  // a multiple of 1, 2 and 3: a stage always serves the same chain
  static constexpr int kCols = MODE == 3 ? 256 : 512;  // TMEM: kGChains x 3 x N
  static_assert(kGChains * 3 * N <= kCols, "the accumulators fit");
  // M = 128 without swizzle takes 16 rows of a: beyond the ones they lie anywhere in shared memory (not used)
  static constexpr int kBarOff = kStages * kStageB + (MODE == 1 ? 8192 : 0);
  static constexpr int kSmem = 1024 + kBarOff + (3 * kStages + 1) * 8 + 16;  // 1024: the base is rounded up
  static_assert(kSmem <= 224 * 1024 && (MODE == 1 || kAGrp % 512 == 0), "fits; groups start on a swizzle atom");
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
  uint64_t* empty = ready + S::kStages;                            // its MMAs (and its rounding) are done
  uint64_t* done = empty + S::kStages;                             // all MMAs of the CTA are complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    s_abort = 0;
    for (int k = 0; k < S::kStages; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(c_su32(full + k)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(c_su32(ready + k)));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(c_su32(empty + k)), "r"(MODE == 2 ? 1 : 3));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(c_su32(done)), "r"(kGChains));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < S::kStages * kGTH * (S::kARow / 16); i += kGThreads) {  // the rows of ones, once
    const int row = i / (S::kARow / 16);
    *reinterpret_cast<uint4*>(sm + (row / kGTH) * S::kStageB + (row % kGTH) * S::kAGrp + kGHR * S::kARow +
                              (i % (S::kARow / 16)) * 16) = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // to the tensor core
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(c_su32(tslot)),
                 "r"(S::kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  griddep_wait();  // the maps are written by the kernels before (the next kernel's early blocks slow this one down:
                   // it lets them launch only by ending)
  const int cx = A.tiles_x, cxy = A.tiles_x * A.tiles_y, n_chunks = cxy * A.n;

  // The CTA's chunks, taken in turn from its n_ch chains (chain i is row blockIdx.x + i * gridDim.x): the j-th is
  // chunk j / n_ch of chain j % n_ch.
  int n_ch = 0, n_own = 0;
  for (int i = 0; i < kGChains; ++i) {
    const int v = blockIdx.x + i * gridDim.x;
    if (v < A.n_rows) {
      ++n_ch;
      n_own += v < n_chunks ? (n_chunks - v + A.n_rows - 1) / A.n_rows : 0;
    }
  }
  // A wait for use j of stage j % kStages; on give-up sets the error bit and the CTA's abort flag.
  auto wait_use = [&](uint64_t* bar, int j, int err) -> bool {
    if (s_abort) return false;
    if (c_wait(bar + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, A.wait_ns) == 0) return true;
    atomicOr(A.error, err);
    s_abort = 1;
    return false;
  };

  if (warp < kGChains) {
    // ---------------------------------------------------------------- copies, a warp per chain
    // Each lane works out the place of one of the chain's chunks, 32 at a time; lanes 0 .. 2 issue a copy each.
    int px = 0, py = 0, pimg = 0, k = 0, last = -1;
    for (int j = warp; warp < n_ch && j < n_own; j += n_ch, ++k) {
      if (k % 32 == 0) {
        const int chunk = blockIdx.x + warp * gridDim.x + (k + lane) * A.n_rows;
        pimg = chunk / cxy;
        const int rem = chunk - pimg * cxy;
        py = rem / cx * kGTH;
        px = rem % cx * kGTW;
      }
      const int x0 = __shfl_sync(0xffffffffu, px, k % 32), y0 = __shfl_sync(0xffffffffu, py, k % 32);
      const int img = __shfl_sync(0xffffffffu, pimg, k % 32);
      uint64_t* bar = full + j % S::kStages;
      int ok = 1;
      if (lane == 0) {
        ok = j < S::kStages || wait_use(empty, j - S::kStages, 256);
        if (ok)
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(c_su32(bar)), "r"(S::kTx) : "memory");
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      const uint32_t st = c_su32(sm) + (j % S::kStages) * S::kStageB, sg = st + S::kAB, sf = sg + S::kGB;
      if (lane < kGTH) {
        if (MODE != 1) g_tma4(&amap, st + lane * S::kAGrp, bar, 0, x0 - 1, y0 + lane - 1, img);
        else if (lane == 0) g_tma4(&amap, sf, bar, 0, x0 - 1, y0 - 1, img);
      } else if (lane == kGTH) {
        g_tma4(&gmap, MODE == 3 ? sf : sg, bar, 0, x0, y0, img);
      }
      __syncwarp();
      last = j;
    }
    // the last copies land before the CTA can leave (earlier ones have been waited for by their readers)
    if (lane == 0)
      for (int j = last; j >= 0 && j > last - S::kStages; j -= n_ch)
        if (c_wait(full + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, kCDrainNs) != 0) atomicOr(A.error, 2048);
  } else if (warp < kGRoundWarp) {
    // ---------------------------------------------------------------- MMAs, a warp per chain (one thread issues an
    // MMA per 59 cycles, so one alone would hold the tensor core up)
    if (lane == 0) {
      constexpr uint32_t id = g_idesc(128, S::N);
      constexpr int kAK = 16 * S::kAPos, kGK = S::kGRow / 2;  // 16 positions
      const int chain = warp - kGChains;
      const uint32_t d = tmem + chain * 3 * S::N;
      for (int j = chain; chain < n_ch && j < n_own; j += n_ch) {
        if (!wait_use(full, j, 256)) break;
        if (MODE != 2 && !wait_use(ready, j, 256)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st = c_su32(sm) + (j % S::kStages) * S::kStageB;
        const uint64_t ad = MODE == 1 ? g_desc8(st, S::kARow) : g_desc32(st, S::kARow);
        const uint64_t bd = MODE == 3 ? g_desc8(st + S::kAB, 512) : g_desc32(st + S::kAB, 512);
#pragma unroll
        for (int r = 0; r < kGTH; ++r)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
              c_mma(d + kx * S::N, ad + (uint64_t)((r * S::kAGrp + kx * S::kAPos + h * kAK) / 16),
                    bd + (uint64_t)((r * S::kGRow + h * kGK) / 16), id, j > chain || r > 0 || h > 0);
        c_commit(empty + j % S::kStages);
      }
      // completes once every MMA issued (by all three) has: also after an abort, so the tensor memory is never freed
      // under one
      c_commit(done);
      if (c_wait(done, 0u, A.wait_ns > kCDrainNs ? A.wait_ns : kCDrainNs) != 0) atomicOr(A.error, 512);
    }
  } else if (MODE != 2) {
    // ---------------------------------------------------------------- rounding of FP32 maps
    const int t = tid - 32 * kGRoundWarp;
    for (int j = 0; j < n_own; ++j) {
      int ok = 1;
      if (lane == 0) ok = wait_use(full, j, 1024);
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      // every lane tests the phase itself: the copies are visible to it
      if (c_wait(full + j % S::kStages, (uint32_t)(j / S::kStages) & 1u, kCDrainNs) != 0) break;
      unsigned char* st = sm + (j % S::kStages) * S::kStageB;
      const float4* f = reinterpret_cast<const float4*>(st + S::kAB + S::kGB);
      for (int i = t; i < S::FW * S::FH; i += 64) {
        const float4 v = f[i];
        const uint4 w = make_uint4(c_pack(v.x, v.y), c_pack(v.z, 0.f), 0u, 0u);
        if (MODE == 3) {
          reinterpret_cast<uint4*>(st + S::kAB)[i] = w;  // [row][position]
        } else {  // row y of the four is row y of the first pixel row's three, y - 1 of the second's
          const int y = i / S::FW, x = i - y * S::FW;
#pragma unroll
          for (int r = 0; r < kGTH; ++r)
            if (y - r >= 0 && y - r < kGHR) *reinterpret_cast<uint4*>(st + r * S::kAGrp + (y - r) * S::kARow + x * 16) = w;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the tensor core
      __syncwarp();
      if (lane == 0) {
        g_arrive(ready + j % S::kStages);
        g_arrive(empty + j % S::kStages);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();  // the MMAs are complete (the issuing threads have waited for them)
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // ---- the chains' partial rows, [ky][kx][o][c] then the biases: warp w reads accumulator rows 32w ..
  if (!s_abort && warp < (MODE == 1 ? 1 : 4)) {
    const int ky = MODE == 1 ? lane >> 3 : warp, c = MODE == 1 ? lane & 7 : lane;
    for (int i = 0; i < kGChains; ++i) {
      const int v = blockIdx.x + i * gridDim.x;
      if (v >= A.n_rows) break;
      float* out = A.partial + (size_t)v * A.seg;
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        float d[S::N];
#pragma unroll
        for (int h = 0; h < S::N / 16; ++h) {
          float u[16];
          c_tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (i * 3 + kx) * S::N + 16 * h, u);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int q = 0; q < 16; ++q) d[16 * h + q] = u[q];
        }
        if (ky < 3 && c < S::CIN) {
#pragma unroll
          for (int o = 0; o < S::COUT; ++o) out[((ky * 3 + kx) * S::COUT + o) * S::CIN + c] = d[o];
        }
        if (ky == 3 && c == 0 && kx == 0) {
#pragma unroll
          for (int o = 0; o < S::COUT; ++o) out[9 * S::COUT * S::CIN + o] = d[o];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kCols));
  }
}

namespace {

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
                             : encode_map32(enc, &am, a.a_h, a.n, a.H, a.W, kGHW, kGHR)) &&
                  (MODE == 3 ? encode_rgba(enc, &gm, a.g_f, a.n, a.H, a.W, S::FW, S::FH)
                             : encode_map32(enc, &gm, a.g_h, a.n, a.H, a.W, kGTW, kGTH));
  if (!ok) return cudaErrorInvalidValue;
  return launch_kernel(wgrad_tc_kernel<MODE>, dim3(a.n_ctas), dim3(kGThreads), S::kSmem, s, true, a, am, gm);
}

}  // namespace

cudaError_t launch_refine_wgrad(int mode, const RefineWgradArgs& a, cudaStream_t s) {
  if (mode == 1) return launch_wgrad_tc_t<1>(a, s);
  if (mode == 2) return launch_wgrad_tc_t<2>(a, s);
  if (mode == 3) return launch_wgrad_tc_t<3>(a, s);
  return cudaErrorInvalidValue;
}

void refine_wgrad_shape(RefineWgradArgs& g, int sm_count) {
  g.tiles_x = (g.W + kGTW - 1) / kGTW;
  g.tiles_y = (g.H + kGTH - 1) / kGTH;
  const int64_t blocks = (int64_t)g.tiles_x * ((g.H + 7) / 8) * g.n;  // chains of at least one chunk
  g.n_rows = (int)std::max<int64_t>(1, std::min<int64_t>(blocks, (int64_t)kGChains * sm_count));
  g.n_ctas = std::min(g.n_rows, sm_count);
}

}  // namespace lfk
