// Training of the learned post-smoother on the 5th-generation tensor cores
// (tcgen05, sm_103a): the whole backward pass of the network in one kernel, every
// activation and every intermediate gradient on chip.
//
// k_tc_back, a persistent CTA per SM, walks tiles of 14 x 6 pixels x 8 pairs.  From the
// residual r (tile + 3 pixels) and gD = dL/dN (tile + 2) it forms, per tile,
//   a+- = bf16(relu(+-z1)), z1 = W1 * r           (tile + 2, CUDA cores, float32)
//   z2+- = W2 * a+-                               (tile + 1, MMA)
//   gh = W3^T * gD, h = (relu(z2+) - relu(z2-))/2 (CUDA cores, float32)
//   g+- = bf16(+-gh / 2 where z2+- > 0)           (tile + 1)
//   ga+- = W2^T * g+-                             (tile, MMA)
//   gz1 = ga+ [z1 > 0] - ga- [z1 < 0]             (tile, float32)
// and adds to the weight gradients, each summed over the tile's own pixels p:
//   gW1[tap] += r[p + tap] gz1[p],  gW3[tap] += h[p] gD[p - tap]   (CUDA cores, float32)
//   gW2[tap] += a+[p + tap] g+[p] + a-[p + tap] g-[p]              (MMA, in TMEM across tiles)
//
// One layout serves the three MMA products: [branch][pixel][channel half][pair][8 channels]
// bf16, 256 bytes a pixel.  As the convolutions' A operand it is K-major (K = channels, rows =
// pixel x 8 + pair; 8-row groups 256 B apart, the two channel halves 128 B); as both operands of
// the weight gradient it is MN-major (K = pixel x 8 + pair, 256 B apart; 8-channel groups 128 B),
// and since groups 128 B apart run on into the next pixel, the 128 M rows are the 16 channels of 8
// consecutive pixels: rows 0..47 are the taps dx = 0, 1, 2 of one dy (the others are not used).
// So a K step (two pixels) takes 6 MMAs (3 dy x 2 branches) instead of one per tap and branch.
// One thread alone issues an MMA this small every 74 clocks, 16 together one every 33 (measured in the
// inference kernel), so one thread of every warp issues: a row and branch each of the convolutions, one dy
// and quarter of the K steps each of the weight gradient.
//
// What bounds it: the phases of a tile are serial (one CTA fills the SM's shared memory), the tensor
// core (busy 52 % of the time) and the float32 pipe taking turns.  Before it, the backward pass went through HBM
// with 13 launches and about 20 passes over [pixel][pair][16] float32 activations, and layers 1 and
// 3 summed their weight gradients with 9 and 144 threads a block.  Loss and gradient at h = 1/256,
// k = 64 (all kernels): 9.91 ms before, 1.32 ms with this kernel and the fused forward.
//
// Every mbarrier wait is bounded; a wait that gives up increments an error counter, the kernel
// stops walking tiles, contributes zeros and frees its TMEM.
#include "common.cuh"
#include "smoother.cuh"

#include <cuda_bf16.h>
#include <stdint.h>

namespace pasm {
namespace {

constexpr int PB = 8;                    // pairs per tile
constexpr int TW = 14, TR = 6;           // tile (pixels)
constexpr int HW = TW + 2, HR = TR + 2;  // z2, g+-: 16 x 8 (one 128-row MMA block per row)
constexpr int AW = TW + 4, AR = TR + 4;  // a+-, gD: 18 x 10
constexpr int RW = TW + 6, RR = TR + 6;  // r: 20 x 12
constexpr int kThreads = 512;
constexpr int kGroups = kThreads / 128;  // pixel groups of the layer 1 and 3 weight gradients
constexpr int kWaitLimit = 1 << 22;
constexpr int kCtas = kMaxBackRows;      // persistent: one per SM

constexpr int kPix = 256;                           // bytes of one pixel of one branch
constexpr int kABranch = AR * AW * kPix;
constexpr int kGBranch = HR * HW * kPix;
constexpr int kABytes = 2 * kABranch;
constexpr int kGBytes = 2 * kGBranch + 2 * kPix;    // 2 pixels of slack: the last row's unused outputs read on
constexpr int kFBytes = TR * TW * PB * 16 * 4;      // h, then gz1: [pixel][pair][16] float32
constexpr int kRBytes = RR * RW * PB * 4;
constexpr int kDBytes = AR * AW * PB * 4;
constexpr int kW2Bytes = 9 * 512;                   // bf16, canonical K-major, per tap 2x2 core matrices
constexpr int kWBytes = 2 * 144 * 4;                // layers 1 and 3
constexpr int kSmem = kABytes + kGBytes + kFBytes + kRBytes + kDBytes + 2 * kW2Bytes + kWBytes + 64;
static_assert(kSmem <= 227 * 1024, "one CTA per SM");
static_assert(HW * PB == 128, "one MMA block per row");
// the weight gradient's M rows reach 7 pixels past the last K pixel of the last tap row
static_assert((TR + 2) * AW + TW + 7 < AR * AW, "M rows of the weight gradient stay inside the operand");
constexpr uint32_t kTmemCols = 512;                 // 256 of z2 / ga, 192 of gW2
constexpr uint32_t kTmemW = HR * 2 * 16;            // first column of gW2
constexpr int kGradIssuers = TR * 2;                // MMA-issuing threads after z2: one per row and branch
constexpr int kGradParts = kGradIssuers / 3;        // gW2: 3 dy x kGradParts accumulators
static_assert(kGradIssuers % 3 == 0 && kTmemW + kGradIssuers * 16 <= kTmemCols, "accumulators of gW2");
static_assert(HR * 2 == kThreads / 32, "one issuer of z2 per warp");
static_assert(kThreads * 9 * 4 <= kABytes, "the final reduction reuses the operand space");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle.  K-major: lbo = distance of the two 8-element K
// chunks, sbo = of 8-row groups; MN-major: lbo = distance of 8-element K groups, sbo = of 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// kind::f16, D f32, A and B bf16, N = 16, M = 128; K-major operands, or both MN-major (bits 15, 16)
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(16 >> 3) << 17) |
                            ((uint32_t)(128 >> 4) << 24);
constexpr uint32_t kIdescMN = kIdesc | (1u << 15) | (1u << 16);

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar)));
}

// bounded wait for the mbarrier phase `parity`; true when it completed
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity) {
  uint32_t done = 0;
  for (int it = 0; it < kWaitLimit && !done; ++it) {
    asm volatile(
        "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(parity));
  }
  return done != 0;
}

// The same for the whole CTA: one thread polls, the others wait at the barrier.
__device__ __forceinline__ bool cta_wait(uint64_t* mbar, uint32_t parity) {
  return __syncthreads_or(threadIdx.x == 0 && mbar_wait(mbar, parity)) != 0;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

// 8 pairs of a [pixel][ldk] float32 grid vector on a tile (height x width pixels from (x0, y0)), zero
// outside the grid and for pairs c >= k: asynchronous 16-byte copies where all 8 pairs are real.
__device__ __forceinline__ void load_tile(const float* __restrict__ src, int nx, int ny, int ldk, int k, int x0,
                                          int y0, int c0, int height, int width, float* dst) {
  if (c0 + PB <= k) {
    for (int t = threadIdx.x; t < height * width * 2; t += kThreads) {
      const int hlf = t & 1, col = (t >> 1) % width, row = (t >> 1) / width;
      const int x = x0 + col, y = y0 + row;
      const bool in = x >= 0 && x < nx && y >= 0 && y < ny;
      const float* s = in ? src + ((int64_t)y * nx + x) * ldk + c0 + 4 * hlf : src;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst + (row * width + col) * PB + 4 * hlf)),
                   "l"(s), "r"(in ? 16 : 0));
    }
  } else {
    for (int t = threadIdx.x; t < height * width * PB; t += kThreads) {
      const int q = t % PB, col = (t / PB) % width, row = t / (PB * width);
      const int x = x0 + col, y = y0 + row, c = c0 + q;
      float v = 0.f;
      if (x >= 0 && x < nx && y >= 0 && y < ny && c < k) v = src[((int64_t)y * nx + x) * ldk + c];
      dst[t] = v;
    }
  }
}

// acc[tap] += v[p] w[p + s (tap - centre)] over this thread's pixels of the tile: v = h or gz1
// ([pixel][pair][16], thread = one channel and pair), w a scalar tile `ww` wide whose pixel (off, off)
// is the tile's first.  Thread group g takes every kGroups-th run of 7 pixels; the 3 x 3 window of w
// slides along the run.
template <int S>
__device__ __forceinline__ void tap_sums(const float* v, const float* w, int ww, int off, int c, int q, int g,
                                         float (&acc)[9]) {
  for (int seg = g; seg < TR * 2; seg += kGroups) {
    const int i = seg >> 1, j0 = (seg & 1) * (TW / 2);
    const float* wr = w + ((off + i - 1) * ww + off + j0 - 1) * PB + q;
    float win[3][3];
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) win[dy][dx + 1] = wr[(dy * ww + dx) * PB];
#pragma unroll
    for (int j = 0; j < TW / 2; ++j) {
#pragma unroll
      for (int dy = 0; dy < 3; ++dy) {
        win[dy][0] = win[dy][1];
        win[dy][1] = win[dy][2];
        win[dy][2] = wr[(dy * ww + j + 2) * PB];
      }
      const float x = v[((i * TW + j0 + j) * PB + q) * 16 + c];
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const int tap = S > 0 ? dy * 3 + dx : 8 - (dy * 3 + dx);
          acc[tap] = fmaf(x, win[dy][dx], acc[tap]);
        }
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1)
    k_tc_back(int nx, int ny, int ldk, int k, int tiles_x, int tiles_xy, int n_tiles, const float* __restrict__ W,
              const uint8_t* __restrict__ w2f, const uint8_t* __restrict__ w2t, const float* __restrict__ R,
              const float* __restrict__ gD, float* __restrict__ partial, int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sa = smem;                                        // a+-
  uint8_t* sg = sa + kABytes;                                // g+-
  float* sf = reinterpret_cast<float*>(sg + kGBytes);        // h, then gz1
  float* sr = sf + kFBytes / 4;
  float* sd = sr + kRBytes / 4;
  uint8_t* sw2f = reinterpret_cast<uint8_t*>(sd + kDBytes / 4);
  uint8_t* sw2t = sw2f + kW2Bytes;
  float* sw1 = reinterpret_cast<float*>(sw2t + kW2Bytes);    // [tap][16]
  float* sw3 = sw1 + 144;                                    // [tap][16]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sw3 + 144);   // z2, ga, gW2
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar + 3);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(HR * 2));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + 1)), "r"(kGradIssuers));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + 2)), "r"(kGradIssuers));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
  for (int t = tid; t < kW2Bytes / 16; t += kThreads) {
    reinterpret_cast<uint4*>(sw2f)[t] = __ldg(reinterpret_cast<const uint4*>(w2f) + t);
    reinterpret_cast<uint4*>(sw2t)[t] = __ldg(reinterpret_cast<const uint4*>(w2t) + t);
  }
  for (int t = tid; t < 288; t += kThreads) sw1[t] = __ldg(W + (t < 144 ? t : t + 2304));
  for (int t = tid; t < 2 * kPix / 16; t += kThreads)
    reinterpret_cast<uint4*>(sg + 2 * kGBranch)[t] = make_uint4(0, 0, 0, 0);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tmem_slot;

  // epilogue mapping: TMEM lane m = pixel j x 8 + pair q of a row; rows i = rowgrp, rowgrp + 4
  const int quarter = warp & 3, rowgrp = warp >> 2;
  const int m = quarter * 32 + lane, ej = m / PB, eq = m % PB;
  const uint32_t lanebase = tmem + ((uint32_t)(quarter * 32) << 16);
  // weight-gradient mapping of layers 1 and 3: channel, pair, pixel group
  const int wc = tid & 15, wq = (tid >> 4) & 7, wg = tid >> 7;
  float acc1[9], acc3[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) acc1[t] = acc3[t] = 0.f;

  bool ok = true;
  uint32_t walked = 0, phase = 0;
  int pending = 0;   // barriers with MMAs in flight
  for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++walked) {
    phase = walked & 1u;
    const int txy = tile % tiles_xy, c0 = (tile / tiles_xy) * PB;
    const int x0 = (txy % tiles_x) * TW, y0 = (txy / tiles_x) * TR;
    load_tile(R, nx, ny, ldk, k, x0 - 3, y0 - 3, c0, RR, RW, sr);
    load_tile(gD, nx, ny, ldk, k, x0 - 2, y0 - 2, c0, AR, AW, sd);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // layer 1: a+- as bf16 on the tile + 2, zero outside the grid
    for (int t = tid; t < AR * AW * PB; t += kThreads) {
      const int q = t % PB, pix = t / PB, col = pix % AW, row = pix / AW;
      const int x = x0 - 2 + col, y = y0 - 2 + row;
      float z[16];
#pragma unroll
      for (int o = 0; o < 16; ++o) z[o] = 0.f;
      if (x >= 0 && x < nx && y >= 0 && y < ny) {
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const float v = sr[((row + tap / 3) * RW + (col + tap % 3)) * PB + q];
          const float4* w = reinterpret_cast<const float4*>(sw1 + tap * 16);
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const float4 w4 = w[o];
            z[4 * o + 0] = fmaf(w4.x, v, z[4 * o + 0]);
            z[4 * o + 1] = fmaf(w4.y, v, z[4 * o + 1]);
            z[4 * o + 2] = fmaf(w4.z, v, z[4 * o + 2]);
            z[4 * o + 3] = fmaf(w4.w, v, z[4 * o + 3]);
          }
        }
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        __align__(16) __nv_bfloat162 vp[4], vm[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) {   // relu(+-z) of the rounded z, as in the inference kernel
          const __nv_bfloat162 b = __floats2bfloat162_rn(z[half * 8 + 2 * o], z[half * 8 + 2 * o + 1]);
          const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
          vp[o] = __hmax2(b, zero);
          vm[o] = __hmax2(__hneg2(b), zero);
        }
        uint8_t* dst = sa + pix * kPix + half * 128 + q * 16;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<uint4*>(vp);
        *reinterpret_cast<uint4*>(dst + kABranch) = *reinterpret_cast<uint4*>(vm);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (lane == 0) {   // one row and branch per warp
      const int i = warp >> 1, b = warp & 1;
      const uint64_t ai = smem_desc(smem_u32(sa) + (uint32_t)(b * kABranch + i * AW * kPix), 128, kPix);
      const uint64_t b0 = smem_desc(smem_u32(sw2f), 128, 256);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap)
        mma_bf16(tmem + (uint32_t)((i * 2 + b) * 16), ai + (uint64_t)(((tap / 3 * AW + tap % 3) * kPix) >> 4),
                 b0 + (uint64_t)(tap * 512 >> 4), kIdesc, tap > 0 ? 1u : 0u);
      mma_commit(mbar);
    }
    pending = 1;
    // gh for this thread's two rows while the MMAs run: (W3^T * gD), float32
    float gh[2][16];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = rowgrp + 4 * e;
#pragma unroll
      for (int o = 0; o < 16; ++o) gh[e][o] = 0.f;
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const float v = sd[((i + tap / 3) * AW + (ej + tap % 3)) * PB + eq];
        const float4* w = reinterpret_cast<const float4*>(sw3 + (8 - tap) * 16);
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const float4 w4 = w[o];
          gh[e][4 * o + 0] = fmaf(w4.x, v, gh[e][4 * o + 0]);
          gh[e][4 * o + 1] = fmaf(w4.y, v, gh[e][4 * o + 1]);
          gh[e][4 * o + 2] = fmaf(w4.z, v, gh[e][4 * o + 2]);
          gh[e][4 * o + 3] = fmaf(w4.w, v, gh[e][4 * o + 3]);
        }
      }
    }
    ok = cta_wait(mbar, phase);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int i = rowgrp + 4 * e;
        float vp[16], vm[16];
        tmem_ld16(lanebase + (uint32_t)((i * 2 + 0) * 16), vp);
        tmem_ld16(lanebase + (uint32_t)((i * 2 + 1) * 16), vm);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        const int x = x0 - 1 + ej, y = y0 - 1 + i;
        const bool in = x >= 0 && x < nx && y >= 0 && y < ny;
        if (i >= 1 && i <= TR && ej >= 1 && ej <= TW) {   // h on the tile's own pixels
          float4* dst = reinterpret_cast<float4*>(sf + (((i - 1) * TW + ej - 1) * PB + eq) * 16);
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            float4 h4;
            h4.x = in ? 0.5f * (fmaxf(vp[4 * o], 0.f) - fmaxf(vm[4 * o], 0.f)) : 0.f;
            h4.y = in ? 0.5f * (fmaxf(vp[4 * o + 1], 0.f) - fmaxf(vm[4 * o + 1], 0.f)) : 0.f;
            h4.z = in ? 0.5f * (fmaxf(vp[4 * o + 2], 0.f) - fmaxf(vm[4 * o + 2], 0.f)) : 0.f;
            h4.w = in ? 0.5f * (fmaxf(vp[4 * o + 3], 0.f) - fmaxf(vm[4 * o + 3], 0.f)) : 0.f;
            dst[o] = h4;
          }
        }
        uint8_t* dg = sg + (i * HW + ej) * kPix + eq * 16;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          __align__(16) __nv_bfloat162 gp[4], gm[4];
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const int u = half * 8 + 2 * o;
            gp[o] = __floats2bfloat162_rn(in && vp[u] > 0.f ? 0.5f * gh[e][u] : 0.f,
                                          in && vp[u + 1] > 0.f ? 0.5f * gh[e][u + 1] : 0.f);
            gm[o] = __floats2bfloat162_rn(in && vm[u] > 0.f ? -0.5f * gh[e][u] : 0.f,
                                          in && vm[u + 1] > 0.f ? -0.5f * gh[e][u + 1] : 0.f);
          }
          *reinterpret_cast<uint4*>(dg + half * 128) = *reinterpret_cast<uint4*>(gp);
          *reinterpret_cast<uint4*>(dg + half * 128 + kGBranch) = *reinterpret_cast<uint4*>(gm);
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (!ok) break;
    pending = 6;
    if (lane == 0 && warp < kGradIssuers) {
      // input gradients ga+- of one row and branch (outputs 14, 15 of a row are not used)
      const int i = warp >> 1, b = warp & 1;
      const uint64_t gi = smem_desc(smem_u32(sg) + (uint32_t)(b * kGBranch + i * HW * kPix), 128, kPix);
      const uint64_t t0 = smem_desc(smem_u32(sw2t), 128, 256);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap)
        mma_bf16(tmem + (uint32_t)((i * 2 + b) * 16), gi + (uint64_t)(((tap / 3 * HW + tap % 3) * kPix) >> 4),
                 t0 + (uint64_t)(tap * 512 >> 4), kIdesc, tap > 0 ? 1u : 0u);
      mma_commit(mbar + 1);
      // weight gradient of one dy over a quarter of the K steps, in an accumulator of its own: K = two
      // pixels of the tile a step; rows = 16 channels of the pixels dx = 0..7
      const int dy = warp % 3, part = warp / 3;
      const uint32_t acc = tmem + kTmemW + (uint32_t)((part * 3 + dy) * 16);
      const uint64_t am = smem_desc(smem_u32(sa), kPix, 128);
      const uint64_t gm = smem_desc(smem_u32(sg), kPix, 128);
      for (int st = part; st < TR * TW / 2; st += kGradParts) {
        const int r = st / (TW / 2), j = 2 * (st % (TW / 2));
#pragma unroll
        for (int q = 0; q < 2; ++q)
          mma_bf16(acc, am + (uint64_t)((q * kABranch + ((r + 1 + dy) * AW + j + 1) * kPix) >> 4),
                   gm + (uint64_t)((q * kGBranch + ((r + 1) * HW + j + 1) * kPix) >> 4), kIdescMN,
                   (walked > 0 || st > part || q > 0) ? 1u : 0u);
      }
      mma_commit(mbar + 2);
    }
    tap_sums<-1>(sf, sd, AW, 2, wc, wq, wg, acc3);
    ok = cta_wait(mbar + 1, phase);   // its barrier: h is read, gz1 takes its place
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
      for (int i = rowgrp; i < TR; i += 4) {
        float vp[16], vm[16];
        tmem_ld16(lanebase + (uint32_t)((i * 2 + 0) * 16), vp);
        tmem_ld16(lanebase + (uint32_t)((i * 2 + 1) * 16), vm);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        if (ej < TW) {
          const bool in = x0 + ej < nx && y0 + i < ny;
          const uint8_t* pa = sa + ((i + 2) * AW + ej + 2) * kPix + eq * 16;
          float4* dst = reinterpret_cast<float4*>(sf + ((i * TW + ej) * PB + eq) * 16);
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            // the sign of z1: a+ > 0 or a- > 0 (never both)
            const uint4 up = *reinterpret_cast<const uint4*>(pa + half * 128);
            const uint4 um = *reinterpret_cast<const uint4*>(pa + half * 128 + kABranch);
            const uint32_t p4[4] = {up.x, up.y, up.z, up.w}, m4[4] = {um.x, um.y, um.z, um.w};
            float g8[8];
#pragma unroll
            for (int o = 0; o < 8; ++o) {
              const uint32_t mask = o & 1 ? 0xFFFF0000u : 0xFFFFu;
              const int u = half * 8 + o;
              g8[o] = in ? ((p4[o / 2] & mask) ? vp[u] : 0.f) - ((m4[o / 2] & mask) ? vm[u] : 0.f) : 0.f;
            }
            dst[half * 2] = make_float4(g8[0], g8[1], g8[2], g8[3]);
            dst[half * 2 + 1] = make_float4(g8[4], g8[5], g8[6], g8[7]);
          }
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    ok = __syncthreads_and(ok);
    tap_sums<1>(sf, sr, RW, 3, wc, wq, wg, acc1);
    // the next tile overwrites the operands
    ok = cta_wait(mbar + 2, phase) && ok;
    asm volatile("tcgen05.fence::after_thread_sync;");
  }
  if (!ok && tid == 0) {
    atomicAdd(err, 1);
    // MMAs that a wait gave up on still read shared memory: wait (bounded) before it is reused
    for (int b = 0; b < 3; ++b)
      if (pending >> b & 1) mbar_wait(mbar + b, phase);
  }
  __syncthreads();
  // this CTA's row of partial sums, in the order of the weights; zeros without tiles or after an error
  float* out = partial + (size_t)blockIdx.x * kNNWeights;
  const bool have = ok && walked > 0;
  if (warp < 2) {
    // accumulator row dx * 16 + ci (rows 48.. unused), columns dy * 16 + co
#pragma unroll 1
    for (int dy = 0; dy < 3; ++dy) {
      float v[16];
      if (have) {
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + kTmemW + (uint32_t)(dy * 16), v);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll 1
        for (int part = 1; part < kGradParts; ++part) {
          float u[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + kTmemW + (uint32_t)((part * 3 + dy) * 16), u);
          asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
          for (int o = 0; o < 16; ++o) v[o] += u[o];
        }
      } else {
#pragma unroll
        for (int o = 0; o < 16; ++o) v[o] = 0.f;
      }
      const int row = warp * 32 + lane, dx = row >> 4, ci = row & 15;
      if (dx < 3) {
        float4* dst = reinterpret_cast<float4*>(out + 144 + ((dy * 3 + dx) * 16 + ci) * 16);
#pragma unroll
        for (int o = 0; o < 4; ++o) dst[o] = make_float4(v[4 * o], v[4 * o + 1], v[4 * o + 2], v[4 * o + 3]);
      }
    }
  }
  // layers 1 and 3: over the 8 pairs and the pixel groups, in a fixed order
  float* red = reinterpret_cast<float*>(smem);   // [kThreads / 16][9][16]
  for (int pass = 0; pass < 2; ++pass) {
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 9; ++t) red[((tid >> 4) * 9 + t) * 16 + wc] = have ? (pass ? acc3[t] : acc1[t]) : 0.f;
    __syncthreads();
    if (tid < 144) {
      float s = 0.f;
      for (int r = 0; r < kThreads / 16; ++r) s += red[r * 144 + tid];
      out[(pass ? 144 + 2304 : 0) + tid] = s;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// Layer 2's kernel W[tap][ci][co] (float32, device) in the canonical bf16 operand layout of the
// B matrix (row n = output channel, k = input channel, per tap two 8 x 8 core matrices along n,
// 256 B apart, and two along k, 128 B apart), and the kernel of the input gradient,
// Wt[tap][co][ci] = W[8 - tap][ci][co] (output and input channels exchanged), in the same layout.
__global__ void k_tc_w2_layout(const float* __restrict__ W, uint16_t* __restrict__ fwd, uint16_t* __restrict__ flip) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 2304) return;
  const int tap = t / 256, ci = (t / 16) % 16, co = t % 16;   // W index t = [tap][ci][co]
  const __nv_bfloat16 b = __float2bfloat16_rn(W[t]);
  const uint16_t bits = *reinterpret_cast<const uint16_t*>(&b);
  fwd[(tap * 512 + (co % 8) * 16 + (co / 8) * 256 + (ci / 8) * 128 + (ci % 8) * 2) / 2] = bits;
  flip[((8 - tap) * 512 + (ci % 8) * 16 + (ci / 8) * 256 + (co / 8) * 128 + (co % 8) * 2) / 2] = bits;
}

}  // namespace

cudaError_t nn_tc_train_prepare() {
  return cudaFuncSetAttribute(k_tc_back, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

void nn_tc_w2_layout(const Launch& L, const float* W2, uint16_t* fwd, uint16_t* flip) {
  L.begin(KC_NN, 2304 * 8.0, 0);
  k_tc_w2_layout<<<(2304 + 255) / 256, 256, 0, L.s>>>(W2, fwd, flip);
  L.bump();
}

int nn_backward_tc(const Launch& L, const NNGrid& g, const float* W, const uint16_t* w2f, const uint16_t* w2t,
                   const float* R, const float* gD, float* partial, int* err) {
  const int tiles_x = (g.nx + TW - 1) / TW, tiles_y = (g.ny + TR - 1) / TR;
  const int n_tiles = tiles_x * tiles_y * (g.ldk / PB);
  const int ctas = n_tiles < kCtas ? n_tiles : kCtas;
  const double pp = (double)g.nx * g.ny * g.ldk;
  L.begin(KC_NN, pp * 8.0, pp * 2.0 * (3 * 2 * 9 * 256 + 4 * 9 * 16));
  k_tc_back<<<ctas, kThreads, kSmem, L.s>>>(g.nx, g.ny, g.ldk, g.k, tiles_x, tiles_x * tiles_y, n_tiles, W,
                                            reinterpret_cast<const uint8_t*>(w2f), reinterpret_cast<const uint8_t*>(w2t),
                                            R, gD, partial, err);
  L.bump();
  return ctas;
}

}  // namespace pasm
