// Tensor-core 3x3 convolution of the U-Net surrogate on the 5th-generation
// tensor cores: implicit GEMM D[pixel][co] = sum over the nine taps and the
// input channels of x[pixel + shift(tap)][ci] w[tap][co][ci], then bias,
// ReLU, an optional mask, bf16 out.  The same kernel computes the data
// gradient on flipped / transposed weights.
//
// Persistent CTAs (one per SM) walk a strided list of output tiles of G
// sub-tiles of 128 pixels (one or two image rows each) x BN output channels,
// channel tiles innermost so that CTAs running side by side share their input
// rows in L2.  The G sub-tiles share the weight box and accumulate into G
// independent accumulators whose products are interleaved: with a narrow N
// one accumulator's chain of dependent products would leave the tensor pipe
// mostly idle.  Roles:
//   warp 0     TMA producer: per K step (one tap, BK input channels) a 4D box
//              of the NHWC input at the tap's shifted origin (zero fill
//              outside the image gives the convolution's zero padding) and a
//              3D box of the weights, into a stage of an S-deep ring that
//              runs on across tiles
//   warp 1     allocates tensor memory (two accumulators of BN FP32 columns);
//              the warp walks the loop together and one elected lane issues
//              tcgen05.mma (kind::f16, bf16 x bf16 -> f32,
//              M = 128, N = BN, K = 16), frees each stage and hands each
//              finished accumulator to the epilogue through tcgen05.commit
//   warps 2-9  epilogue, two per 32-lane quarter of an accumulator: tcgen05.ld,
//              bias / ReLU / mask, bf16 stores; then release the accumulator,
//              so that the next tile's products overlap them
// conv3x3_tc_halo_kernel (below) is the variant taken wherever the image
// width is a multiple of 128 and N <= 128: one input box per channel chunk
// serves the nine taps.
// Every wait on a barrier is bounded; on a timeout the kernel sets bit 2 of
// *err, lets the copies and products already issued finish, frees its tensor
// memory and returns (the host turns the bit into an error status).
#include <cuda.h>

#include <cstdint>
#include <cstdlib>

#include "tcgen05.cuh"
#include "tma.cuh"
#include "tma_host.h"
#include "unet.cuh"

namespace lbk {
namespace nn {
namespace {

// epilogue warps: kEpi for every 32-lane quarter of the accumulators (1, 2 and 4
// on the network's minibatch: 2.89, 2.81 and 2.87 ms)
constexpr int kEpi = 2, kTcThreads = 64 + 128 * kEpi;

// The epilogue's way out.  An accumulator row is a pixel: written from there, a
// lane's 64 bytes are four 16-byte stores, each of a warp's on 16 to 32 lines (2000
// cycles of a tile's 3300 with 128 channels).  The rows pass through 2 KB of shared
// memory per warp instead (64-byte rows, pieces of 16 bytes exchanged by row as
// in a 64-byte swizzle: no bank conflicts on the way in, two at most on the way
// out), so that four lanes store one pixel.
constexpr int kOutBytes = 4 * kEpi * 2048;  // the epilogue warps' rows
__device__ __forceinline__ uint8_t* out_piece(uint8_t* rows, int px, int j) {
  return rows + px * 64 + ((j ^ (px >> 1)) & 3) * 16;
}
// 32 accumulator columns + bias (shared memory, 16-byte aligned), ReLU and rounding
// to bf16: the pairs of this lane's pixel
__device__ __forceinline__ void finish32(uint32_t taddr, const float* bias, int relu,
                                         uint32_t (&out)[16]) {
  uint32_t r[32];
  tmem_ld32(taddr, r);
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bias + j);
    float v[4] = {__uint_as_float(r[j]) + b.x, __uint_as_float(r[j + 1]) + b.y,
                  __uint_as_float(r[j + 2]) + b.z, __uint_as_float(r[j + 3]) + b.w};
    if (relu)
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = fmaxf(v[i], 0.f);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const __nv_bfloat162 o = __floats2bfloat162_rn(v[i], v[i + 1]);
      out[(j + i) / 2] = *reinterpret_cast<const uint32_t*>(&o);
    }
  }
}
__device__ __forceinline__ void out_put(uint8_t* rows, int lane, const uint32_t (&o)[16]) {
  __syncwarp();  // the rows before are read
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<uint4*>(out_piece(rows, lane, j)) =
        make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
  __syncwarp();
}
// Lane's pieces of the 32 pixels' mask (asked for before the accumulators are read),
// and the rows to y (pixel stride C elements), zero where the mask is <= 0.
__device__ __forceinline__ void mask_rows(uint4 (&mk)[4], int lane, int C, const bf16* mask) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (mask)
      mk[k] = *reinterpret_cast<const uint4*>(mask + (long long)(k * 8 + (lane >> 2)) * C +
                                              (lane & 3) * 8);
}
// up: where the first pixel's block of the 2 x 2 upsampled output goes (null: none;
// up_C channels, image rows up_row elements apart).
__device__ __forceinline__ void out_rows(uint8_t* rows, int lane, bf16* y, int C, bool masked,
                                         const uint4 (&mk)[4], bf16* up = nullptr, int up_C = 0,
                                         long long up_row = 0) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int px = k * 8 + (lane >> 2), j = lane & 3;
    uint4 v = *reinterpret_cast<const uint4*>(out_piece(rows, px, j));
    if (masked) {
      const __nv_bfloat162* mm = reinterpret_cast<const __nv_bfloat162*>(&mk[k]);
      uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (!(__low2float(mm[i]) > 0.f)) w[i] &= 0xffff0000u;
        if (!(__high2float(mm[i]) > 0.f)) w[i] &= 0x0000ffffu;
      }
    }
    *reinterpret_cast<uint4*>(y + (long long)px * C + j * 8) = v;
    if (up) {
      bf16* const d = up + (long long)(2 * px) * up_C + j * 8;
      *reinterpret_cast<uint4*>(d) = v;
      *reinterpret_cast<uint4*>(d + up_C) = v;
      *reinterpret_cast<uint4*>(d + up_row) = v;
      *reinterpret_cast<uint4*>(d + up_row + up_C) = v;
    }
  }
}

struct TcArgs {
  int H, W, BW;          // image size; tile width in pixels (128 or 64)
  int ci_off, nchunks;   // first input channel; K steps per tap
  int Cin;               // input channels
  int mtiles, ntiles_n;  // pixel tiles, channel tiles
  int Cy, co_off, relu;  // output channel stride / offset
  int Cout;              // output channels (bias entries)
  const float* bias;
  const bf16* mask;
  int mask_ch;  // masked channels, from the first
  bf16* y;
  bf16* up_y;    // 2 x 2 upsampled output, Cout channels, or null
  unsigned* err;
};

template <int BK, int BN, int G>
struct TcShape {
  static constexpr int A_BYTES = 128 * BK * 2;  // one 128-pixel sub-tile
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE = G * A_BYTES + B_BYTES;
  // one persistent CTA per SM: a ring as deep as ~190 KB of shared memory
  // allows (small stages need many copies in flight to cover their latency)
  static constexpr int S_FIT = 194560 / STAGE;
  static constexpr int S = S_FIT > 32 ? 32 : (S_FIT < 2 ? 2 : S_FIT);
  static constexpr int OUT_OFF = S * STAGE;
  static constexpr int SMEM = OUT_OFF + kOutBytes + 1024;  // + alignment slack
  static_assert(SMEM <= 224 * 1024, "stage ring exceeds shared memory");
  static constexpr uint32_t SBO = 8 * BK * 2;
  static constexpr uint32_t MODE = BK == 64 ? 2 : (BK == 32 ? 4 : 6);  // 128 / 64 / 32 B swizzle
  // kind::f16 instruction descriptor: D f32, A and B bf16, both K-major, N, M = 128
  static constexpr uint32_t IDESC =
      (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(BN >> 3) << 17) | (uint32_t(128 >> 4) << 24);
  static constexpr uint32_t ACC = G * BN;    // columns of one accumulator set
  static constexpr uint32_t TCOLS = 2 * ACC;  // double-buffered
  static_assert(TCOLS <= 512, "accumulators exceed tensor memory");
};

template <int BK, int BN, int G>
__global__ void __launch_bounds__(kTcThreads, 1)
    conv3x3_tc_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mw,
                      const TcArgs a) {
  using Sh = TcShape<BK, BN, G>;
  constexpr int S = Sh::S;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[S], empty[S], acc_full[2], acc_empty[2], fin;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) float sbias[256];
  uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  // (the warp's number as one value for the whole warp: its branches are uniform)
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int ksteps = 9 * a.nchunks;
  const int ntiles = (a.mtiles / G) * a.ntiles_n;  // a tile: G x 128 pixels x BN channels
  pdl_trigger();

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4 * kEpi);  // one arrival per epilogue warp
    }
    mbar_init(&fin, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, Sh::TCOLS);
  pdl_wait();  // the previous kernel's outputs (and any weight update) are visible
  for (int i = threadIdx.x; i < a.Cout; i += blockDim.x) sbias[i] = a.bias ? a.bias[i] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0 && lane == 0) {
    // producer: coordinates once per tile, counters instead of divisions
    int st = 0, it = 0;
    uint32_t ph = 0;  // phase of the current pass over the ring
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const long long pix0 = (long long)(t / a.ntiles_n) * (128 * G);
      const int n0 = (t % a.ntiles_n) * BN;
      int wg[G], hg[G], ig[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const long long pg = pix0 + g * 128;
        wg[g] = int(pg % a.W) - 1;
        hg[g] = int((pg / a.W) % a.H) - 1;
        ig[g] = int(pg / ((long long)a.W * a.H));
      }
      int c0 = 0, kx = 0, ky = 0;
      for (int ks = 0; ks < ksteps; ++ks, ++it) {
        if (it >= S && !mbar_wait_bounded(&empty[st], ph ^ 1u, kTcSpin)) {
          atomicOr(a.err, 2u);
          ok = false;
          break;
        }
        uint8_t* sa = smem + st * Sh::STAGE;
        mbar_arrive_expect_tx(&full[st], Sh::STAGE);
#pragma unroll
        for (int g = 0; g < G; ++g)
          tma_load_4d(sa + g * Sh::A_BYTES, &mx, &full[st], a.ci_off + c0, wg[g] + kx, hg[g] + ky,
                      ig[g]);
        tma_load_3d(sa + G * Sh::A_BYTES, &mw, &full[st], c0, n0, ky * 3 + kx);
        c0 += BK;
        if (c0 == a.Cin) {
          c0 = 0;
          if (++kx == 3) {
            kx = 0;
            ++ky;
          }
        }
        if (++st == S) {
          st = 0;
          ph ^= 1u;
        }
      }
    }
    // every issued copy has landed before the CTA may finish
    for (int j = it > S ? it - S : 0; j < it; ++j)
      if (!mbar_wait_bounded(&full[j % S], uint32_t(j / S) & 1u, kTcSpin)) atomicOr(a.err, 2u);
  } else if (warp == 1) {
    // MMA issuer: the whole warp walks the loop, one lane issues; operands as
    // offsets from a word computed once
    const uint64_t d0 = umma_desc(smem_addr(smem), Sh::SBO, Sh::MODE);
    const uint32_t lo0 = uint32_t(d0), hi = uint32_t(d0 >> 32);
    const bool leader = elect_one();
    int st = 0, tc = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tc) {
      const int buf = tc & 1;
      ok = tc < 2 || mbar_wait_bounded(&acc_empty[buf], uint32_t((tc >> 1) - 1) & 1u, kTcSpin);
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      tc_fence_after();
      const uint32_t d = tmem + uint32_t(buf * Sh::ACC);
      for (int ks = 0; ks < ksteps; ++ks) {
        ok = mbar_wait_bounded(&full[st], ph, kTcSpin);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        tc_fence_after();
        const uint32_t lo = lo0 + uint32_t((st * Sh::STAGE) >> 4);
        // the G sub-tiles accumulate independently: interleaving them keeps
        // several products in flight on the tensor pipe
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
            for (int g = 0; g < G; ++g)
              tc_mma(d + uint32_t(g * BN), lo + uint32_t((g * Sh::A_BYTES + kk * 32) >> 4), hi,
                        lo + uint32_t((G * Sh::A_BYTES + kk * 32) >> 4), hi, Sh::IDESC,
                        kk != 0 || ks != 0);
          tc_commit(&empty[st]);
        }
        __syncwarp();
        if (++st == S) {
          st = 0;
          ph ^= 1u;
        }
      }
      if (ok && leader) tc_commit(&acc_full[buf]);
    }
    if (!ok && leader) atomicOr(a.err, 2u);
    // all products issued by this CTA are complete before its tensor memory is freed
    if (leader) {
      tc_commit(&fin);
      if (!mbar_wait_bounded(&fin, 0u, kTcSpin)) atomicOr(a.err, 2u);
    }
    __syncwarp();
  } else if (warp >= 2) {
    const int q = warp & 3, we = (warp - 2) >> 2;  // tensor-memory lanes 32q .. 32q + 31
    uint8_t* const rows = smem + Sh::OUT_OFF + (warp - 2) * 2048;
    int tc = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++tc) {
      const int buf = tc & 1;
      bool ok = mbar_wait_bounded(&acc_full[buf], uint32_t(tc >> 1) & 1u, kTcSpin);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) atomicOr(a.err, 2u);
        break;
      }
      tc_fence_after();
      const long long pix0 = (long long)(t / a.ntiles_n) * (128 * G);
      const int n0 = (t % a.ntiles_n) * BN;
#pragma unroll 1
      for (int e = we; e < G * (BN / 32); e += kEpi) {
        const int g = e / (BN / 32), c = e % (BN / 32) * 32;
        // this warp's 32 pixels lie in one image row
        const long long pg = pix0 + g * 128;
        const int w0 = int(pg % a.W), h0 = int((pg / a.W) % a.H);
        const int img = int(pg / ((long long)a.W * a.H));
        const long long p = ((long long)img * a.H + h0 + q * 32 / a.BW) * a.W + w0 +
                            (q * 32 % a.BW);
        const long long o = p * a.Cy + a.co_off + n0 + c;
        uint32_t out[16];
        uint4 mk[4];
        const bool masked = a.mask && n0 + c < a.mask_ch;
        mask_rows(mk, lane, a.Cy, masked ? a.mask + o : nullptr);
        finish32(tmem + (uint32_t(q * 32) << 16) + uint32_t(buf * Sh::ACC + g * BN + c),
                 sbias + n0 + c, a.relu, out);
        out_put(rows, lane, out);
        bf16* const up =
            a.up_y ? a.up_y + (((long long)img * a.H + h0 + q * 32 / a.BW) * 4 * a.W +
                               2 * (w0 + q * 32 % a.BW)) * a.Cout + n0 + c
                   : nullptr;
        out_rows(rows, lane, a.y + o, a.Cy, masked, mk, up, a.Cout, 2ll * a.W * a.Cout);
      }
      // this warp's reads of the accumulator are done: hand it back
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, Sh::TCOLS);
  }
}

// ---- halo variant: one input box per channel chunk serves all nine taps
// Tiles of G image rows x 128 pixels (images of width a multiple of 128), BK
// input channels at a time.  A box of the rows h0 - 1 .. h0 + G and columns w0 -
// 1 .. w0 + 128 (zero fill outside the image) goes into a ring of SA; the weights
// of three taps (ky, kx = 0, 1, 2) into a ring of NB.  Sub-tile g's operand for
// tap (ky, kx) is the 128 rows starting kx rows into row g + ky of the box.
// Where a layer's weights fit the ring (3 nchunks <= NB, one channel tile) they
// stay there for all of a CTA's tiles.
// Bound by latency on small images (one or two tiles a CTA: the first box takes
// 2000 to 4600 cycles, then a product 35 to 55 each) and by the products' reads of
// shared memory on large ones.  Per layer of one 512 x 512 image, against a box
// per ky (three times G rows of input, and the weights again for every tile),
// one thread's divergent loop issuing the products and four epilogue warps
// storing from the accumulators' layout: 16 -> 32 channels 15.3 -> 12.9 us, 32 ->
// 32 with pooling 20.3 -> 17.0, with the head 24.3 -> 18.2, 64 -> 32 25.5 ->
// 20.9, 128 -> 64 (256 x 256) 18.3 -> 16.3, 64 -> 64 13.1 -> 11.9; a forward pass
// 277 -> 237.
template <int BK, int BN, int G>
struct HaloShape {
  static constexpr int ROWS = 130;                 // pixels per box row
  static constexpr int RB = BK * 2;                // bytes per pixel row (one swizzle span)
  static constexpr int al(int n) { return (n + 1023) / 1024 * 1024; }
  static constexpr int A_TX = (G + 2) * ROWS * RB, A_STAGE = al(A_TX);
  static constexpr int B_TAP = BN * RB;            // bytes of one tap's weights
  static constexpr int B_TX = 3 * B_TAP, B_SLOT = al(B_TX);
  // of 227 KB, less the epilogue's rows, bias, head and barriers
  static constexpr int ROOM = 232448 - 1024 - kOutBytes - (8 * BN * 4 + 2048 + 64);
  static constexpr int SA = 3 * A_STAGE + 6 * B_SLOT <= ROOM ? 3 : 2;
  static constexpr int NB_FIT = (ROOM - SA * A_STAGE) / B_SLOT;
  static constexpr int NB = NB_FIT > 12 ? 12 : NB_FIT;
  static_assert(NB >= 2, "no room for the weights");
  static constexpr int B_OFF = SA * A_STAGE;
  static constexpr int OUT_OFF = B_OFF + NB * B_SLOT;
  static constexpr int SMEM = OUT_OFF + kOutBytes + 1024;
  static constexpr uint32_t SBO = 8 * RB;
  static constexpr uint32_t MODE = BK == 64 ? 2 : (BK == 32 ? 4 : 6);  // 128 / 64 / 32 B swizzle
  static constexpr uint32_t IDESC =
      (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(BN >> 3) << 17) | (uint32_t(128 >> 4) << 24);
  static constexpr uint32_t ACC = G * BN;
  static constexpr uint32_t TCOLS = 2 * ACC < 32 ? 32 : 2 * ACC;
  static_assert(TCOLS <= 512, "accumulators exceed tensor memory");
};

struct HaloArgs {
  int H, W, rows_t, cols_t;  // image size; tiles per image column / row
  int ci_off, nchunks;       // first input channel; 64-channel chunks
  int ntiles, ntiles_n;      // tiles; channel tiles
  int Cy, co_off, relu, Cout;
  const float* bias;
  const bf16* mask;
  int mask_ch;  // masked channels, from the first
  bf16* y;
  bf16* up_y;    // 2 x 2 upsampled output, Cout channels, or null
  unsigned* err;
  // fused 1x1 head (null head_y: none): with one channel tile holding all
  // Cout channels of a pixel, head_y[p][o] = head_b[o] + sum_c head_w[o][c]
  // y[p][c] over the bf16 values stored, in channel order (the arithmetic of
  // the separate head kernel, so the result is the same)
  const float* head_w;
  const float* head_b;
  float* head_y;
  int head_out;
  // fused 2 x 2 average pooling of the output (null pool_y: none; G even and
  // no mask): pool_y [N][H/2][W/2][pool_Cy], channels pool_off + n0 + c
  bf16* pool_y;
  int pool_Cy, pool_off;
};

template <int BK, int BN, int G>
__global__ void __launch_bounds__(kTcThreads, 1)
    conv3x3_tc_halo_kernel(const __grid_constant__ CUtensorMap mx,
                           const __grid_constant__ CUtensorMap mw, const HaloArgs a) {
  using Sh = HaloShape<BK, BN, G>;
  constexpr int SA = Sh::SA, NB = Sh::NB;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t fullA[SA], emptyA[SA], fullB[NB], emptyB[NB];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], fin;
  __shared__ uint32_t tmem_base;
  __shared__ __align__(16) float sbias[256];
  __shared__ __align__(16) float shead[BN + 1][8];  // [c][o], then the head's bias
  uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  // (the warp's number as one value for the whole warp: its branches are uniform)
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int bsteps = 3 * a.nchunks;  // weight boxes of a tile
  const bool resident = bsteps <= NB && a.ntiles_n == 1;
  const bool head = a.head_y != nullptr;
  const bool pool = a.pool_y != nullptr;
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < SA; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&emptyA[s], 1);
    }
    for (int s = 0; s < NB; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyB[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4 * kEpi);
    }
    mbar_init(&fin, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, Sh::TCOLS);
  pdl_wait();  // the previous kernel's outputs (and any weight update) are visible
  for (int i = threadIdx.x; i < a.Cout; i += blockDim.x) sbias[i] = a.bias ? a.bias[i] : 0.f;
  if (head)
    for (int i = threadIdx.x; i < 8 * (BN + 1); i += blockDim.x) {
      const int c = i >> 3, o = i & 7;
      shead[c][o] = o >= a.head_out ? 0.f : (c < BN ? a.head_w[o * BN + c] : a.head_b[o]);
    }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  // tile t -> (image, first row, first column, first output channel)
  auto tile_at = [&](int t, int& img, int& h0, int& w0, int& n0) {
    const int gm = t / a.ntiles_n;
    n0 = (t % a.ntiles_n) * BN;
    const int per_img = a.rows_t * a.cols_t;
    img = gm / per_img;
    const int r = gm % per_img;
    h0 = (r / a.cols_t) * G;
    w0 = (r % a.cols_t) * 128;
  };

  if (warp == 0 && lane == 0) {
    int ia = 0, ib = 0;  // boxes issued
    bool ok = true;
    auto room = [&](uint64_t* empty, int i, int n) {  // slot of box i of a ring of n is free
      if (i >= n && !mbar_wait_bounded(&empty[i % n], uint32_t(i / n - 1) & 1u, kTcSpin)) {
        atomicOr(a.err, 2u);
        ok = false;
      }
      return ok;
    };
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x) {
      int img, h0, w0, n0;
      tile_at(t, img, h0, w0, n0);
      for (int c = 0; c < a.nchunks && ok; ++c) {
        if (!room(emptyA, ia, SA)) break;
        mbar_arrive_expect_tx(&fullA[ia % SA], Sh::A_TX);
        tma_load_4d(smem + ia % SA * Sh::A_STAGE, &mx, &fullA[ia % SA], a.ci_off + c * BK, w0 - 1,
                    h0 - 1, img);
        ++ia;
        if (resident && ib == bsteps) continue;
        for (int ky = 0; ky < 3; ++ky, ++ib) {
          if (!room(emptyB, ib, NB)) break;
          mbar_arrive_expect_tx(&fullB[ib % NB], Sh::B_TX);
          tma_load_4d(smem + Sh::B_OFF + ib % NB * Sh::B_SLOT, &mw, &fullB[ib % NB], c * BK, n0, 0,
                      ky);
        }
      }
    }
    // every issued copy has landed before the CTA may finish
    for (int j = ia > SA ? ia - SA : 0; j < ia; ++j)
      if (!mbar_wait_bounded(&fullA[j % SA], uint32_t(j / SA) & 1u, kTcSpin)) atomicOr(a.err, 2u);
    for (int j = ib > NB ? ib - NB : 0; j < ib; ++j)
      if (!mbar_wait_bounded(&fullB[j % NB], uint32_t(j / NB) & 1u, kTcSpin)) atomicOr(a.err, 2u);
  } else if (warp == 1) {
    const uint64_t d0 = umma_desc(smem_addr(smem), Sh::SBO, Sh::MODE);
    const uint32_t lo0 = uint32_t(d0), hi = uint32_t(d0 >> 32);
    const bool leader = elect_one();
    int sa = 0, sb = 0, tc = 0;
    uint32_t pa = 0, pb = 0;  // phases of the current passes over the rings
    bool ok = true;
    for (int t = blockIdx.x; t < a.ntiles && ok; t += gridDim.x, ++tc) {
      const int buf = tc & 1;
      ok = tc < 2 || mbar_wait_bounded(&acc_empty[buf], uint32_t((tc >> 1) - 1) & 1u, kTcSpin);
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      tc_fence_after();
      const uint32_t d = tmem + uint32_t(buf * Sh::ACC);
      if (resident) sb = 0;  // (and their first phase has passed from then on)
      for (int c = 0; c < a.nchunks && ok; ++c) {
        ok = mbar_wait_bounded(&fullA[sa], pa, kTcSpin);
        const uint32_t la = lo0 + uint32_t((sa * Sh::A_STAGE) >> 4);
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          ok = ok && mbar_wait_bounded(&fullB[sb], pb, kTcSpin);
          if (!(ok = __all_sync(0xffffffffu, ok))) break;
          tc_fence_after();
          // The swizzle follows the absolute shared-memory address (as the TMA
          // wrote it), so an operand may start at any row with the
          // base-offset field left at 0 (measured: setting it to the row's
          // phase, or starting at the aligned group with that phase, gives
          // wrong products).
          const uint32_t lb = lo0 + uint32_t((Sh::B_OFF + sb * Sh::B_SLOT) >> 4);
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
              for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                for (int g = 0; g < G; ++g)
                  tc_mma(d + uint32_t(g * BN),
                         la + uint32_t((((g + ky) * Sh::ROWS + kx) * Sh::RB + kk * 32) >> 4), hi,
                         lb + uint32_t((kx * Sh::B_TAP + kk * 32) >> 4), hi, Sh::IDESC,
                         kk != 0 || kx != 0 || ky != 0 || c != 0);
            if (!resident) tc_commit(&emptyB[sb]);
            if (ky == 2) tc_commit(&emptyA[sa]);
          }
          __syncwarp();
          if (++sb == NB && !resident) {
            sb = 0;
            pb ^= 1u;
          }
        }
        if (++sa == SA) {
          sa = 0;
          pa ^= 1u;
        }
      }
      if (ok && leader) tc_commit(&acc_full[buf]);
    }
    if (!ok && leader) atomicOr(a.err, 2u);
    if (leader) {
      tc_commit(&fin);
      if (!mbar_wait_bounded(&fin, 0u, kTcSpin)) atomicOr(a.err, 2u);
    }
    __syncwarp();
  } else if (warp >= 2) {
    const int q = warp & 3, we = (warp - 2) >> 2;
    uint8_t* const rows = smem + Sh::OUT_OFF + (warp - 2) * 2048;
    int tc = 0;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++tc) {
      int img, h0, w0, n0;
      tile_at(t, img, h0, w0, n0);
      const long long p0 = ((long long)img * a.H + h0) * a.W + w0 + q * 32;
      // the mask of an item (a row's 32 channels), one item ahead: its latency
      // passes during the wait and the item before (32 -> 64 channels, half of them
      // masked, at 8 x 256 x 512: 71 us, asked for in place 84, without a mask 54)
      uint4 mk[4];
      auto item_at = [&](int e) {
        return (p0 + (long long)(e / (BN / 32)) * a.W) * a.Cy + a.co_off + n0 + e % (BN / 32) * 32;
      };
      auto masked = [&](int e) { return a.mask && n0 + e % (BN / 32) * 32 < a.mask_ch; };
      if (we < G * (BN / 32)) mask_rows(mk, lane, a.Cy, masked(we) ? a.mask + item_at(we) : nullptr);
      const int buf = tc & 1;
      bool ok = mbar_wait_bounded(&acc_full[buf], uint32_t(tc >> 1) & 1u, kTcSpin);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) atomicOr(a.err, 2u);
        break;
      }
      tc_fence_after();
      const uint32_t ta = tmem + (uint32_t(q * 32) << 16) + uint32_t(buf * Sh::ACC);
      bool pooled = false;
      if constexpr (G % 2 == 0) {
        if (pool) {
          // rows in pairs: four lanes hold two neighbouring pixels of both and
          // write their 2 x 2 average too, in the order of the separate pooling
          // kernel ((x00 + x01) + x10 + x11) / 4 over the bf16 values
          pooled = true;
#pragma unroll 1
          for (int e = we; e < G / 2 * (BN / 32); e += kEpi) {
            const int g0 = e / (BN / 32) * 2, c = e % (BN / 32) * 32;
            const long long pp = ((long long)img * (a.H / 2) + (h0 + g0) / 2) * (a.W / 2) +
                                 (w0 + q * 32) / 2;
            bf16* yp = a.pool_y + pp * a.pool_Cy + a.pool_off + n0 + c;
            uint4 v[2][2][2];  // [row][half of the pixels][left, right]
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
              uint32_t out[16];
              finish32(ta + uint32_t((g0 + rr) * BN + c), sbias + n0 + c, a.relu, out);
              out_put(rows, lane, out);
              bf16* y = a.y + (p0 + (long long)(g0 + rr) * a.W) * a.Cy + a.co_off + n0 + c;
#pragma unroll
              for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                  const int px = 16 * k + 2 * (lane >> 2) + s, j = lane & 3;
                  v[rr][k][s] = *reinterpret_cast<const uint4*>(out_piece(rows, px, j));
                  *reinterpret_cast<uint4*>(y + (long long)px * a.Cy + j * 8) = v[rr][k][s];
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              uint32_t pk[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                auto at = [&](int rr, int s) {
                  return reinterpret_cast<const __nv_bfloat162*>(&v[rr][k][s])[i];
                };
                float lo = __low2float(at(0, 0)) + __low2float(at(0, 1));
                float hi = __high2float(at(0, 0)) + __high2float(at(0, 1));
                lo += __low2float(at(1, 0));
                hi += __high2float(at(1, 0));
                lo = 0.25f * (lo + __low2float(at(1, 1)));
                hi = 0.25f * (hi + __high2float(at(1, 1)));
                const __nv_bfloat162 pb = __floats2bfloat162_rn(lo, hi);
                pk[i] = *reinterpret_cast<const uint32_t*>(&pb);
              }
              *reinterpret_cast<uint4*>(yp + (long long)(8 * k + (lane >> 2)) * a.pool_Cy +
                                        (lane & 3) * 8) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
        }
      }
      if (head) {
        // a row's BN channels, over which the head's sums run in order
#pragma unroll 1
        for (int g = we; g < G; g += kEpi) {
          const long long p = p0 + (long long)g * a.W;
          float4 s0 = *reinterpret_cast<const float4*>(&shead[BN][0]);
          float4 s1 = *reinterpret_cast<const float4*>(&shead[BN][4]);
          const bool wide = a.head_out > 4;
#pragma unroll 1
          for (int c = 0; c < BN; c += 32) {
            uint32_t out[16];
            uint4 mk[4];  // (a convolution with the head has no mask)
            finish32(ta + uint32_t(g * BN + c), sbias + n0 + c, a.relu, out);
            out_put(rows, lane, out);
            out_rows(rows, lane, a.y + p * a.Cy + a.co_off + n0 + c, a.Cy, false, mk);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const __nv_bfloat162 hv = *reinterpret_cast<const __nv_bfloat162*>(&out[j / 2]);
              const float f = j % 2 ? __high2float(hv) : __low2float(hv);
              const float4 w = *reinterpret_cast<const float4*>(&shead[c + j][0]);
              s0.x = fmaf(f, w.x, s0.x);
              s0.y = fmaf(f, w.y, s0.y);
              s0.z = fmaf(f, w.z, s0.z);
              s0.w = fmaf(f, w.w, s0.w);
              if (wide) {
                const float4 u = *reinterpret_cast<const float4*>(&shead[c + j][4]);
                s1.x = fmaf(f, u.x, s1.x);
                s1.y = fmaf(f, u.y, s1.y);
                s1.z = fmaf(f, u.z, s1.z);
                s1.w = fmaf(f, u.w, s1.w);
              }
            }
          }
          const float r[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
          for (int o = 0; o < 8; ++o)
            if (o < a.head_out) a.head_y[(p + lane) * a.head_out + o] = r[o];
        }
      } else if (!pooled) {
#pragma unroll 1
        for (int e = we; e < G * (BN / 32); e += kEpi) {
          const int g = e / (BN / 32), c = e % (BN / 32) * 32, en = e + kEpi;
          uint4 cur[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) cur[i] = mk[i];
          if (en < G * (BN / 32))
            mask_rows(mk, lane, a.Cy, masked(en) ? a.mask + item_at(en) : nullptr);
          uint32_t out[16];
          finish32(ta + uint32_t(g * BN + c), sbias + n0 + c, a.relu, out);
          out_put(rows, lane, out);
          bf16* const up = a.up_y ? a.up_y + (((long long)img * a.H + h0 + g) * 4 * a.W +
                                              2 * (w0 + q * 32)) * a.Cout + n0 + c
                                  : nullptr;
          out_rows(rows, lane, a.y + item_at(e), a.Cy, masked(e), cur, up, a.Cout,
                   2ll * a.W * a.Cout);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, Sh::TCOLS);
  }
}

template <int BK, int BN, int G>
cudaError_t launch_halo(const CUtensorMap& mx, const CUtensorMap& mw, const HaloArgs& t,
                        cudaStream_t s) {
  using Sh = HaloShape<BK, BN, G>;
  static int sms = 0;
  if (!sms) {
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_halo_kernel<BK, BN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
  }
  const unsigned grid = unsigned(t.ntiles < sms ? t.ntiles : sms);
  return launch_pdl(conv3x3_tc_halo_kernel<BK, BN, G>, dim3(grid), dim3(kTcThreads), Sh::SMEM, s,
                    mx, mw, t);
}

template <int BK, int BN, int G>
cudaError_t launch_tc(const CUtensorMap& mx, const CUtensorMap& mw, const TcArgs& t,
                      cudaStream_t s) {
  using Sh = TcShape<BK, BN, G>;
  static int sms = 0;
  if (!sms) {
    cudaError_t e = cudaFuncSetAttribute(conv3x3_tc_kernel<BK, BN, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
  }
  // one CTA per SM: the ring fills the shared memory, the accumulators the TMEM
  const long long tiles = (long long)(t.mtiles / G) * t.ntiles_n;
  const unsigned grid = unsigned(tiles < sms ? tiles : sms);
  return launch_pdl(conv3x3_tc_kernel<BK, BN, G>, dim3(grid), dim3(kTcThreads), Sh::SMEM, s, mx,
                    mw, t);
}

// G sub-tiles per tile (independent accumulators); the widest shapes stay
// within 227 KB of shared memory and 512 TMEM columns
template <int BK, int BN>
cudaError_t launch_g(int g, const CUtensorMap& mx, const CUtensorMap& mw, const TcArgs& t,
                     cudaStream_t s) {
  if (BN == 32 && BK < 64 && g == 8) return launch_tc<BK, BN, (BN == 32 && BK < 64) ? 8 : 1>(mx, mw, t, s);
  if (BN <= 64 && g == 4) return launch_tc<BK, BN, (BN <= 64) ? 4 : 1>(mx, mw, t, s);
  if (BN <= 128 && g == 2) return launch_tc<BK, BN, (BN <= 128) ? 2 : 1>(mx, mw, t, s);
  if (g == 1) return launch_tc<BK, BN, 1>(mx, mw, t, s);
  return cudaErrorInvalidValue;
}

template <int BK>
cudaError_t launch_bn(int bn, int g, const CUtensorMap& mx, const CUtensorMap& mw,
                      const TcArgs& t, cudaStream_t s) {
  switch (bn) {
    case 32: return launch_g<BK, 32>(g, mx, mw, t, s);
    case 64: return launch_g<BK, 64>(g, mx, mw, t, s);
    case 128: return launch_g<BK, 128>(g, mx, mw, t, s);
    case 256: return launch_g<BK, 256>(g, mx, mw, t, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

bool conv3x3_tc_supported(const ConvArgs& a) {
  const long long npix = (long long)a.N * a.H * a.W;
  const bool rows = a.W % 128 == 0 || (a.W == 64 && a.H % 2 == 0);
  return rows && npix % 128 == 0 && a.Cin % 16 == 0 && a.Cout % 32 == 0 && a.Cout <= 256 &&
         a.Cx % 8 == 0 &&
         a.Cy % 8 == 0 && a.ci_off % 8 == 0 && a.co_off % 8 == 0 && a.ci_off + a.Cin <= a.Cx &&
         a.co_off + a.Cout <= a.Cy;
}

// the halo variant: images of width a multiple of 128, output tiles of at
// most 128 channels (its three-tap weight box bounds N)
template <int BK>
cudaError_t launch_halo_bk(int BN, int G, const CUtensorMap& mx, const CUtensorMap& mw,
                           const HaloArgs& t, cudaStream_t s) {
  switch (BN * 16 + G) {
    case 32 * 16 + 8: return launch_halo<BK, 32, (BK < 64 ? 8 : 2)>(mx, mw, t, s);
    case 32 * 16 + 4: return launch_halo<BK, 32, (BK < 64 ? 4 : 2)>(mx, mw, t, s);
    case 32 * 16 + 2: return launch_halo<BK, 32, 2>(mx, mw, t, s);
    case 32 * 16 + 1: return launch_halo<BK, 32, 1>(mx, mw, t, s);
    case 64 * 16 + 4: return launch_halo<BK, 64, (BK < 64 ? 4 : 2)>(mx, mw, t, s);
    case 64 * 16 + 2: return launch_halo<BK, 64, 2>(mx, mw, t, s);
    case 64 * 16 + 1: return launch_halo<BK, 64, 1>(mx, mw, t, s);
    case 128 * 16 + 2: return launch_halo<BK, 128, (BK < 64 ? 2 : 1)>(mx, mw, t, s);
    case 128 * 16 + 1: return launch_halo<BK, 128, 1>(mx, mw, t, s);
    default: return cudaErrorInvalidValue;
  }
}

static cudaError_t conv3x3_tc_halo(const ConvArgs& a, unsigned* err, cudaStream_t s, bool* used) {
  *used = false;
  if (const char* e = getenv("LBPF_CONV_HALO"))
    if (atoi(e) == 0) return cudaSuccess;
  if (a.W % 128 || a.Cin % 16) return cudaSuccess;
  // the widest channel chunk: splitting 64 channels into 32-wide chunks (to
  // fit 8 rows per tile instead of 4) measured slower
  const int BK = a.Cin % 64 == 0 ? 64 : (a.Cin % 32 == 0 ? 32 : 16);
  int BN = 128;
  while (BN > 32 && a.Cout % BN) BN >>= 1;
  if (a.Cout % BN) return cudaSuccess;
  // rows per tile: about 256 accumulator columns (within shared memory), as
  // many tiles as SMs where the image allows, G dividing the image height
  int G = 256 / BN;
  if (BK == 64) G = BN == 128 ? 1 : 2;
  const long long row_tiles = (long long)a.N * a.H * (a.W / 128);
  while (G > 1 && (a.H % G || (row_tiles / G) * (a.Cout / BN) < 152)) G >>= 1;
  if (a.H % G) return cudaSuccess;
  const CUtensorMapSwizzle sw = swizzle_for(BK);
  CUtensorMap mx, mw;
  {
    const uint64_t dims[4] = {uint64_t(a.Cx), uint64_t(a.W), uint64_t(a.H), uint64_t(a.N)};
    const uint64_t strides[3] = {uint64_t(a.Cx) * 2, uint64_t(a.W) * a.Cx * 2,
                                 uint64_t(a.H) * a.W * a.Cx * 2};
    const uint32_t box[4] = {uint32_t(BK), 130, uint32_t(G + 2), 1};
    if (!encode_tiled(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(a.x), dims,
                      strides, box, sw))
      return cudaErrorInvalidValue;
  }
  {
    // weights [ky][kx][Cout][Cin] viewed as (Cin, Cout, kx, ky)
    const uint64_t dims[4] = {uint64_t(a.Cin), uint64_t(a.Cout), 3, 3};
    const uint64_t strides[3] = {uint64_t(a.Cin) * 2, uint64_t(a.Cout) * a.Cin * 2,
                                 3ull * a.Cout * a.Cin * 2};
    const uint32_t box[4] = {uint32_t(BK), uint32_t(BN), 3, 1};
    if (!encode_tiled(&mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(a.w), dims,
                      strides, box, sw))
      return cudaErrorInvalidValue;
  }
  HaloArgs t;
  t.H = a.H;
  t.W = a.W;
  t.rows_t = a.H / G;
  t.cols_t = a.W / 128;
  t.ci_off = a.ci_off;
  t.nchunks = a.Cin / BK;
  t.ntiles_n = a.Cout / BN;
  t.ntiles = a.N * t.rows_t * t.cols_t * t.ntiles_n;
  t.Cy = a.Cy;
  t.co_off = a.co_off;
  t.relu = a.relu;
  t.Cout = a.Cout;
  t.bias = a.bias;
  t.mask = a.mask;
  t.mask_ch = a.mask_ch;
  t.y = a.y;
  t.err = err;
  // the head rides along when one tile holds every channel of a pixel
  const bool fuse = a.head_y && BN == a.Cout && a.co_off == 0 && a.head_out >= 1 &&
                    a.head_out <= 8 && !a.mask;
  t.head_w = fuse ? a.head_w : nullptr;
  t.head_b = fuse ? a.head_b : nullptr;
  t.head_y = fuse ? a.head_y : nullptr;
  t.head_out = fuse ? a.head_out : 0;
  if (a.head_done) *a.head_done = fuse ? 1 : 0;
  // the pooling of the next level rides along when a tile holds row pairs
  const bool fpool = a.pool_y && G % 2 == 0 && !a.mask && a.H % 2 == 0 && a.pool_Cy % 8 == 0 &&
                     a.pool_off % 8 == 0 && !fuse;
  t.pool_y = fpool ? a.pool_y : nullptr;
  t.pool_Cy = a.pool_Cy;
  t.pool_off = a.pool_off;
  if (a.pool_done) *a.pool_done = fpool ? 1 : 0;
  const bool fup = a.up_y && !fuse && !fpool;
  t.up_y = fup ? a.up_y : nullptr;
  if (a.up_done) *a.up_done = fup ? 1 : 0;
  *used = true;
  switch (BK) {
    case 64: return launch_halo_bk<64>(BN, G, mx, mw, t, s);
    case 32: return launch_halo_bk<32>(BN, G, mx, mw, t, s);
    default: return launch_halo_bk<16>(BN, G, mx, mw, t, s);
  }
}

cudaError_t conv3x3_tc(const ConvArgs& a, unsigned* err, cudaStream_t s) {
  if (!conv3x3_tc_supported(a) || !err) return cudaErrorInvalidValue;
  {
    bool used = false;
    const cudaError_t e = conv3x3_tc_halo(a, err, s, &used);
    if (used || e != cudaSuccess) return e;
  }
  const long long npix = (long long)a.N * a.H * a.W;
  const int BK = a.Cin % 64 == 0 ? 64 : (a.Cin % 32 == 0 ? 32 : 16);
  // the widest N that still gives half the SMs a tile: a product of 128 pixels
  // reads as much of the input whatever its N (8 x 32 x 64 pixels, 256 channels:
  // 20 us at N = 256, 24 at 64), but few tiles leave SMs idle (one image of 64 x
  // 64: 19 us at 256, 14 at 64)
  const long long mt = npix / 128;
  int BN = 256;
  while (BN > 32 && a.Cout % BN) BN >>= 1;
  while (BN > 64 && mt * (a.Cout / BN) < 76) BN >>= 1;
  if (const char* e = getenv("LBPF_CONV_MAX_BN")) {
    const int cap = atoi(e);
    while (BN > 32 && BN > cap) BN >>= 1;
  }
  const int BW = a.W % 128 == 0 ? 128 : 64;
  // sub-tiles per tile: about 256 accumulator columns per K step, as many
  // tiles as SMs where the image allows, G dividing the pixel tiles
  int G = 256 / BN;
  const int gmax = BN == 32 ? (BK < 64 ? 8 : 4) : (BN == 64 ? 4 : (BN == 128 ? 2 : 1));
  if (G > gmax) G = gmax;
  while (G > 1 && (mt % G || (mt / G) * (a.Cout / BN) < 152)) G >>= 1;
  if (const char* e = getenv("LBPF_CONV_G")) {
    const int want = atoi(e);
    while (G > 1 && G > want) G >>= 1;
  }
  CUtensorMap mx, mw;
  {
    const uint64_t dims[4] = {uint64_t(a.Cx), uint64_t(a.W), uint64_t(a.H), uint64_t(a.N)};
    const uint64_t strides[3] = {uint64_t(a.Cx) * 2, uint64_t(a.W) * a.Cx * 2,
                                 uint64_t(a.H) * a.W * a.Cx * 2};
    const uint32_t box[4] = {uint32_t(BK), uint32_t(BW), uint32_t(128 / BW), 1};
    if (!encode_tiled(&mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(a.x), dims,
                      strides, box, swizzle_for(BK)))
      return cudaErrorInvalidValue;
  }
  {
    const uint64_t dims[3] = {uint64_t(a.Cin), uint64_t(a.Cout), 9};
    const uint64_t strides[2] = {uint64_t(a.Cin) * 2, uint64_t(a.Cout) * a.Cin * 2};
    const uint32_t box[3] = {uint32_t(BK), uint32_t(BN), 1};
    if (!encode_tiled(&mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(a.w), dims,
                      strides, box, swizzle_for(BK)))
      return cudaErrorInvalidValue;
  }
  TcArgs t;
  t.H = a.H;
  t.W = a.W;
  t.BW = BW;
  t.ci_off = a.ci_off;
  t.nchunks = a.Cin / BK;
  t.Cy = a.Cy;
  t.co_off = a.co_off;
  t.relu = a.relu;
  t.bias = a.bias;
  t.mask = a.mask;
  t.mask_ch = a.mask_ch;
  t.y = a.y;
  t.up_y = a.up_y;
  if (a.up_done) *a.up_done = a.up_y ? 1 : 0;
  t.err = err;
  t.mtiles = int(npix / 128);
  t.ntiles_n = a.Cout / BN;
  t.Cout = a.Cout;
  t.Cin = a.Cin;
  switch (BK) {
    case 64: return launch_bn<64>(BN, G, mx, mw, t, s);
    case 32: return launch_bn<32>(BN, G, mx, mw, t, s);
    default: return launch_bn<16>(BN, G, mx, mw, t, s);
  }
}

}  // namespace nn
}  // namespace lbk
