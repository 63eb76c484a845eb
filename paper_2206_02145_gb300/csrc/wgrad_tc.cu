// Weight gradient of the network's 3x3 convolutions on the 5th-generation
// tensor cores: dW[tap][co][ci] = sum over the pixels p of x[p + shift(tap)][ci]
// dy[p][co], as products D[(tap, ci)][co] with K = 16 pixels.  Both operands
// lie in shared memory as the TMA writes them, one row of channels per pixel, so
// both are "MN-major": the pixel is K.
//
// A CTA owns CB input channels (64, 32 or 16) of all nine taps x BN output
// channels (64 or 32) and a run of patches of 4 image rows x 32 pixels.  Per
// patch the TMA brings dy (one box) and x with a halo row above and below three
// times, at the three column shifts kx, so that every tap's pixels start on
// a whole swizzle group: tap (ky, kx) is box kx from row ky on.  The rows of D
// are made of groups of CB channels, 128 / CB of them, whose pixels lie one
// fixed step apart: with CB = 64 the pairs (ky 0, 1) of each kx, the pair (kx 0,
// 1) of ky 2, and ky 2, kx 2; with fewer channels ky = 0, 1, 2 of one kx per
// product.  The step after the last tap reads whatever lies there, into rows of
// D that nobody reads.  Pixels outside the image are zeros (the TMA's fill); a
// patch's rows below the image are left out.
//   warp 0     TMA producer, a ring of S patches
//   warp 1     tensor memory; one lane issues the products (8 steps x NT per patch)
//   warps 2-5  where asked, sum dy over the pixels meanwhile (the bias gradient, by
//              the CTAs of the first input channels); then write D and the sums
//              to this run's row of the partials
// wgrad_sum_kernel adds the rows in a fixed order.
//
// Bound by shared memory: a product of 128 x BN reads 4 KB + BN x 32 bytes for
// BN / 4 cycles of tensor work; per 16 pixels 9.2 KB of x come in per 64
// channels.  In FP32 sums a run is at most 32 patches (256 products in a row).
// Minibatch of 8 x 256 x 512 pixels, per layer, against the warp-level
// mma.sync kernels (unet.cu): 16 -> 32 channels 173 -> 34 us, 32 -> 32 84 -> 40,
// 64 -> 32 165 -> 70, at half the width and height 128 -> 64 163 -> 40, at a
// quarter 256 -> 128 163 -> 38, at an eighth 256 -> 256 84 -> 24.
// Every wait is bounded, as in conv_tc.cu.
#include "tcgen05.cuh"
#include "tma_host.h"
#include "unet.cuh"

namespace lbk {
namespace nn {
namespace {

constexpr int kWgThreads = 192, kWgRows = 4, kWgCols = 32, kWgPix = kWgRows * kWgCols;
constexpr int kWgMaxRun = 32;  // patches per run at most

template <int CB, int BN>
struct WgShape {
  static constexpr int PA = CB * 2, PB = BN * 2;           // bytes per pixel row
  static constexpr int ROW = kWgCols * PA;                 // an image row of a box
  static constexpr int BOX = (kWgRows + 2) * ROW;          // the box of one kx
  static constexpr int X_BYTES = 3 * BOX, DY_BYTES = kWgPix * PB;
  static constexpr int STAGE = X_BYTES + DY_BYTES;
  static constexpr int CTAS = CB == 64 ? 1 : 2;            // per SM
  static constexpr int S = CB == 16 ? (BN == 32 ? 4 : 3) : 2;
  static constexpr int SMEM = S * STAGE + 1024;            // + alignment slack
  static constexpr int G = 128 / CB;                       // channel groups per product
  static constexpr int NT = CB == 64 ? 5 : 3;              // products per step
  static constexpr uint32_t COLS = NT * BN;
  static constexpr uint32_t TCOLS = COLS <= 128 ? 128 : (COLS <= 256 ? 256 : 512);
  static constexpr uint32_t mode(int n) { return n == 64 ? 2 : (n == 32 ? 4 : 6); }
  // kind::f16: D f32, A and B bf16, both MN-major, N, M = 128
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                    (uint32_t(BN >> 3) << 17) | (uint32_t(128 >> 4) << 24);
  static_assert(SMEM * CTAS <= 226 * 1024 && TCOLS * CTAS <= 512 && STAGE % 1024 == 0, "");
  // product t: byte offset of its first group and the step to the next
  static constexpr int start(int t) {
    return CB < 64 ? t * BOX : (t < 3 ? t * BOX : (t == 3 ? 2 * ROW : 2 * BOX + 2 * ROW));
  }
  static constexpr int step(int t) { return CB == 64 && t == 3 ? BOX : ROW; }
  // tap of group j of product t, or -1
  __host__ __device__ static constexpr int tap(int t, int j) {
    if (CB < 64) return j < 3 ? 3 * j + t : -1;
    if (t < 3) return 3 * j + t;
    return t == 3 ? 6 + j : (j == 0 ? 8 : -1);
  }
  // the last group of a step starts at most here: inside the stage
  static_assert(start(NT - 1) + (kWgRows - 1) * ROW + (G - 1) * step(NT - 1) + ROW <= STAGE, "");
};

// A K = 16 step of an MN-major operand: rows of one swizzle span per pixel, 8
// pixels per swizzle group (`group` bytes), the next span of channels `span`
// bytes on.
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t saddr, uint32_t span, uint32_t group,
                                                 uint32_t mode) {
  return umma_desc(saddr, group, mode) & ~(uint64_t(0x3FFF) << 16) |
         uint64_t((span >> 4) & 0x3FFFu) << 16;
}

struct WgTcArgs {
  int H, W, pw, ph;        // image; patches per image row / column
  int ci_off, co_off, Cin, Cout;
  int ncb, nchunks, run, patches;  // input channel blocks; runs, patches per run, patches
  int with_bias;
  float* part;             // [nchunks][9 Cout Cin + (with_bias ? Cout : 0)]
  unsigned* err;
};

template <int CB, int BN>
__global__ void __launch_bounds__(kWgThreads, WgShape<CB, BN>::CTAS)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mdy,
                    const WgTcArgs a) {
  using Sh = WgShape<CB, BN>;
  constexpr int S = Sh::S;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[S], empty[S], done;
  __shared__ uint32_t tmem_base;
  __shared__ float sbias[1024 / BN][BN + 1];
  uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int tile = blockIdx.x / a.nchunks, ck = blockIdx.x % a.nchunks;
  const int ci0 = (tile % a.ncb) * CB, co0 = (tile / a.ncb) * BN;
  const int pbeg = ck * a.run, pend = min(pbeg + a.run, a.patches);
  const bool bias = a.with_bias && ci0 == 0;
  const size_t row = size_t(9) * a.Cout * a.Cin + (a.with_bias ? a.Cout : 0);
  float* const part = a.part + size_t(ck) * row;
  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], bias ? 5 : 1);  // the products, and the four summing warps
    }
    mbar_init(&done, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, Sh::TCOLS);
  pdl_wait();  // the previous kernel's outputs are visible
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0 && lane == 0) {
    int it = 0;
    for (int p = pbeg; p < pend; ++p, ++it) {
      const int st = it % S;
      if (it >= S && !mbar_wait_bounded(&empty[st], uint32_t(it / S - 1) & 1u, kTcSpin)) {
        atomicOr(a.err, 2u);
        break;
      }
      const int img = p / (a.pw * a.ph), r = p % (a.pw * a.ph);
      const int h0 = (r / a.pw) * kWgRows, w0 = (r % a.pw) * kWgCols;
      uint8_t* sa = smem + st * Sh::STAGE;
      mbar_arrive_expect_tx(&full[st], Sh::STAGE);
#pragma unroll
      for (int kx = 0; kx < 3; ++kx)
        tma_load_4d(sa + kx * Sh::BOX, &mx, &full[st], a.ci_off + ci0, w0 + kx - 1, h0 - 1, img);
      tma_load_4d(sa + Sh::X_BYTES, &mdy, &full[st], a.co_off + co0, w0, h0, img);
    }
    // every issued copy has landed before the CTA may finish
    for (int j = it > S ? it - S : 0; j < it; ++j)
      if (!mbar_wait_bounded(&full[j % S], uint32_t(j / S) & 1u, kTcSpin)) atomicOr(a.err, 2u);
  } else if (warp == 1) {
    // the whole warp walks the patches, one lane issues
    const uint32_t s0 = smem_addr(smem);
    const uint64_t da = umma_desc_mn(s0, Sh::step(0), 8 * Sh::PA, Sh::mode(CB));
    const uint64_t db = umma_desc_mn(s0 + Sh::X_BYTES, 0, 8 * Sh::PB, Sh::mode(BN));
    const uint32_t a_hi = uint32_t(da >> 32), b_hi = uint32_t(db >> 32);
    const bool leader = elect_one();
    bool ok = true;
    for (int p = pbeg, it = 0; p < pend; ++p, ++it) {
      const int st = it % S;
      ok = mbar_wait_bounded(&full[st], uint32_t(it / S) & 1u, kTcSpin);
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      tc_fence_after();
      // image rows of the patch: those below the image are left out, so that
      // they don't multiply the halo's values by zero
      const int rows = a.H % kWgRows ? min(kWgRows, a.H - p % (a.pw * a.ph) / a.pw * kWgRows) : kWgRows;
      const uint32_t so = uint32_t(st * Sh::STAGE) >> 4;
      const uint32_t a_lo = uint32_t(da) + so, b_lo = uint32_t(db) + so;
      if (leader) {
#pragma unroll
        for (int k = 0; k < kWgPix / 16; ++k) {
          if (k / (kWgCols / 16) >= rows) break;
#pragma unroll
          for (int t = 0; t < Sh::NT; ++t)
            tc_mma(tmem + uint32_t(t * BN),
                   a_lo + uint32_t((k * 16 * Sh::PA + Sh::start(t)) >> 4) +
                       (uint32_t((Sh::step(t) - Sh::step(0)) >> 4) << 16),
                   a_hi, b_lo + uint32_t((k * 16 * Sh::PB) >> 4), b_hi, Sh::IDESC,
                   k != 0 || it != 0);
        }
        tc_commit(&empty[st]);
      }
      __syncwarp();
    }
    if (!ok && leader) atomicOr(a.err, 2u);
    if (leader) {
      tc_commit(&done);  // (also after a time-out: products in flight end before the CTA does)
      if (!mbar_wait_bounded(&done, 0u, kTcSpin)) atomicOr(a.err, 2u);
    }
    __syncwarp();
  } else if (warp >= 2) {
    const int q = warp & 3, tid = q * 32 + lane;
    bool ok = true;
    if (bias) {
      // thread: 16-byte piece c of the pixels r + 8 n, n of this thread's share;
      // the piece holds channels 8 (c ^ swizzle of the row)
      constexpr int PC = BN / 8, SH = 16 / PC;  // pieces per pixel; threads per (piece, r)
      const int c = tid % PC, r = (tid / PC) % 8, sh = tid / (PC * 8);
      const int ch = 8 * (c ^ (BN == 64 ? r : r >> 1));
      float sum[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) sum[j] = 0.f;
      for (int p = pbeg, it = 0; p < pend; ++p, ++it) {
        const int st = it % S;
        ok = mbar_wait_bounded(&full[st], uint32_t(it / S) & 1u, kTcSpin);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          if (lane == 0) atomicOr(a.err, 2u);
          break;
        }
        const uint8_t* sb = smem + st * Sh::STAGE + Sh::X_BYTES + c * 16;
#pragma unroll
        for (int n = sh; n < kWgPix / 8; n += SH) {
          const uint4 v = *reinterpret_cast<const uint4*>(sb + (n * 8 + r) * Sh::PB);
          const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            sum[2 * j] += __low2float(h[j]);
            sum[2 * j + 1] += __high2float(h[j]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
      }
      // the 8 SH sums of every channel, in a fixed order
#pragma unroll
      for (int j = 0; j < 8; ++j) sbias[r * SH + sh][ch + j] = sum[j];
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (ok && tid < BN) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8 * SH; ++k) t += sbias[k][tid];
        part[size_t(9) * a.Cout * a.Cin + co0 + tid] = t;
      }
    }
    ok = ok && __all_sync(0xffffffffu, mbar_wait_bounded(&done, 0u, kTcSpin));
    if (!ok && lane == 0) atomicOr(a.err, 2u);
    tc_fence_after();
    if (ok) {
      const int m = q * 32 + lane, j = m / CB, ci = ci0 + m % CB;
#pragma unroll 1
      for (int t = 0; t < Sh::NT; ++t) {
        const int tap = Sh::tap(t, j);
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          uint32_t r[32];
          tmem_ld32(tmem + (uint32_t(q * 32) << 16) + uint32_t(t * BN + c), r);
          if (tap >= 0) {
            float* o = part + (size_t(tap) * a.Cout + co0 + c) * a.Cin + ci;
#pragma unroll
            for (int i = 0; i < 32; ++i) o[size_t(i) * a.Cin] = __uint_as_float(r[i]);
          }
        }
      }
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

// dw[i] += the sum over the runs of part[c * row + i], i < n, and db[i - n] for
// n <= i < row.  A block of 256 threads takes 1024 / G entries, four to a thread;
// its G groups sum every Gth run each, four in flight, and the G sums are added
// in order.  G = 32 where 8 groups would leave most SMs without a block: 9,248
// entries of 304 runs 10.0 -> 6.3 us, 36,928 of 147 8.4 -> 6.8, but 73,792 of 76
// 7.3 -> 8.9.
template <int G>
__global__ void __launch_bounds__(256) wgrad_sum_kernel(const float* __restrict__ part, int row,
                                                        int n, int nchunks, float* dw, float* db) {
  constexpr int NL = 256 / G;
  __shared__ float4 red[G][NL];
  const int g = threadIdx.x / NL, l = threadIdx.x % NL;
  const int i = (blockIdx.x * NL + l) * 4;  // row and n are multiples of 4
  pdl_trigger();
  pdl_wait();
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (i < row) {
    const float* p = part + i;
#pragma unroll 4
    for (int c = g; c < nchunks; c += G) {
      const float4 v = *reinterpret_cast<const float4*>(p + size_t(c) * row);
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
  }
  red[g][l] = s;
  __syncthreads();
  if (g == 0 && i < row) {
    float4* o = reinterpret_cast<float4*>(i < n ? dw + i : db + (i - n));
    float4 t = *o;
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const float4 v = red[k][l];
      t.x += v.x;
      t.y += v.y;
      t.z += v.z;
      t.w += v.w;
    }
    *o = t;
  }
}

struct WgPlan {
  int cb, bn, ncb, tiles, patches, run, nchunks;
};
// Runs: as many CTAs as the SMs hold at once, or a multiple of that where a run
// would be longer than kWgMaxRun patches.
bool wg_plan(int Cout, int Cin, int N, int H, int W, WgPlan* p) {
  if (Cout % 32 || Cin % 16 || N < 1 || H < 1 || W < 1 || W % kWgCols) return false;
  p->cb = Cin % 64 == 0 ? 64 : (Cin % 32 == 0 ? 32 : 16);
  p->bn = Cout % 64 == 0 ? 64 : 32;
  p->ncb = Cin / p->cb;
  p->tiles = p->ncb * (Cout / p->bn);
  const long long patches = (long long)N * ((H + kWgRows - 1) / kWgRows) *
                            ((W + kWgCols - 1) / kWgCols);
  if (patches > (1 << 30)) return false;
  p->patches = int(patches);
  int slots = 152 * (p->cb == 64 ? 1 : 2) / p->tiles;
  if (slots < 1) slots = 1;
  const int waves = int((patches + (long long)slots * kWgMaxRun - 1) / ((long long)slots * kWgMaxRun));
  const long long want = (long long)slots * waves;
  p->run = int((patches + want - 1) / want);
  p->nchunks = (p->patches + p->run - 1) / p->run;
  return (long long)p->tiles * p->nchunks < (1ll << 31);
}
size_t wg_row(int Cout, int Cin, bool bias) {
  return size_t(9) * Cout * Cin + (bias ? Cout : 0);
}

template <int CB, int BN>
cudaError_t launch_wg(const CUtensorMap& mx, const CUtensorMap& mdy, const WgTcArgs& t, int grid,
                      cudaStream_t s) {
  using Sh = WgShape<CB, BN>;
  const cudaError_t e = cudaFuncSetAttribute(
      wgrad_tc_kernel<CB, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
  if (e != cudaSuccess) return e;
  return launch_pdl(wgrad_tc_kernel<CB, BN>, dim3(unsigned(grid)), dim3(kWgThreads), Sh::SMEM, s,
                    mx, mdy, t);
}

}  // namespace

size_t wgrad_tc_scratch(int Cout, int Cin, int N, int H, int W) {
  WgPlan p;
  return wg_plan(Cout, Cin, N, H, W, &p) ? size_t(p.nchunks) * wg_row(Cout, Cin, true) : 0;
}

cudaError_t wgrad_tc(const WgradArgs& a, bool* used, cudaStream_t s) {
  *used = false;
  const int N = int(a.npix / ((long long)a.H * a.W));
  WgPlan p;
  if (!a.err || !a.part || a.Cdy % 8 || a.Cx % 8 || a.co_off % 8 || a.ci_off % 8 ||
      !wg_plan(a.Cout, a.Cin, N, a.H, a.W, &p))
    return cudaSuccess;
  const size_t row = wg_row(a.Cout, a.Cin, a.db != nullptr);
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
  if (size_t(p.nchunks) * row > a.part_cap || row > size_t(1) << 30 || !al16(a.x) || !al16(a.dy) ||
      !al16(a.part) || !al16(a.dw) || !al16(a.db))
    return cudaSuccess;
  auto map = [&](CUtensorMap* m, const bf16* base, int C, int box_c, int rows) {
    const uint64_t dims[4] = {uint64_t(C), uint64_t(a.W), uint64_t(a.H), uint64_t(N)};
    const uint64_t str[3] = {uint64_t(C) * 2, uint64_t(a.W) * C * 2, uint64_t(a.H) * a.W * C * 2};
    const uint32_t box[4] = {uint32_t(box_c), uint32_t(kWgCols), uint32_t(rows), 1};
    return encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(base), dims, str,
                        box, swizzle_for(box_c));
  };
  CUtensorMap mx, mdy;
  if (!map(&mx, a.x, a.Cx, p.cb, kWgRows + 2) || !map(&mdy, a.dy, a.Cdy, p.bn, kWgRows))
    return cudaErrorInvalidValue;
  WgTcArgs t;
  t.H = a.H;
  t.W = a.W;
  t.pw = (a.W + kWgCols - 1) / kWgCols;
  t.ph = (a.H + kWgRows - 1) / kWgRows;
  t.ci_off = a.ci_off;
  t.co_off = a.co_off;
  t.Cin = a.Cin;
  t.Cout = a.Cout;
  t.ncb = p.ncb;
  t.nchunks = p.nchunks;
  t.run = p.run;
  t.patches = p.patches;
  t.with_bias = a.db != nullptr;
  t.part = a.part;
  t.err = a.err;
  const int grid = p.tiles * p.nchunks;
  cudaError_t e;
  switch (p.cb * 2 + (p.bn == 64)) {
    case 64 * 2 + 1: e = launch_wg<64, 64>(mx, mdy, t, grid, s); break;
    case 64 * 2: e = launch_wg<64, 32>(mx, mdy, t, grid, s); break;
    case 32 * 2 + 1: e = launch_wg<32, 64>(mx, mdy, t, grid, s); break;
    case 32 * 2: e = launch_wg<32, 32>(mx, mdy, t, grid, s); break;
    case 16 * 2 + 1: e = launch_wg<16, 64>(mx, mdy, t, grid, s); break;
    default: e = launch_wg<16, 32>(mx, mdy, t, grid, s); break;
  }
  if (e != cudaSuccess) return e;
  const int n = int(wg_row(a.Cout, a.Cin, false));
  *used = true;
  if (row < size_t(2 * 152) * 128)
    return launch_pdl(wgrad_sum_kernel<32>, dim3(unsigned((row + 31) / 32)), dim3(256), 0, s,
                      static_cast<const float*>(a.part), int(row), n, p.nchunks, a.dw, a.db);
  return launch_pdl(wgrad_sum_kernel<8>, dim3(unsigned((row + 127) / 128)), dim3(256), 0, s,
                    static_cast<const float*>(a.part), int(row), n, p.nchunks, a.dw, a.db);
}

}  // namespace nn
}  // namespace lbk
