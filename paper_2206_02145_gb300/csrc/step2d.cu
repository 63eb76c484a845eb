// Fused coupled LB step in 2D: D2Q9 flow f (Eqs. 4-12), D2Q9 solute g
// (Eqs. 13-18) and D2Q9 phase field h (Eqs. 19-23).
//
// Streaming is done in push form: the thread of node s holds its own
// populations, forms every moment locally, collides and writes the
// post-collision value of direction a to s + c_a.  That is the same update
// as the pull form of the paper's equations; it needs no stored macroscopic
// fields, only phi(t-1) for d(phi)/dt.  Per node and step the HBM traffic is
// 27 populations read + 27 written + phi(t-1) read + phi(t) written (224 B in
// FP32 with flow, 152 B without, 116 B with 16-bit populations).
//
// Populations are deviations d_a = p_a - w_a M_ref (M_ref = 1 for f, U_ref
// for g, -1 for h); the phi ring holds phi + 1.
//
// Two parts of the step need neighbour data, both served from shared memory:
// grad(phi) (Eq. 3, 21, 23) needs phi(t) of a one-node halo, summed from the
// halo's h populations, and Eq. 19 writes
// a_s^2 h(r + c, t+1) = h*(r) - (1 - a_s^2(r)) h(r + c, t), i.e. needs the old
// h of the destination node.
//
// step2d_tma_kernel (FP32 and 16-bit storage): persistent CTAs of 128 threads
// stream tiles through a 2-stage shared-memory pipeline.  Per tile one thread
// issues three TMA tensor loads on one mbarrier: f and g of the tile, h of the
// tile plus halo (box starting 16 bytes left of the tile so that its innermost
// coordinate stays aligned), and the phi ring of the tile.  While a tile is
// computed and pushed, the next one is in flight.  Halo positions outside
// the domain (the TMA fills them with zeros) are patched on edge tiles only.
//
// What bounds it, and what was taken for that (coupled steps, GB300, 6.69 TB/s
// copy rate):
//  - FP32 beyond the L2: how the memory is asked.  Tiles are 64 columns wide
//    (256-byte rows), and at most kStageBytes of stages are resident per SM:
//    with every CTA that fits, the h halos are read twice (666 MB from DRAM per
//    2480 x 2080 step against 587) and the step takes 224 us instead of 177.
//    1024^2: 48.4 -> 40.1 us (0.87 of the copy rate); 2480 x 2080: 250 -> 177
//    (0.98).
//  - 16-bit storage: instructions, and the waits between them.  A thread of a large
//    grid holds two nodes, 2 rows apart, on the packed two-lane FP32 instructions
//    (lbpf_device.cuh): 590 warp instructions per 32 nodes instead of 906, 2.3 issued
//    per cycle and SM instead of 2.8.  1024^2: 38.2 -> 29.1 us; 2480 x 2080: 119.
//  - small grids: the chain of a tile.  Tiles of 32 x 4 with one node per
//    thread give the most CTAs; boundary tiles run the same arithmetic as inner
//    ones with precomputed steps.  128^2 without flow: 3.6 -> 3.2 us.
// The shapes are chosen in shape_of().
//
// step2d_kernel (FP64 storage): one thread per node, one tile per CTA, the
// same per-node code.
#include <algorithm>
#include <numeric>

#include "step2d_tile.cuh"
#include "tma_host.h"

namespace lbk {
namespace {

constexpr int kSpin = 1 << 22;  // bound on mbarrier polls before giving up

// ---- FP64 (and reference) kernel: one tile per CTA ------------------------------
template <typename T, typename R, bool FLOW, int TX, int TY, bool CHM>
__global__ void __launch_bounds__(TX* TY)
    step2d_kernel(const Model m, const PopPtrs sp, const PopPtrs dp,
                  const R* __restrict__ ring_prev, R* __restrict__ ring_cur,
                  unsigned* __restrict__ err) {
  constexpr int SX = TX + 2, SY = TY + 2;
  constexpr int QF = FLOW ? 9 : 0;
  constexpr int NT = TX * TY;
  __shared__ R sh_phi[SY][SX];
  __shared__ R sh_h[9][SY][SX];

  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * TX + tx;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int x = x0 + tx, y = y0 + ty;
  const int nx = m.nx, ny = m.ny, px = m.px;
  const bool active = x < nx && y < ny;
  const int idx = y * px + x;

  R f[9], g[9], h[9];
  R dphi_prev = R(0);
  if (active) {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      if (FLOW) f[a] = Pop<T>::template ld<R>(static_cast<const T*>(sp.p[a]) + idx);
      g[a] = Pop<T>::template ld<R>(static_cast<const T*>(sp.p[QF + a]) + idx);
      h[a] = Pop<T>::template ld<R>(static_cast<const T*>(sp.p[QF + 9 + a]) + idx);
    }
    dphi_prev = ring_prev[idx];
  }
  if (active) {
    R s = R(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      s += h[a];
      sh_h[a][ty + 1][tx + 1] = h[a];
    }
    sh_phi[ty + 1][tx + 1] = s;
  }
  // halo ring (and positions of a partial tile): phi and h of the mapped node
  for (int i = tid; i < SX * SY; i += NT) {
    const int lx = i % SX, ly = i / SX;
    int gx = x0 + lx - 1, gy = y0 + ly - 1;
    if (lx >= 1 && lx <= TX && ly >= 1 && ly <= TY && gx < nx && gy < ny) continue;
    gx = grad_coord(gx, nx, m.bc[0]);
    gy = grad_coord(gy, ny, m.bc[1]);
    const int j = gy * px + gx;
    R s = R(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const R v = Pop<T>::template ld<R>(static_cast<const T*>(sp.p[QF + 9 + a]) + j);
      sh_h[a][ly][lx] = v;
      s += v;
    }
    sh_phi[ly][lx] = s;
  }
  __syncthreads();
  const bool solids = m.solid && m.solid_tiles[blockIdx.y * gridDim.x + blockIdx.x];
  if (!active) return;
  const Grid2D gr(m);
  unsigned sm[1] = {0};  // solid neighbours
  if (solids)
    for (int a = 0; a < 9; ++a)
      sm[0] |= solid_mapped(m, x + D2_CX[a], y + D2_CY[a]) ? 1u << a : 0u;
  R Unew;
  const unsigned o = unsigned(ty * px + tx) * unsigned(sizeof(T));
  auto work = [&](auto edge) {
    collide_push_2d<T, R, FLOW, CHM, true, decltype(edge)::value, false, SX, 0>(
        gr, coef<R>(m), x, y, [&](int q) { return q < QF ? f[q] : g[q - QF]; }, h, sh_phi[ty + 1][tx + 1],
        dphi_prev, &sh_phi[ty + 1][tx + 1],
        [&](int a, int dy, int dx) { return sh_h[a][ty + 1 + dy][tx + 1 + dx]; },
        [](int, int) { return R(0); }, sm, R(coef<R>(m).ref_g),
        static_cast<T*>(dp.p[0]) + (size_t(y0) * px + x0), o, o, err, Unew);
  };
  if (solids || x0 < 1 || x0 + TX > nx - 1 || y0 < 1 || y0 + TY > ny - 1) work(std::true_type{});
  else work(std::false_type{});
  ring_cur[idx] = sh_phi[ty + 1][tx + 1];
}

// ---- TMA-pipelined persistent kernel ------------------------------------------

// MASK: the variant with the solid-node path; CHM: the central Hermite MRT
// flow collision; PAIR: two nodes per thread (step2d_tile.cuh).
template <typename T, bool FLOW, int TX, int TY, bool PAIR, int S, bool MASK, bool CHM>
__global__ void __launch_bounds__(tile_threads<TX, TY, PAIR>(), 512 / tile_threads<TX, TY, PAIR>())
    step2d_tma_kernel(const __grid_constant__ CUtensorMap tm_fg,
                      const __grid_constant__ CUtensorMap tm_h,
                      const __grid_constant__ CUtensorMap tm_ring,
                      const __grid_constant__ CUtensorMap tm_uown,
                      const __grid_constant__ CUtensorMap tm_uhal, const Model m,
                      const T* __restrict__ src, T* __restrict__ dst,
                      float* __restrict__ ring_cur, unsigned* __restrict__ err, int ntx,
                      int ntiles, int c) {
  using R = float;
  using L = Tiles2D<T, FLOW, TX, TY>;
  constexpr int SX = TX + 2, SY = TY + 2;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[S];
  __shared__ R sh_phi[SY][SX];
  __shared__ unsigned char sh_solid[MASK ? SX * SY : 1];
  const Grid2D gr(m);
  const int tid = threadIdx.x;
  const int first = blockIdx.x, G = gridDim.x;

  // The CTA's tiles are first, first + G, first + 2G, ... in row-major order.
  // Columns and rows advance by (G mod ntx, G div ntx) with one carry, in
  // uniform registers (every thread of the CTA has the same), so that the
  // tile's origin is a uniform base of all its addresses.
  struct Cursor {
    int tile, col, row;
  };
  const int gcol = G % ntx, grow = G / ntx;
  auto advance = [&](Cursor& q) {
    q.tile += G;
    q.col += gcol;
    q.row += grow;
    if (q.col >= ntx) {
      q.col -= ntx;
      ++q.row;
    }
  };
  auto issue = [&](const Cursor& q, int s) {
    issue_tile_2d<T, FLOW, TX, TY>(&tm_fg, &tm_h, &tm_ring, &tm_uown, &tm_uhal, c, &full[s],
                                   smem + s * L::STAGE, q.col * TX, q.row * TY);
  };
  Cursor work{first, first % ntx, first / ntx};
  Cursor load = work;  // the next tile to load, S tiles ahead of the work

  if (tid == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&full[s], 1);
    fence_barrier_init();
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < S; ++k) {
    if (tid == 0 && load.tile < ntiles) issue(load, k);
    advance(load);
  }

  // the solid flag of a tile, read one tile ahead
  auto flag = [&](const Cursor& q) -> unsigned char {
    return MASK && q.tile < ntiles ? m.solid_tiles[q.row * ntx + q.col] : 0;
  };
  unsigned char solids = flag(work);

  for (int k = 0; work.tile < ntiles; ++k) {
    const int s = k % S;
    Cursor next = work;
    advance(next);
    const unsigned char next_solids = flag(next);
    const bool ok = mbar_wait_bounded(&full[s], uint32_t((k / S) & 1), kSpin);
    if (!tile_2d<T, FLOW, TX, TY, PAIR, MASK, CHM>(gr, m, src, dst, ring_cur, err, work.col * TX,
                                                   work.row * TY, c, smem + s * L::STAGE,
                                                   &sh_phi[0][0], sh_solid, solids != 0, !ok)) {
      // a tile never arrived: report, let the copies in flight land, stop
      if (tid == 0) {
        atomicOr(err, 2u);
        for (int j = 1; j < S; ++j) {
          const int kk = k + j;
          if (first + kk * G < ntiles)
            mbar_wait_bounded(&full[kk % S], uint32_t((kk / S) & 1), kSpin);
        }
      }
      __syncthreads();
      return;
    }
    __syncthreads();  // stage s and sh_phi are free again
    if (tid == 0 && load.tile < ntiles) {
      fence_proxy_async_smem();
      issue(load, s);
    }
    advance(load);
    work = next;
    solids = next_solids;
  }
}

// ---- host side: tensor maps and launches -------------------------------------------
constexpr int kStages = 2;

// Tile shapes of the step: columns, rows, two nodes per thread or one.
enum { SH_SMALL = 0, SH_WIDE = 1, SH_PAIR = 2 };
constexpr int kShapeX[3] = {32, 64, 64}, kShapeY[3] = {4, 2, 4};
constexpr int kPairTiles = 1500;  // fewest 64 x 4 tiles (about ten a SM) for SH_PAIR

// FP32 states beyond the L2 take the wide tiles, 16-bit states of at least
// kPairTiles tiles two nodes per thread, everything else (and the FP64 kernel)
// the small tiles.  Measured, us per coupled step (small / wide / pair):
//   FP32  775 x 650 19.0 / 19.3 / 18.8, 1024^2 40.7 / 40.1 / 40.3,
//         1555 x 2023 119 / 113 / 118, 2480 x 2080 188 / 177 / 200
//   FP16  512^2 11.1 / - / 12.9, 640^2 14.3 / - / 14.9, 775 x 650 17.7 / 18.9 /
//         15.7, 1024^2 30.8 / 32.2 / 29.1, 2480 x 2080 135 / 141 / 119
// (FP32 with a baffle of solid nodes, 775 x 650: 19.6 / 20.0 / 22.7).
int shape_of(const Model& m) {
  if (m.storage == ST_FP64) return SH_SMALL;
  if (m.storage == ST_FP32) {
    const double state = 2.0 * double(m.plane) * double((m.qf + 2 * m.qs) * 4 + 4);
    return state > kL2Bytes ? SH_WIDE : SH_SMALL;
  }
  const long long tiles = (long long)((m.nx + kShapeX[SH_PAIR] - 1) / kShapeX[SH_PAIR]) *
                          ((m.ny + kShapeY[SH_PAIR] - 1) / kShapeY[SH_PAIR]);
  return tiles >= kPairTiles ? SH_PAIR : SH_SMALL;
}


// A warp per tile of the TMA kernel: does the tile or its one-node halo (mapped
// like the gradient stencil) hold a solid node?  (A thread per tile is a chain of
// 204 loads: 120 us of lbpf_set_solid's 400 at 775 x 650.)
__global__ void solid_tiles_kernel(const Model m, unsigned char* flags, int ntx, int nty, int tx,
                                   int ty) {
  const int t = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (t >= ntx * nty) return;
  const int x0 = (t % ntx) * tx, y0 = (t / ntx) * ty;
  const int xe = x0 + tx < m.nx ? x0 + tx : m.nx, ye = y0 + ty < m.ny ? y0 + ty : m.ny;
  bool any = false;
#pragma unroll 2
  for (int y = y0 - 1; y <= ye; ++y)
    for (int x = x0 - 1 + lane; x <= xe; x += 32) any |= solid_mapped(m, x, y);
  any = __any_sync(0xffffffffu, any);
  if (lane == 0) flags[t] = any ? 1 : 0;
}

template <typename T, bool FLOW, int kTX, int kTY, bool PAIR>
cudaError_t prepare_t(const Model& m, void* const pops[2], void* const rings[2], StepMaps* out) {
  using L = Tiles2D<T, FLOW, kTX, kTY>;
  const CUtensorMapDataType dt = pop_tensor_type(m.storage);
  const uint64_t q = uint64_t(L::QFG + 9);
  for (int b = 0; b < 2; ++b) {
    const uint64_t dims3[3] = {uint64_t(m.nx), uint64_t(m.ny), q};
    const uint64_t str3[2] = {uint64_t(m.px) * sizeof(T), uint64_t(m.plane) * sizeof(T)};
    const uint32_t box_fg[3] = {kTX, kTY, uint32_t(L::QFG)};
    const uint32_t box_h[3] = {uint32_t(L::BXH), kTY + 2, 9};
    const uint64_t dims2[2] = {uint64_t(m.nx), uint64_t(m.ny)};
    const uint64_t str2[1] = {uint64_t(m.px) * 4};
    const uint32_t box_r[2] = {kTX, kTY};
    if (!encode_tiled(&out->fg[b], dt, 3, pops[b], dims3, str3, box_fg) ||
        !encode_tiled(&out->h[b], dt, 3, pops[b], dims3, str3, box_h) ||
        !encode_tiled(&out->ring[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, rings[b], dims2, str2, box_r))
      return cudaErrorInvalidValue;
  }
  if (L::REL) {
    // the two U planes as one 3D tensor; the plane is the third coordinate
    if (!m.uring) return cudaErrorInvalidValue;
    const uint64_t dimsu[3] = {uint64_t(m.nx), uint64_t(m.ny), 2};
    const uint64_t stru[2] = {uint64_t(m.px) * 2, uint64_t(m.plane) * 2};
    const uint32_t box_uo[3] = {kTX, kTY, 1};
    const uint32_t box_uh[3] = {uint32_t(L::BXU), kTY + 2, 1};
    if (!encode_tiled(&out->uown, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, m.uring, dimsu, stru, box_uo) ||
        !encode_tiled(&out->uhal, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, m.uring, dimsu, stru, box_uh))
      return cudaErrorInvalidValue;
  } else {
    out->uown = out->ring[0];  // unused
    out->uhal = out->ring[0];
  }
  const int smem = kStages * L::STAGE;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  auto setup = [&](auto kern, int* ctas) {
    int per_sm = 0;
    cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (r == cudaSuccess)
      r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                        tile_threads<kTX, kTY, PAIR>(), smem);
    *ctas = sms * (per_sm > 0 ? per_sm : 1);
    return r;
  };
  if ((e = setup(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, false, false>,
                 &out->ctas_v[0])) != cudaSuccess ||
      (e = setup(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, true, false>,
                 &out->ctas_v[1])) != cudaSuccess)
    return e;
  if constexpr (FLOW) {  // the central Hermite MRT exists with flow only
    if ((e = setup(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, false, true>,
                   &out->ctas_v[2])) != cudaSuccess ||
        (e = setup(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, true, true>,
                   &out->ctas_v[3])) != cudaSuccess)
      return e;
  }
  // populations and ring of both buffers beyond the L2: bound the copies in flight
  const double state = 2.0 * double(m.plane) * double(q * sizeof(T) + 4 + (L::REL ? 2 : 0));
  if (state > kL2Bytes) {
    const int most = std::max(1, kStageBytes / smem);
    for (int v = 0; v < 4; ++v) out->ctas_v[v] = std::min(out->ctas_v[v], sms * most);
  }
  out->ctas = out->ctas_v[0];
  out->smem = smem;
  out->ready = 1;
  return cudaSuccess;
}

template <typename T, bool FLOW, int kTX, int kTY, bool PAIR>
cudaError_t launch_tma_t(const Model& m, const StepMaps& maps, int c, const void* src, void* dst,
                         void* ring_cur, unsigned* err, cudaStream_t s) {
  const int ntx = (m.nx + kTX - 1) / kTX, nty = (m.ny + kTY - 1) / kTY;
  const int ntiles = ntx * nty;
  const int v = (m.solid ? 1 : 0) + (FLOW && m.chm ? 2 : 0);
  // a number of CTAs coprime to the tiles per row: every CTA then meets the
  // (slower) edge columns equally often
  int grid = ntiles < maps.ctas_v[v] ? ntiles : maps.ctas_v[v];
  while (grid < ntiles && grid > 1 && std::gcd(grid, ntx) > 1) --grid;
  auto go = [&](auto kern) {
    kern<<<grid, tile_threads<kTX, kTY, PAIR>(), maps.smem, s>>>(
        maps.fg[c], maps.h[c], maps.ring[c], maps.uown, maps.uhal, m, static_cast<const T*>(src),
        static_cast<T*>(dst), static_cast<float*>(ring_cur), err, ntx, ntiles, c);
  };
  if (v == 0) go(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, false, false>);
  else if (v == 1) go(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, true, false>);
  if constexpr (FLOW) {
    if (v == 2) go(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, false, true>);
    else if (v == 3) go(step2d_tma_kernel<T, FLOW, kTX, kTY, PAIR, kStages, true, true>);
  }
  return cudaGetLastError();
}

template <typename T, typename R, bool FLOW>
cudaError_t launch_plain_t(const Model& m, const void* src, void* dst, const void* ring_prev,
                           void* ring_cur, unsigned* err, cudaStream_t s) {
  constexpr int kTX = kShapeX[SH_SMALL], kTY = kShapeY[SH_SMALL];
  dim3 block(kTX, kTY);
  dim3 grid((m.nx + kTX - 1) / kTX, (m.ny + kTY - 1) / kTY);
  const PopPtrs sp = pop_ptrs(m, const_cast<void*>(src), sizeof(T));
  const PopPtrs dp = pop_ptrs(m, dst, sizeof(T));
  if (FLOW && m.chm)
    step2d_kernel<T, R, FLOW, kTX, kTY, FLOW><<<grid, block, 0, s>>>(
        m, sp, dp, static_cast<const R*>(ring_prev), static_cast<R*>(ring_cur), err);
  else
    step2d_kernel<T, R, FLOW, kTX, kTY, false><<<grid, block, 0, s>>>(
        m, sp, dp, static_cast<const R*>(ring_prev), static_cast<R*>(ring_cur), err);
  return cudaGetLastError();
}

// fn(shape X, shape Y, pair) for the tile shape of m, of those compiled for T
template <typename T, typename F>
cudaError_t with_shape(const Model& m, F fn) {
  using std::integral_constant;
  const int sh = shape_of(m);
  auto go = [&](auto i) {
    constexpr int I = decltype(i)::value;
    return fn(integral_constant<int, kShapeX[I]>{}, integral_constant<int, kShapeY[I]>{},
              integral_constant<bool, I == SH_PAIR>{});
  };
  if constexpr (sizeof(T) == 4) {
    if (sh == SH_WIDE) return go(integral_constant<int, SH_WIDE>{});
  } else {
    if (sh == SH_PAIR) return go(integral_constant<int, SH_PAIR>{});
  }
  return go(integral_constant<int, SH_SMALL>{});
}

template <typename T>
cudaError_t prepare_any(const Model& m, void* const pops[2], void* const rings[2],
                        StepMaps* out) {
  return with_shape<T>(m, [&](auto x, auto y, auto p) {
    return m.flow ? prepare_t<T, true, x(), y(), p()>(m, pops, rings, out)
                  : prepare_t<T, false, x(), y(), p()>(m, pops, rings, out);
  });
}

template <typename T>
cudaError_t launch_any(const Model& m, const StepMaps& maps, int c, const void* src, void* dst,
                       void* ring_cur, unsigned* err, cudaStream_t s) {
  return with_shape<T>(m, [&](auto x, auto y, auto p) {
    return m.flow
               ? launch_tma_t<T, true, x(), y(), p()>(m, maps, c, src, dst, ring_cur, err, s)
               : launch_tma_t<T, false, x(), y(), p()>(m, maps, c, src, dst, ring_cur, err, s);
  });
}

}  // namespace

cudaError_t prepare_step2d(const Model& m, void* const pops[2], void* const rings[2],
                           StepMaps* out) {
  out->ready = 0;
  switch (m.storage) {
    case ST_FP64: return cudaSuccess;  // one-tile kernel, no maps
    case ST_FP16: return prepare_any<__half>(m, pops, rings, out);
    case ST_BF16: return prepare_any<__nv_bfloat16>(m, pops, rings, out);
    default: return prepare_any<float>(m, pops, rings, out);
  }
}

size_t solid_tile_count(const Model& m) {
  const int tx = kShapeX[shape_of(m)], ty = kShapeY[shape_of(m)];
  return size_t((m.nx + tx - 1) / tx) * size_t((m.ny + ty - 1) / ty);
}

cudaError_t launch_solid_tiles(const Model& m, unsigned char* flags, cudaStream_t s) {
  if (m.dim != 2 || !m.solid) return cudaErrorInvalidValue;
  const int tx = kShapeX[shape_of(m)], ty = kShapeY[shape_of(m)];
  const int ntx = (m.nx + tx - 1) / tx, nty = (m.ny + ty - 1) / ty;
  solid_tiles_kernel<<<(ntx * nty + 3) / 4, 128, 0, s>>>(m, flags, ntx, nty, tx, ty);
  return cudaGetLastError();
}

cudaError_t launch_step2d(const Model& m, const StepMaps& maps, int c, const void* src, void* dst,
                          const void* ring_prev, void* ring_cur, unsigned* err, cudaStream_t s) {
  if (m.storage == ST_FP64)
    return m.flow ? launch_plain_t<double, double, true>(m, src, dst, ring_prev, ring_cur, err, s)
                  : launch_plain_t<double, double, false>(m, src, dst, ring_prev, ring_cur, err, s);
  if (!maps.ready) return cudaErrorNotReady;
  switch (m.storage) {
    case ST_FP16: return launch_any<__half>(m, maps, c, src, dst, ring_cur, err, s);
    case ST_BF16: return launch_any<__nv_bfloat16>(m, maps, c, src, dst, ring_cur, err, s);
    default: return launch_any<float>(m, maps, c, src, dst, ring_cur, err, s);
  }
}

}  // namespace lbk
