// Fused coupled LB step in 3D: D3Q19 flow f (Eqs. 4-12), D3Q7 solute g
// (Eqs. 13-18) and D3Q7 phase field h (Eqs. 19-23), push streaming (same
// update as the pull form of the equations).  Per node and step the HBM
// traffic is 33 populations read + 33 written + the phi ring read and written
// (272 B in FP32, 146 B with 16-bit populations).  grad(phi) uses the D3Q19
// stencil; phi(t) and the destination's old h of Eq. 19 come from a one-node
// halo in shared memory.  Populations are deviations d_a = p_a - w_a M_ref
// as in 2D; the ring holds phi + 1.
//
// step3d_column_kernel (FP32 arithmetic: FP32, FP16 and BF16 storage): a CTA
// walks a column of nodes along z, fed plane by plane by the TMA (below).
// step3d_kernel (FP64): one thread per node, one 16 x 4 x 2 tile per CTA; the
// tile's own populations and the halo's h are loaded by the CTA, then every
// node collides and pushes (step3d_core.cuh).
#include <algorithm>

#include "step3d_core.cuh"
#include "tma.cuh"
#include "tma_host.h"

namespace lbk {
namespace {

// ---- FP64 step kernel: one tile per CTA -----------------------------------------
// Bound by the FP64 pipe.  So a warp takes one path: a tile two rows from a face
// holds nodes of both kinds in a warp, and a branch per node runs the arithmetic
// twice (64^3 coupled 361 -> 231 us, 16 x 256 x 256 1661 -> 863).  Three CTAs an SM: with the central
// Hermite MRT that takes 168 registers and a few spills, at 190 and two 6 x 69 x 44
// takes 88 us instead of 75.
template <typename T, typename R, bool FLOW, bool CHM, int TX, int TY, int TZ>
__global__ void __launch_bounds__(TX* TY* TZ, 3)
    step3d_kernel(const Model m, const T* __restrict__ src, T* __restrict__ dst,
                  const R* __restrict__ ring_prev, R* __restrict__ ring_cur,
                  unsigned* __restrict__ err) {
  constexpr int SX = TX + 2, SY = TY + 2, SZ = TZ + 2;
  constexpr int QF = FLOW ? 19 : 0;
  constexpr int NT = TX * TY * TZ;
  __shared__ R sh_phi[SZ][SY][SX];
  __shared__ R sh_h[7][SZ][SY][SX];

  const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, z0 = blockIdx.z * TZ;
  const int x = x0 + tx, y = y0 + ty, z = z0 + tz;
  const int nx = m.nx, ny = m.ny, nz = m.nz, px = m.px;
  const long long P = m.plane;
  const int slab = ny * px;
  const bool active = x < nx && y < ny && z < nz;
  const int idx = z * slab + y * px + x;

  R f[19], g[7], h[7];
  R dphi_prev = R(0);
  if (active) {
#pragma unroll
    for (int a = 0; a < 19; ++a)
      if (FLOW) f[a] = Pop<T>::template ld<R>(src + (a * P + idx));
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      g[a] = Pop<T>::template ld<R>(src + ((QF + a) * P + idx));
      h[a] = Pop<T>::template ld<R>(src + ((QF + 7 + a) * P + idx));
    }
    dphi_prev = ring_prev[idx];
    R s = R(0);
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      s += h[a];  // Eq. 22: phi = -1 + sum d_h
      sh_h[a][tz + 1][ty + 1][tx + 1] = h[a];
    }
    sh_phi[tz + 1][ty + 1][tx + 1] = s;
  }
  const int tid = (tz * TY + ty) * TX + tx;
  for (int i = tid; i < SX * SY * SZ; i += NT) {
    const int lx = i % SX, ly = (i / SX) % SY, lz = i / (SX * SY);
    int gx = x0 + lx - 1, gy = y0 + ly - 1, gz = z0 + lz - 1;
    if (lx >= 1 && lx <= TX && ly >= 1 && ly <= TY && lz >= 1 && lz <= TZ && gx < nx &&
        gy < ny && gz < nz)
      continue;
    if (gx > nx || gy > ny || gz > nz) continue;  // beyond the halo of a partial tile
    gx = grad_coord(gx, nx, m.bc[0]);
    gy = grad_coord(gy, ny, m.bc[1]);
    gz = grad_coord(gz, nz, m.bc[2]);
    const int j = gz * slab + gy * px + gx;
    R s = R(0);
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      const R v = Pop<T>::template ld<R>(src + ((QF + 7 + a) * P + j));
      sh_h[a][lz][ly][lx] = v;
      s += v;
    }
    sh_phi[lz][ly][lx] = s;
  }
  __syncthreads();
  unsigned sm = 0;  // solid neighbours
  if (m.solid && active)
    for (int a = 0; a < 19; ++a)
      sm |= solid_mapped3(m, x + D3_CX[a], y + D3_CY[a], z + D3_CZ[a]) ? 1u << a : 0u;
  const Grid3D gr(m);
  R Unew;
  const unsigned o = unsigned(ty * px + tx) * unsigned(sizeof(T));
  const R dphi = sh_phi[tz + 1][ty + 1][tx + 1];
  auto work = [&](auto edge) {
    collide_push_3d<T, R, FLOW, CHM, true, decltype(edge)::value, false>(
        gr, coef<R>(m), x, y, z, [&](int q) { return q < QF ? f[q] : g[q - QF]; }, h, dphi,
        dphi_prev,
        [&](int dz, int dy, int dx) { return sh_phi[tz + 1 + dz][ty + 1 + dy][tx + 1 + dx]; },
        [&](int a, int dz, int dy, int dx) {
          return sh_h[a][tz + 1 + dz][ty + 1 + dy][tx + 1 + dx];
        },
        [](int, int, int) { return R(0); }, sm, R(coef<R>(m).ref_g),
        dst + ((long long)z * slab + (long long)y0 * px + x0), o, false, err, Unew);
  };
  // one path per warp: a warp with nodes of both kinds would run both
  const bool edge = __any_sync(
      0xffffffffu, active && (sm || x < 1 || x > nx - 2 || y < 1 || y > ny - 2 || z < 1 || z > nz - 2));
  if (!active) return;
  if (edge) work(std::true_type{});
  else work(std::false_type{});
  ring_cur[idx] = dphi;
}

// ---- the column kernel (FP32 arithmetic) ------------------------------------------
// One CTA per column of 32 x 8 nodes and chunk of zc planes, walked along z.
// Per plane the TMA brings, on one mbarrier and one plane ahead, the nodes' own
// f and g (one box of all their arrays), phi(t-1), and h of the plane after
// with a one-node halo in x and y (box starting 16 bytes left of the column so
// that the innermost coordinate stays aligned) into a ring of four planes, so
// every h plane of the column is read once.  phi + 1 of the halo-extended
// planes lives in a ring of its own; a thread keeps its own h in registers
// from the sum of phi to the collision.  One barrier per plane: after it, the
// planes of the step before are read by nobody, and thread 0 issues the next
// copies into them.
//
// Bound by HBM in FP32 (0.90 of the measured copy rate at 256^3); with 16-bit
// storage (0.55) instruction issue and the waits of a plane's chain share the
// time; on small grids that chain alone.  So the halo positions outside the domain get
// their h from the thread that sums phi there: a pass and a barrier of their own
// before that sum had cost the chain 0.35 us of 1.85 a plane (64^3 19.8 -> 17.8 us).
// Per step, against the kernel that moved every tile's arrays to shared memory by
// the threads' own loads: 256^3 FP32 957 -> 762 us, FP16 942 -> 659; 203 x 150 x 134
// FP32 281 -> 229, FP16 284 -> 198; 64^3 FP32 31 -> 18, FP16 36 -> 19.  Columns of 32 x 4
// (128 threads) and of 64 x 4, before that pass was joined: 844 and 863 us at 256^3
// (797 for 32 x 8), FP16 724 and 776 (698): a larger share of halo, 10 / 8 against
// 6 / 4 rows of h; warps that wait on one another's barriers.  256 threads are held to 128
// registers, two CTAs an SM.  Without flow a CTA has half the data and arithmetic of a
// plane, and two do not keep an SM busy: three, at 80 registers without spills.  Per
// step, two CTAs -> three -> one barrier: 97 x 63 x 83 FP32 28.5 -> 22.7 -> 18.6 us, FP16 30.4
// -> 25.4 -> 20.4; 128^3 71.3 -> 63.3 -> 55.5 and 72.4 -> 64.5 -> 54; 256^3 451 -> 396 -> 370 and
// 422 -> 358 -> 328.
//
// 16-bit storage keeps g relative to a per-node U (two FP16 planes, as in
// the 2D step): the node's own reference is read from plane c, its new U
// written there, and every pushed g is encoded against the destination's
// reference in plane c ^ 1, carried with the h ring.
// MASK: the variant with solid nodes; m.solid_tiles says of every 32 x 4 x 8
// nodes whether they or their one-node halo hold a solid node, and a chunk with
// any such carries a ring of the nodes' flags too.
template <typename T, bool FLOW, int TX, int TY>
struct Col3D {
  static constexpr int QFG = (FLOW ? 19 : 0) + 7;
  static constexpr int HX = 16 / int(sizeof(T)), BXH = TX + 2 * HX, SX = TX + 2, SY = TY + 2;
  static constexpr bool REL = sizeof(T) == 2;
  static constexpr int HXU = 8, BXU = TX + 2 * HXU;
  static constexpr int HPLANE = SY * BXH;  // one array of an h plane
  static constexpr int FG_BYTES = QFG * TY * TX * int(sizeof(T));
  static constexpr int H_BYTES = 7 * HPLANE * int(sizeof(T));
  static constexpr int RING_BYTES = TY * TX * 4;
  static constexpr int UOWN_BYTES = REL ? TY * TX * 2 : 0;
  static constexpr int UHAL_BYTES = REL ? SY * BXU * 2 : 0;
  static constexpr int al(int b) { return (b + 127) / 128 * 128; }
  // own data of a plane, two of them; h (and the encoding reference), four
  static constexpr int OFF_RING = al(FG_BYTES), OFF_UOWN = OFF_RING + al(RING_BYTES);
  static constexpr int OWN = OFF_UOWN + al(UOWN_BYTES);
  static constexpr int HAL = al(H_BYTES) + al(UHAL_BYTES);
  static constexpr int OFF_HAL = 2 * OWN;
  static constexpr int OFF_PHI = OFF_HAL + 4 * HAL;
  static constexpr int SMEM = OFF_PHI + al(4 * SX * SY * 4);
  static constexpr int OWN_TX = FG_BYTES + RING_BYTES + UOWN_BYTES;
  static constexpr int HAL_TX = H_BYTES + UHAL_BYTES;
};

// blocks of nodes with a flag for solid nodes: rows of a column, so that a
// column's flags are those of a few blocks
constexpr int kFlagX = 32, kFlagY = 4, kFlagZ = 8;
// CTAs (of 256 threads) an SM holds
constexpr int col_ctas(bool flow) { return flow ? 2 : 3; }
constexpr int kSpin3 = 1 << 22;  // bound on mbarrier polls before giving up

template <typename T, bool FLOW, int TX, int TY, bool CHM, bool MASK>
__global__ void __launch_bounds__(TX* TY, col_ctas(FLOW))
    step3d_column_kernel(const __grid_constant__ CUtensorMap tm_fg,
                         const __grid_constant__ CUtensorMap tm_h,
                         const __grid_constant__ CUtensorMap tm_ring,
                         const __grid_constant__ CUtensorMap tm_uown,
                         const __grid_constant__ CUtensorMap tm_uhal, const Model m,
                         const T* __restrict__ src, T* __restrict__ dst,
                         float* __restrict__ ring_cur, unsigned* __restrict__ err, int zc, int c) {
  using L = Col3D<T, FLOW, TX, TY>;
  static_assert(TX == kFlagX && TY % kFlagY == 0, "a column is made of whole blocks");
  constexpr int NT = TX * TY;
  constexpr int SX = L::SX, SY = L::SY, PL = SX * SY, HPLANE = L::HPLANE;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[2], first[1];
  __shared__ unsigned char sh_solid[MASK ? 4 : 1][MASK ? PL : 1];
  float* const sh_phi = reinterpret_cast<float*>(smem + L::OFF_PHI);
  const Grid3D gr(m);
  const Coef<float>& cf = m.cf;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int x = x0 + tx, y = y0 + ty;
  const int nx = gr.nx, ny = gr.ny, nz = gr.nz, px = gr.px, slab = gr.slab;
  const int zs = blockIdx.z * zc;
  const int ze = zs + zc < nz ? zs + zc : nz;
  const int nfy = (ny + kFlagY - 1) / kFlagY;
  auto flag = [&](int fy, int fz) {  // of the column's blocks of nodes in x
    return MASK && m.solid && fy < nfy &&
           m.solid_tiles[(size_t(fz) * nfy + fy) * gridDim.x + blockIdx.x] != 0;
  };
  bool solids = false;
  for (int fz = zs / kFlagZ; MASK && fz <= (ze - 1) / kFlagZ; ++fz)
    for (int fy = 0; fy < TY / kFlagY; ++fy) solids |= flag(y0 / kFlagY + fy, fz);
  // 16-bit storage: the blocks of 32 x 4 nodes away from the faces (see aniso_3d)
  const int yb = y & ~(kFlagY - 1);
  const bool inner_xy = x0 >= 1 && x0 + TX <= nx - 1 && yb >= 1 && yb + kFlagY <= ny - 1;
  const bool rim = x0 == 0 || y0 == 0 || x0 + TX >= nx || y0 + TY >= ny;

  // slot of plane z in the h, phi and flag rings
  auto slot = [&](int z) { return (z - zs + 1) & 3; };
  auto h_slot = [&](int z) { return reinterpret_cast<T*>(smem + L::OFF_HAL + slot(z) * L::HAL); };
  auto u_slot = [&](int z) {
    return reinterpret_cast<__half*>(smem + L::OFF_HAL + slot(z) * L::HAL + L::al(L::H_BYTES));
  };
  auto load_h = [&](int z, uint64_t* bar) {  // thread 0
    const int gz = grad_coord(z, nz, gr.bc[2]);
    tma_load_4d(h_slot(z), &tm_h, bar, x0 - L::HX, y0 - 1, gz, L::QFG);
    if (L::REL) tma_load_4d(u_slot(z), &tm_uhal, bar, x0 - L::HXU, y0 - 1, gz, c ^ 1);
  };
  auto load_step = [&](int z) {  // thread 0: own data of plane z, h of plane z + 1
    uint64_t* const bar = &full[(z - zs) & 1];
    unsigned char* const own = smem + ((z - zs) & 1) * L::OWN;
    mbar_arrive_expect_tx(bar, L::OWN_TX + L::HAL_TX);
    tma_load_4d(own, &tm_fg, bar, x0, y0, z, 0);
    tma_load_3d(own + L::OFF_RING, &tm_ring, bar, x0, y0, z);
    if (L::REL) tma_load_4d(own + L::OFF_UOWN, &tm_uown, bar, x0, y0, z, c);
    load_h(z + 1, bar);
  };
  // phi + 1 of plane z with halo (and the solid flags) from its h: each
  // thread's own node from the h it keeps for the collision, the ring around
  // the column's nodes by one thread a position.  That thread also gives the
  // positions outside the domain their h: the nearest node's, which the box
  // holds, or across a periodic edge the far side's.  (In a partial column the ring
  // runs through positions of idle threads, which write nothing there and store no
  // result.)
  const int oh = (ty + 1) * L::BXH + tx + L::HX, op = (ty + 1) * SX + tx + 1;
  const int vx = nx - x0 < TX ? nx - x0 : TX, vy = ny - y0 < TY ? ny - y0 : TY;
  const bool on_ring = (x == nx && y <= ny) || (y == ny && x <= nx);
  static_assert(2 * SX + 2 * TY <= NT, "a thread for every position of the ring");
  auto sum_phi = [&](int z, float(&h)[7]) {
    T* const hs = h_slot(z);
    float* const ps = sh_phi + slot(z) * PL;
    float s = 0.f;
#pragma unroll
    for (int a = 0; a < 7; ++a) {
      h[a] = Pop<T>::template ld<float>(hs + a * HPLANE + oh);
      s = a == 0 ? h[0] : add_r(s, h[a]);
    }
    if (!on_ring) ps[op] = s;
    if (tid < 2 * (vx + 2) + 2 * vy) {
      int lx, ly, i = tid;
      if (i < 2 * (vx + 2)) {
        lx = i < vx + 2 ? i : i - (vx + 2);
        ly = i < vx + 2 ? 0 : vy + 1;
      } else {
        i -= 2 * (vx + 2);
        lx = i & 1 ? vx + 1 : 0;
        ly = 1 + i / 2;
      }
      T* const p = hs + ly * L::BXH + lx + L::HX - 1;
      T v[7];
      const int gx = x0 + lx - 1, gy = y0 + ly - 1;
      if (!rim || (gx >= 0 && gx < nx && gy >= 0 && gy < ny)) {
#pragma unroll
        for (int a = 0; a < 7; ++a) v[a] = p[a * HPLANE];
      } else {
        const int wx = grad_coord(gx, nx, gr.bc[0]), wy = grad_coord(gy, ny, gr.bc[1]);
        const int sx = wx - x0 + 1, sy = wy - y0 + 1;  // the mapped node in the box
        __half* const us = u_slot(z);
        __half* const ud = us + ly * L::BXU + lx + L::HXU - 1;
        if (sx >= 0 && sx < SX && sy >= 0 && sy < SY) {
          const T* const hf = hs + sy * L::BXH + sx + L::HX - 1;
#pragma unroll
          for (int a = 0; a < 7; ++a) v[a] = hf[a * HPLANE];
          if (L::REL) *ud = us[sy * L::BXU + sx + L::HXU - 1];
        } else {
          const int gz = grad_coord(z, nz, gr.bc[2]);
          const long long j = (long long)gz * slab + (long long)wy * px + wx, P = gr.plane;
#pragma unroll
          for (int a = 0; a < 7; ++a) v[a] = src[(L::QFG + a) * P + j];
          if (L::REL) *ud = m.uring[(c ^ 1) * P + j];
        }
#pragma unroll
        for (int a = 0; a < 7; ++a) p[a * HPLANE] = v[a];
      }
      float r = 0.f;
#pragma unroll
      for (int a = 0; a < 7; ++a) r += Pop<T>::template ld<float>(&v[a]);
      ps[ly * SX + lx] = r;
    }
    if (MASK && solids) {
      const int gz = grad_coord(z, nz, gr.bc[2]);
      for (int i = tid; i < PL; i += NT) {
        const int gx = x0 + i % SX - 1, gy = y0 + i / SX - 1;
        unsigned char v = 0;
        if (gx <= nx && gy <= ny)
          v = m.solid[(long long)gz * slab + (long long)grad_coord(gy, ny, gr.bc[1]) * px +
                      grad_coord(gx, nx, gr.bc[0])];
        sh_solid[MASK ? slot(z) : 0][MASK ? i : 0] = v;
      }
    }
  };

  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&first[0], 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (tid == 0) {
    mbar_arrive_expect_tx(&first[0], 2 * L::HAL_TX);
    load_h(zs - 1, &first[0]);
    load_h(zs, &first[0]);
    load_step(zs);
  }
  bool ok = mbar_wait_bounded(&first[0], 0, kSpin3);
  float h[7], hn[7];  // the node's own h in planes z and z + 1
  sum_phi(zs - 1, h);
  sum_phi(zs, h);

  const int o = ty * TX + tx;
  const unsigned e = unsigned(ty * px + tx);
  for (int z = zs; z < ze; ++z) {
    const int k = z - zs;
    ok = mbar_wait_bounded(&full[k & 1], uint32_t(k >> 1) & 1u, kSpin3) && ok;
    sum_phi(z + 1, hn);
    if (__syncthreads_or(!ok)) {
      // a plane never arrived: report, let the copies in flight land, stop
      if (tid == 0) {
        atomicOr(err, 2u);
        mbar_wait_bounded(&full[k & 1], uint32_t(k >> 1) & 1u, kSpin3);
      }
      __syncthreads();
      return;
    }
    if (tid == 0 && z + 1 < ze) {
      fence_proxy_async_smem();
      load_step(z + 1);
    }
    const unsigned char* const own = smem + (k & 1) * L::OWN;
    const T* const fg = reinterpret_cast<const T*>(own);
    const float* const ring = reinterpret_cast<const float*>(own + L::OFF_RING);
    const __half* const uo = reinterpret_cast<const __half*>(own + L::OFF_UOWN);
    const float* ps[3];
    const T* hp[3];
    const __half* up[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      ps[d] = sh_phi + slot(z + d - 1) * PL + op;
      hp[d] = h_slot(z + d - 1) + oh;
      up[d] = u_slot(z + d - 1) + (ty + 1) * L::BXU + tx + L::HXU;
    }
    unsigned sm = 0;  // solid neighbours (bit a: direction a, 0 the node itself)
    if (MASK && solids)
#pragma unroll
      for (int a = 0; a < 19; ++a)
        sm |= sh_solid[MASK ? slot(z + D3_CZ[a]) : 0][MASK ? op + D3_CY[a] * SX + D3_CX[a] : 0]
                  ? 1u << a
                  : 0u;
    const float dphi = ps[1][0];
    float Rg = cf.ref_g, Unew;
    if constexpr (L::REL) Rg = __half2float(uo[o]);
    const long long org = (long long)z * slab + (long long)y0 * px + x0;
    const bool y_first = L::REL && inner_xy && z >= 1 && z <= nz - 2 &&
                         !(solids && flag(y / kFlagY, z / kFlagZ));
    auto work = [&](auto edge) {
      collide_push_3d<T, float, FLOW, CHM, MASK, decltype(edge)::value, L::REL>(
          gr, cf, x, y, z, [&](int q) { return Pop<T>::template ld<float>(fg + q * (TY * TX) + o); },
          h, dphi, ring[o],
          [&](int dz, int dy, int dx) { return ps[dz + 1][dy * SX + dx]; },
          [&](int a, int dz, int dy, int dx) {
            return Pop<T>::template ld<float>(hp[dz + 1] + a * HPLANE + dy * L::BXH + dx);
          },
          [&](int dz, int dy, int dx) { return __half2float(up[dz + 1][dy * L::BXU + dx]); }, sm,
          Rg, dst + org, e * unsigned(sizeof(T)), y_first, err, Unew);
    };
    // boundary logic only for the warps that have a node on a domain face or
    // next to a solid node
    const bool edge =
        z < 1 || z > nz - 2 ||
        __any_sync(0xffffffffu, sm != 0 || x < 1 || x > nx - 2 || y < 1 || y > ny - 2);
    if (edge) work(std::true_type{});
    else work(std::false_type{});
    // phi(t) of every node, and the new U of every node but the solid ones
    if (!edge || (x < nx && y < ny)) {
      (ring_cur + org)[e] = dphi;
      if constexpr (L::REL)
        if (!(sm & 1u)) (m.uring + (c * gr.plane + org))[e] = __float2half_rn(Unew);
    }
#pragma unroll
    for (int a = 0; a < 7; ++a) h[a] = hn[a];
  }
}

// A column's nodes (above), and the planes per chunk: the fewest plane steps
// of the busiest slot, with col_ctas CTAs on each of 152 SMs and a chunk of zc planes
// costing its first planes' h as well (about a plane and a half; 64^3: 46, 24 and
// 18 us at 16, 8 and 4 planes).  At 256^3 4, 8 and 16 planes take 779, 763 and 773
// us (FP16 697, 660 and 657), at 203 x 150 x 134 229, 229 and 236, at 40 x 44 x 48
// 14.1, 24.5 and 45.5 (11.2 at the 2 planes chosen there): so never more than 8, but
// where gridDim.z asks for it.  On 17 grids the choice is within 8 % of the best of 1 to
// 32 planes.
constexpr int kColX = 32, kColY = 8;

int col_planes(const Model& m) {
  const long long cols = (long long)((m.nx + kColX - 1) / kColX) * ((m.ny + kColY - 1) / kColY);
  const int slots = 152 * col_ctas(m.flow);
  int best = 8;
  double cost = 1e300;
  const int least = (m.nz + 65534) / 65535;  // gridDim.z
  for (int zc = std::max(8, least); zc >= least; --zc) {
    const long long ctas = cols * ((m.nz + zc - 1) / zc);
    const double t = double((ctas + slots - 1) / slots) * (zc + 1.5);
    if (t < cost) cost = t, best = zc;
  }
  return std::min(best, m.nz);
}

template <typename T, bool FLOW>
cudaError_t prepare3_t(const Model& m, void* const pops[2], void* const rings[2], StepMaps* out) {
  constexpr int TX = kColX, TY = kColY;
  using L = Col3D<T, FLOW, TX, TY>;
  const uint64_t nx = m.nx, ny = m.ny, nz = m.nz, es = sizeof(T);
  for (int b = 0; b < 2; ++b) {
    const uint64_t dims[4] = {nx, ny, nz, uint64_t(L::QFG + 7)};
    const uint64_t str[3] = {m.px * es, ny * m.px * es, uint64_t(m.plane) * es};
    const uint32_t box_fg[4] = {TX, TY, 1, uint32_t(L::QFG)};
    const uint32_t box_h[4] = {uint32_t(L::BXH), uint32_t(L::SY), 1, 7};
    const uint64_t dimr[3] = {nx, ny, nz}, strr[2] = {uint64_t(m.px) * 4, ny * m.px * 4};
    const uint32_t box_r[3] = {TX, TY, 1};
    if (!encode_tiled(&out->fg[b], pop_tensor_type(m.storage), 4, pops[b], dims, str, box_fg) ||
        !encode_tiled(&out->h[b], pop_tensor_type(m.storage), 4, pops[b], dims, str, box_h) ||
        !encode_tiled(&out->ring[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, rings[b], dimr, strr,
                      box_r))
      return cudaErrorInvalidValue;
  }
  if (L::REL) {
    if (!m.uring) return cudaErrorInvalidValue;
    const uint64_t dims[4] = {nx, ny, nz, 2};
    const uint64_t str[3] = {uint64_t(m.px) * 2, ny * m.px * 2, uint64_t(m.plane) * 2};
    const uint32_t box_o[4] = {TX, TY, 1, 1}, box_h[4] = {uint32_t(L::BXU), uint32_t(L::SY), 1, 1};
    if (!encode_tiled(&out->uown, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, m.uring, dims, str, box_o) ||
        !encode_tiled(&out->uhal, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, m.uring, dims, str, box_h))
      return cudaErrorInvalidValue;
  } else {
    out->uown = out->uhal = out->ring[0];  // unused
  }
  auto setup = [&](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
  };
  cudaError_t e;
  if ((e = setup(step3d_column_kernel<T, FLOW, TX, TY, false, false>)) != cudaSuccess ||
      (e = setup(step3d_column_kernel<T, FLOW, TX, TY, false, true>)) != cudaSuccess ||
      (e = setup(step3d_column_kernel<T, FLOW, TX, TY, FLOW, false>)) != cudaSuccess ||
      (e = setup(step3d_column_kernel<T, FLOW, TX, TY, FLOW, true>)) != cudaSuccess)
    return e;
  out->smem = L::SMEM;
  out->ready = 1;
  return cudaSuccess;
}

template <typename T, bool FLOW>
cudaError_t launch3_column_t(const Model& m, const StepMaps& maps, int c, const void* src,
                             void* dst, void* ring_cur, unsigned* err, cudaStream_t s) {
  constexpr int TX = kColX, TY = kColY;
  const int zc = col_planes(m);
  const dim3 grid((m.nx + TX - 1) / TX, (m.ny + TY - 1) / TY, (m.nz + zc - 1) / zc);
  auto kern =
      m.solid ? (FLOW && m.chm ? step3d_column_kernel<T, FLOW, TX, TY, FLOW, true>
                               : step3d_column_kernel<T, FLOW, TX, TY, false, true>)
              : (FLOW && m.chm ? step3d_column_kernel<T, FLOW, TX, TY, FLOW, false>
                               : step3d_column_kernel<T, FLOW, TX, TY, false, false>);
  kern<<<grid, TX * TY, maps.smem, s>>>(
      maps.fg[c], maps.h[c], maps.ring[c], maps.uown, maps.uhal, m, static_cast<const T*>(src),
      static_cast<T*>(dst), static_cast<float*>(ring_cur), err, zc, c);
  return cudaGetLastError();
}

// one warp per kFlagX x kFlagY x kFlagZ block of nodes: does it or its one-node
// halo (mapped like the gradient stencil) hold a solid node?
__global__ void solid_chunks_kernel(const Model m, unsigned char* flags, int ntx, int nty,
                                    int nzc) {
  const int t = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (t >= ntx * nty * nzc) return;
  const int x0 = (t % ntx) * kFlagX, y0 = ((t / ntx) % nty) * kFlagY,
            z0 = (t / (ntx * nty)) * kFlagZ;
  const int xe = x0 + kFlagX < m.nx ? x0 + kFlagX : m.nx;
  const int ye = y0 + kFlagY < m.ny ? y0 + kFlagY : m.ny;
  const int ze = z0 + kFlagZ < m.nz ? z0 + kFlagZ : m.nz;
  bool any = false;
  for (int z = z0 - 1; z <= ze && !any; ++z) {
#pragma unroll 2
    for (int y = y0 - 1; y <= ye; ++y)
      for (int x = x0 - 1 + lane; x <= xe; x += 32) any |= solid_mapped3(m, x, y, z);
    any = __any_sync(0xffffffffu, any);
  }
  if (lane == 0) flags[t] = any ? 1 : 0;
}

// ---- host side -------------------------------------------------------------------
template <typename T, typename R, bool FLOW>
cudaError_t launch3_plain_t(const Model& m, const void* src, void* dst, const void* ring_prev,
                            void* ring_cur, unsigned* err, cudaStream_t s) {
  constexpr int TX = 16, TY = 4, TZ = 2;
  dim3 block(TX, TY, TZ);
  dim3 grid((m.nx + TX - 1) / TX, (m.ny + TY - 1) / TY, (m.nz + TZ - 1) / TZ);
  auto kern = FLOW && m.chm ? step3d_kernel<T, R, FLOW, FLOW, TX, TY, TZ>
                            : step3d_kernel<T, R, FLOW, false, TX, TY, TZ>;
  kern<<<grid, block, 0, s>>>(m, static_cast<const T*>(src), static_cast<T*>(dst),
                              static_cast<const R*>(ring_prev), static_cast<R*>(ring_cur), err);
  return cudaGetLastError();
}

template <typename T>
cudaError_t prepare3_any(const Model& m, void* const pops[2], void* const rings[2],
                         StepMaps* out) {
  return m.flow ? prepare3_t<T, true>(m, pops, rings, out)
                : prepare3_t<T, false>(m, pops, rings, out);
}
template <typename T>
cudaError_t launch3_any(const Model& m, const StepMaps& maps, int c, const void* src, void* dst,
                        void* ring_cur, unsigned* err, cudaStream_t s) {
  return m.flow ? launch3_column_t<T, true>(m, maps, c, src, dst, ring_cur, err, s)
                : launch3_column_t<T, false>(m, maps, c, src, dst, ring_cur, err, s);
}

}  // namespace

size_t solid_chunk_count(const Model& m) {
  return size_t((m.nx + kFlagX - 1) / kFlagX) * size_t((m.ny + kFlagY - 1) / kFlagY) *
         size_t((m.nz + kFlagZ - 1) / kFlagZ);
}

cudaError_t launch_solid_chunks(const Model& m, unsigned char* flags, cudaStream_t s) {
  if (m.dim != 3 || !m.solid) return cudaErrorInvalidValue;
  const int ntx = (m.nx + kFlagX - 1) / kFlagX, nty = (m.ny + kFlagY - 1) / kFlagY,
            nzc = (m.nz + kFlagZ - 1) / kFlagZ;
  const int n = ntx * nty * nzc;
  solid_chunks_kernel<<<(n + 3) / 4, 128, 0, s>>>(m, flags, ntx, nty, nzc);
  return cudaGetLastError();
}

cudaError_t prepare_step3d(const Model& m, void* const pops[2], void* const rings[2],
                           StepMaps* out) {
  out->ready = 0;
  switch (m.storage) {
    case ST_FP64: return cudaSuccess;  // one-tile kernel, no maps
    case ST_FP16: return prepare3_any<__half>(m, pops, rings, out);
    case ST_BF16: return prepare3_any<__nv_bfloat16>(m, pops, rings, out);
    default: return prepare3_any<float>(m, pops, rings, out);
  }
}

cudaError_t launch_step3d(const Model& m, const StepMaps& maps, int c, const void* src, void* dst,
                          const void* ring_prev, void* ring_cur, unsigned* err, cudaStream_t s) {
  if (m.storage == ST_FP64)
    return m.flow ? launch3_plain_t<double, double, true>(m, src, dst, ring_prev, ring_cur, err, s)
                  : launch3_plain_t<double, double, false>(m, src, dst, ring_prev, ring_cur, err, s);
  if (!maps.ready) return cudaErrorNotReady;
  switch (m.storage) {
    case ST_FP16: return launch3_any<__half>(m, maps, c, src, dst, ring_cur, err, s);
    case ST_BF16: return launch3_any<__nv_bfloat16>(m, maps, c, src, dst, ring_cur, err, s);
    default: return launch3_any<float>(m, maps, c, src, dst, ring_cur, err, s);
  }
}

}  // namespace lbk
