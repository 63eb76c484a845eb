// One tile of the TMA-fed 2D step, shared by the single-grid and the batched
// persistent kernels: shared-memory layout of a pipeline stage, the three TMA
// loads that fill it, and the work on a filled stage (edge patching, phi + 1
// of the halo-extended tile, per-node collide and push).
#pragma once

#include "step2d_core.cuh"
#include "tma.cuh"

namespace lbk {

template <typename T, bool FLOW, int TX, int TY>
struct Tiles2D {
  static constexpr int QFG = (FLOW ? 9 : 0) + 9;   // f and g arrays
  static constexpr int HX = 16 / int(sizeof(T));   // halo box starts HX left of the tile
  static constexpr int BXH = TX + 2 * HX;          // h box width
  static constexpr int FG_BYTES = QFG * TY * TX * int(sizeof(T));
  static constexpr int H_BYTES = 9 * (TY + 2) * BXH * int(sizeof(T));
  static constexpr int RING_BYTES = TY * TX * 4;
  // 16-bit storage: g relative to a per-node U (the own reference of the tile
  // and a halo box of the encoding reference, FP16, starting 8 left of the
  // tile so that the box starts on a 16-byte boundary)
  static constexpr bool REL = sizeof(T) == 2;
  static constexpr int HXU = 8, BXU = TX + 2 * HXU;
  static constexpr int UOWN_BYTES = REL ? TY * TX * 2 : 0;
  static constexpr int UHAL_BYTES = REL ? (TY + 2) * BXU * 2 : 0;
  static constexpr int al(int b) { return (b + 127) / 128 * 128; }
  static constexpr int OFF_H = al(FG_BYTES);
  static constexpr int OFF_RING = OFF_H + al(H_BYTES);
  static constexpr int OFF_UOWN = OFF_RING + al(RING_BYTES);
  static constexpr int OFF_UHAL = OFF_UOWN + al(UOWN_BYTES);
  static constexpr int STAGE = OFF_UHAL + al(UHAL_BYTES);
  static constexpr int TX_BYTES = FG_BYTES + H_BYTES + RING_BYTES + UOWN_BYTES + UHAL_BYTES;
};

// Fill one stage: f and g of the tile, h with its halo, the phi ring; with
// 16-bit storage also the tile's U reference (plane c) and the halo of the
// encoding reference (plane c ^ 1).
template <typename T, bool FLOW, int TX, int TY>
__device__ __forceinline__ void issue_tile_2d(const CUtensorMap* tm_fg, const CUtensorMap* tm_h,
                                              const CUtensorMap* tm_ring,
                                              const CUtensorMap* tm_uown,
                                              const CUtensorMap* tm_uhal, int c, uint64_t* bar,
                                              unsigned char* st, int x0, int y0) {
  using L = Tiles2D<T, FLOW, TX, TY>;
  mbar_arrive_expect_tx(bar, L::TX_BYTES);
  tma_load_3d(st, tm_fg, bar, x0, y0, 0);
  tma_load_3d(st + L::OFF_H, tm_h, bar, x0 - L::HX, y0 - 1, L::QFG);
  tma_load_2d(st + L::OFF_RING, tm_ring, bar, x0, y0);
  if (L::REL) {
    tma_load_3d(st + L::OFF_UOWN, tm_uown, bar, x0, y0, c);
    tma_load_3d(st + L::OFF_UHAL, tm_uhal, bar, x0 - L::HXU, y0 - 1, c ^ 1);
  }
}

// Threads that work on a TX x TY tile.  PAIR: a thread holds the two nodes
// (tx, ty) and (tx, ty + TY / 2), so that interior tiles run on the packed
// two-lane FP32 instructions.
template <int TX, int TY, bool PAIR>
constexpr int tile_threads() {
  return PAIR ? TX * TY / 2 : TX * TY;
}

// Work on a filled stage `st` for the tile at (x0, y0).  Called by all
// threads of the CTA; contains CTA barriers.  sh_phi: (TY + 2) x (TX + 2).
// `bad`: this thread saw the stage's loads time out; the first barrier tells
// every thread, and the tile is given up before its first global write
// (returns false).  MASK: solid nodes are handled (sh_solid: (TY + 2) x (TX + 2)
// bytes); `solids`: the tile or its halo holds one.  CHM: the flow collides by
// the central Hermite MRT.
template <typename T, bool FLOW, int TX, int TY, bool PAIR, bool MASK, bool CHM>
__device__ __forceinline__ bool tile_2d(const Grid2D& gr, const Model& m,
                                        const T* __restrict__ src, T* __restrict__ dst,
                                        float* __restrict__ ring_cur, unsigned* __restrict__ err,
                                        int x0, int y0, int c, unsigned char* st,
                                        float* sh_phi_flat, unsigned char* sh_solid, bool solids,
                                        bool bad) {
  using R = float;
  using L = Tiles2D<T, FLOW, TX, TY>;
  constexpr int NT = tile_threads<TX, TY, PAIR>(), SX = TX + 2, SY = TY + 2;
  constexpr int V = PAIR ? 2 : 1, DY = TY / 2;
  constexpr int QF = FLOW ? 9 : 0;
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int nx = gr.nx, ny = gr.ny, px = gr.px;
  R(*sh_phi)[SX] = reinterpret_cast<R(*)[SX]>(sh_phi_flat);
  const T* fgs = reinterpret_cast<const T*>(st);
  T* hsm = reinterpret_cast<T*>(st + L::OFF_H);
  const float* rings = reinterpret_cast<const float*>(st + L::OFF_RING);
  const __half* uown = reinterpret_cast<const __half*>(st + L::OFF_UOWN);
  __half* uhal = reinterpret_cast<__half*>(st + L::OFF_UHAL);
  constexpr int HPLANE = SY * L::BXH;
  if (MASK && solids) {  // the tile's solid flags with halo, for the general path
    for (int i = tid; i < SX * SY; i += NT) {
      const int gx = x0 + i % SX - 1, gy = y0 + i / SX - 1;
      unsigned char v = 0;
      if (gx <= nx && gy <= ny)
        v = gr.solid[(long long)grad_coord(gy, ny, gr.bcy) * px + grad_coord(gx, nx, gr.bcx)];
      sh_solid[i] = v;
    }
  }
  if (x0 == 0 || y0 == 0 || x0 + TX >= nx || y0 + TY >= ny) {
    // halo positions outside the domain: the nearest node, which the tile
    // holds, or across a periodic edge the far side (or, where the tile spans
    // the domain, its own other side)
    for (int i = tid; i < SX * SY; i += NT) {
      const int lx = i % SX, ly = i / SX;
      int gx = x0 + lx - 1, gy = y0 + ly - 1;
      if (gx >= 0 && gx < nx && gy >= 0 && gy < ny) continue;
      if (gx > nx || gy > ny) continue;  // beyond the halo of a partial tile
      const int wx = grad_coord(gx, nx, gr.bcx), wy = grad_coord(gy, ny, gr.bcy);
      const int sx = wx - x0 + 1, sy = wy - y0 + 1;  // the mapped node in the tile's box
      T* const hd = hsm + ly * L::BXH + lx + L::HX - 1;
      __half* const ud = uhal + ly * L::BXU + lx + L::HXU - 1;
      if (sx >= 0 && sx < SX && sy >= 0 && sy < SY) {
        const T* const hf = hsm + sy * L::BXH + sx + L::HX - 1;
#pragma unroll
        for (int a = 0; a < 9; ++a) hd[a * HPLANE] = hf[a * HPLANE];
        if (L::REL) *ud = uhal[sy * L::BXU + sx + L::HXU - 1];
      } else {
        const long long j = (long long)wy * px + wx, P = gr.plane;
#pragma unroll
        for (int a = 0; a < 9; ++a) hd[a * HPLANE] = src[(QF + 9 + a) * P + j];
        if (L::REL) *ud = gr.uring[(c ^ 1) * gr.plane + j];
      }
    }
    __syncthreads();
  }
  // phi + 1 of the halo-extended tile: each thread's own positions from the
  // h it keeps for the collision, the ring around the tile by a pass
  const T* hown = hsm + (ty + 1) * L::BXH + tx + L::HX;
  using N = std::conditional_t<PAIR, float2, float>;
  auto h_at = [&](int a, int off) -> N {  // h_a at `off` from the thread's node(s)
    const T* p = hown + a * HPLANE + off;
    if constexpr (PAIR)
      return make_float2(Pop<T>::template ld<R>(p), Pop<T>::template ld<R>(p + DY * L::BXH));
    else
      return Pop<T>::template ld<R>(p);
  };
  N h[9], dphi;
  {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      h[a] = h_at(a, 0);
      dphi = a == 0 ? h[0] : add_r(dphi, h[a]);
    }
    if constexpr (PAIR) {
      sh_phi[ty + 1][tx + 1] = dphi.x;
      sh_phi[ty + 1 + DY][tx + 1] = dphi.y;
    } else {
      sh_phi[ty + 1][tx + 1] = dphi;
    }
  }
  constexpr int NRING = 2 * SX + 2 * TY;
  for (int i = tid; i < NRING; i += NT) {
    int lx, ly;
    if (i < 2 * SX) {
      lx = i % SX;
      ly = i < SX ? 0 : SY - 1;
    } else {
      lx = (i - 2 * SX) & 1 ? SX - 1 : 0;
      ly = 1 + (i - 2 * SX) / 2;
    }
    const T* hp = hsm + ly * L::BXH + lx + L::HX - 1;
    R sum = R(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) sum += Pop<T>::template ld<R>(hp + a * HPLANE);
    sh_phi[ly][lx] = sum;
  }
  if (__syncthreads_or(bad)) return false;

  const int x = x0 + tx, y = y0 + ty;
  const int o = ty * TX + tx;
  auto two = [](float v, float w) -> N {
    if constexpr (PAIR) return make_float2(v, w);
    else return v;
  };
  // g is stored relative to the node's own U reference (16-bit storage); the
  // collision takes the deviations from it as they are
  const Coef<N>& cf = coef<N>(m);
  N Rg = cf.ref_g, Unew;
  if constexpr (L::REL) Rg = two(__half2float(uown[o]), __half2float(uown[o + (V - 1) * DY * TX]));
  const __half* uc = uhal + (ty + 1) * L::BXU + tx + L::HXU;
  const size_t org = size_t(y0) * px + x0;
  const unsigned e0 = unsigned(ty * px + tx), e1 = e0 + unsigned(DY * px);
  unsigned sm[V], near = 0;  // solid neighbours (bit a: direction a, 0 the node itself)
#pragma unroll
  for (int k = 0; k < V; ++k) {
    sm[k] = 0;
    if (MASK && solids)
#pragma unroll
      for (int a = 0; a < 9; ++a)
        sm[k] |= sh_solid[(ty + k * DY + 1 + D2_CY[a]) * SX + tx + 1 + D2_CX[a]] ? 1u << a : 0u;
    near |= sm[k];
  }
  auto work = [&](auto edge) {
    collide_push_2d<T, N, FLOW, CHM, MASK, decltype(edge)::value, L::REL, SX, DY>(
        gr, cf, x, y,
        [&](int q) {
          const T* p = fgs + q * (TY * TX) + o;
          return two(Pop<T>::template ld<R>(p), Pop<T>::template ld<R>(p + (V - 1) * DY * TX));
        },
        h, dphi, two(rings[o], rings[o + (V - 1) * DY * TX]), &sh_phi[ty + 1][tx + 1],
        [&](int a, int dy, int dx) { return h_at(a, dy * L::BXH + dx); },
        [&](int dy, int dx) {
          const __half* p = uc + dy * L::BXU + dx;
          return two(__half2float(p[0]), __half2float(p[(V - 1) * DY * L::BXU]));
        },
        sm, Rg, dst + org, e0 * unsigned(sizeof(T)), e1 * unsigned(sizeof(T)), err, Unew);
  };
  // boundary logic only for the warps that have a node on a domain edge or
  // next to a solid node
  const bool edge = __any_sync(0xffffffffu, near != 0 || x < 1 || x > nx - 2 || y < 1 ||
                                                y + (V - 1) * DY > ny - 2);
  if (edge) work(std::true_type{});
  else work(std::false_type{});
  // phi(t) of every node, and the new U of every node but the solid ones
  float* ring_t = ring_cur + org;
  __half* un = L::REL ? gr.uring + (c * gr.plane + (long long)org) : nullptr;
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const unsigned e = k ? e1 : e0;
    if (!edge || (x < nx && y + k * DY < ny)) {
      ring_t[e] = lane(dphi, k);
      if constexpr (L::REL)
        if (!(sm[k] & 1u)) un[e] = __float2half_rn(lane(Unew, k));
    }
  }
  return true;
}

}  // namespace lbk
