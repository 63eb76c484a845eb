// Per-node part of the 2D coupled step, shared by the step kernels: moments,
// anisotropy, collisions of f, g and h, and the push of every direction to
// its destination (Eqs. 3-23).  The caller has the node's own population
// deviations in registers and the tile's phi + 1 and h deviations (with a
// one-node halo) in shared memory.
#pragma once

#include "lbpf_device.cuh"

namespace lbk {

// Solid nodes (2D mask): is the node at (x, y), mapped like a gradient
// neighbour (periodic wrap, else nearest node), solid?
__device__ __forceinline__ bool solid_mapped(const Model& m, int x, int y) {
  x = grad_coord(x, m.nx, m.bc[0]);
  y = grad_coord(y, m.ny, m.bc[1]);
  return m.solid[(long long)y * m.px + x] != 0;
}

// What the step needs of a grid besides the model constants.
struct Grid2D {
  int nx, ny, px, bcx, bcy, fold;
  long long plane;
  __half* uring;
  const unsigned char* solid;
  __device__ __forceinline__ explicit Grid2D(const Model& m)
      : nx(m.nx), ny(m.ny), px(m.px), bcx(m.bc[0]), bcy(m.bc[1]), fold(m.fold), plane(m.plane),
        uring(m.uring), solid(m.solid) {}
};

// Central Hermite MRT of the flow populations (2D; the collision of the
// paper's flow solver, read as the C ABI documents for LBPF_COLL_CHM).
// d: pre-collision deviations f - w; drho, rho, (mx, my): their zeroth and
// first moments; (vx, vy) = u*; F the force; wf, wb, wh the rates.  The
// moments are formed from the deviations with the weights' own moments
// (1, 0, 0, 1/3, 1/3, 0, 0, 0, 1/9) taken out analytically, so that FP32
// keeps the small quantities: raw moments e_pq -> central Hermite moments
// about u* -> relaxation by order -> raw moments -> populations through the
// inverse of the D2Q9 raw-moment matrix.  out: post-collision deviations.
template <typename N>
__device__ __forceinline__ void chm_post_2d(const N (&d)[9], N drho, N rho, N mx, N my, N vx, N vy,
                                            N Fx, N Fy, const Coef<N>& c, N (&out)[9]) {
  using S = typename Lanes<N>::S;
  const N t3 = splat<N>(S(1.0 / 3.0)), t9 = splat<N>(S(1.0 / 9.0)), two = splat<N>(S(2));
  const N t23 = splat<N>(S(2) * S(1.0 / 3.0)), half = splat<N>(S(0.5)), quarter = splat<N>(S(0.25));
  // a sum of products: add(p, q, s) = s + p q, sub(p, q, s) = s - p q
  auto add = [](N p, N q, N s) { return fma_r(p, q, s); };
  auto sub = [](N p, N q, N s) { return fma_r(neg_r(p), q, s); };
  // raw moments of the deviations
  const N e00 = drho, e10 = mx, e01 = my;
  const N dd = add_r(add_r(d[5], d[6]), add_r(d[7], d[8]));
  const N e20 = add_r(add_r(d[1], d[3]), dd), e02 = add_r(add_r(d[2], d[4]), dd);
  const N e11 = add_r(sub_r(d[5], d[6]), sub_r(d[7], d[8]));
  const N e21 = sub_r(add_r(d[5], d[6]), add_r(d[7], d[8]));
  const N e12 = sub_r(sub_r(d[5], d[6]), sub_r(d[7], d[8]));
  const N e22 = dd, t3e = prod_r(t3, e00, c.mzero);
  const N vxx = mul_r(vx, vx), vyy = mul_r(vy, vy), vxy = mul_r(vx, vy);
  const N vx2 = mul_r(two, vx), vy2 = mul_r(two, vy), vxy2 = mul_r(two, vxy);
  const N vxy4 = mul_r(splat<N>(S(4)), vxy), vxxy = mul_r(vxx, vy), vxyy = mul_r(vx, vyy);
  const N vxy2y = mul_r(vxy2, vy), vxy2x = mul_r(vxy2, vx), vxxyy = mul_r(vxx, vyy);
  // central Hermite moments about (vx, vy)
  const N h1 = sub(vx, rho, e10), h2 = sub(vy, rho, e01);
  const N hxx = add(vxx, rho, sub(vx2, e10, sub_r(e20, t3e)));
  const N hyy = add(vyy, rho, sub(vy2, e01, sub_r(e02, t3e)));
  const N hxy = add(vxy, rho, sub(vy, e10, sub(vx, e01, e11)));
  const N hxxy = add(mul_r(t3, vy), e00,
                     sub(t3, e01,
                         sub(vxxy, rho,
                             add(vxy2, e10, sub(vy, e20, add(vxx, e01, sub(vx2, e11, e21)))))));
  const N hxyy = add(mul_r(t3, vx), e00,
                     sub(t3, e10,
                         sub(vxyy, rho,
                             add(vxy2, e01, sub(vx, e02, add(vyy, e10, sub(vy2, e11, e12)))))));
  N hxxyy = sub(vy2, e21, sub(vx2, e12, e22));
  hxxyy = add(vxy4, e11, add(vyy, e20, add(vxx, e02, hxxyy)));
  hxxyy = add(vxxyy, rho, sub(vxy2x, e01, sub(vxy2y, e10, hxxyy)));
  hxxyy = add(t23, fma_r(vx, e10, mul_r(vy, e01)), sub(t3, add_r(e20, e02), hxxyy));
  hxxyy = add(t9, e00, sub(mul_r(t3, fma_r(vx, vx, vyy)), e00, hxxyy));
  // relaxation towards rho and zeros; the force in the first order
  const N one = splat<N>(S(1)), kf = c.keep_f, gf = fma_r(splat<N>(S(-0.5)), c.omega_f, one);
  const N kh = sub_r(one, c.chm_wh), kb = sub_r(one, c.chm_wb);
  const N h1s = fma_r(kf, h1, mul_r(gf, Fx)), h2s = fma_r(gf, Fy, mul_r(kf, h2));
  const N sum = add_r(hxx, hyy), dv = mul_r(kf, sub_r(hxx, hyy));
  const N hxxs = mul_r(half, fma_r(kb, sum, dv)), hyys = mul_r(half, fma_r(kb, sum, neg_r(dv)));
  const N hxys = mul_r(kf, hxy);
  // central (raw) moments after collision, then raw moments of the deviations
  const N k20 = add(t3, rho, hxxs), k02 = add(t3, rho, hyys);
  const N k21 = fma_r(t3, h2s, mul_r(kh, hxxy)), k12 = fma_r(t3, h1s, mul_r(kh, hxyy));
  const N f10 = add(vx, rho, h1s), f01 = add(vy, rho, h2s);
  const N f20 = add(vxx, rho, add(vx2, h1s, add_r(hxxs, t3e)));
  const N f02 = add(vyy, rho, add(vy2, h2s, add_r(hyys, t3e)));
  const N f11 = add(vxy, rho, add(vy, h1s, add(vx, h2s, hxys)));
  const N f21 =
      add(vxxy, rho, add(vxy2, h1s, add(vy, k20, add(vxx, h2s, add(vx2, hxys, k21)))));
  const N f12 =
      add(vxyy, rho, add(vxy2, h2s, add(vx, k02, add(vyy, h1s, add(vy2, hxys, k12)))));
  N f22 = fma_r(kh, hxxyy, mul_r(t3, add_r(hxxs, hyys)));
  f22 = add(vy2, k21, add(vx2, k12, add(t9, e00, f22)));
  f22 = add(vxy4, hxys, add(vyy, k20, add(vxx, k02, f22)));
  f22 = add(vxxyy, rho, add(vxy2x, h2s, add(vxy2y, h1s, f22)));
  // populations (D2Q9 order: rest, +x, +y, -x, -y, ++, -+, --, +-)
  out[0] = add_r(sub_r(sub_r(e00, f20), f02), f22);
  out[1] = mul_r(half, sub_r(sub_r(add_r(f10, f20), f12), f22));
  out[3] = mul_r(half, sub_r(add_r(sub_r(f20, f10), f12), f22));
  out[2] = mul_r(half, sub_r(sub_r(add_r(f01, f02), f21), f22));
  out[4] = mul_r(half, sub_r(add_r(sub_r(f02, f01), f21), f22));
  out[5] = mul_r(quarter, add_r(add_r(add_r(f11, f21), f12), f22));
  out[6] = mul_r(quarter, add_r(sub_r(sub_r(f21, f11), f12), f22));
  out[7] = mul_r(quarter, add_r(sub_r(sub_r(f11, f21), f12), f22));
  out[8] = mul_r(quarter, add_r(sub_r(f12, add_r(f11, f21)), f22));
}

// What the collisions of one node (or of a thread's two nodes, N = float2)
// need, so that each direction costs a few FMAs:
//   f*: (1 - w_f) d + w_f w [E0 + cu (E1 + E2 cu)] + guo w [cF (3 + 9 cu) - 3 u*.F]
//       (Eq. 4, 5, 8, 9 with c_s^2 = 1/3, d = f - w)
//   g*: (1 - w_U) d + w (K0 + K1 cu)            (Eqs. 13-16, d = g - w U_ref)
//   h*: (1 - w_phi) d + w (H0 - c.H)            (Eqs. 19-21, d = h + w)
// The order and rounding of every operation is written out (fma_r, mul_r,
// add_r), so that one and two nodes per thread give the same bits.
template <typename N>
struct Node2D {
  using S = typename Lanes<N>::S;
  N U;                                 // Eq. 17
  N usx, usy, Fx, Fy, E0, E1, E2, G0;  // flow (with the central Hermite MRT unused)
  N keep_U, K0, K1, keep_phi, H0, Hx, Hy, inv_a2, keep_old;
  N us_s, us_d, F_s, F_d, H_s, H_d;    // sums and differences of the two components
};

// Moments, gradient, anisotropy and the coefficients above (Eqs. 3-23) of a
// node with population deviations f, g, phi + 1 = dphi (dphi_prev one step
// earlier), the g reference Rg and the eight neighbours' phi + 1.  Returns the
// finite_mark of phi, U and rho.
template <typename N, bool FLOW, bool CHM>
__device__ __forceinline__ N node_2d(const Coef<N>& c, int fold, const N (&f)[9], const N (&g)[9], N dphi,
                                        N dphi_prev, N Rg, N pE, N pW, N pN, N pS, N pNE, N pNW,
                                        N pSE, N pSW, Node2D<N>& o, N (&fchm)[9]) {
  using S = typename Lanes<N>::S;
  const N one = splat<N>(S(1)), half = splat<N>(S(0.5));
  // ---- local moments (Eqs. 11, 12, 17, 22) ----------------------------------
  const N phi = sub_r(dphi, one);
  N dU = g[0];
#pragma unroll
  for (int a = 1; a < 9; ++a) dU = add_r(dU, g[a]);
  // g deviations are taken from w_a Rg; the collision (Eqs. 13-16) is linear
  // in them, so any per-node Rg gives the same populations
  const N U = o.U = add_r(Rg, dU);
  N drho = splat<N>(S(0)), mx = drho, my = drho;
  if (FLOW) {
    drho = f[0];
#pragma unroll
    for (int a = 1; a < 9; ++a) drho = add_r(drho, f[a]);
    mx = add_r(add_r(sub_r(f[1], f[3]), sub_r(f[5], f[6])), sub_r(f[8], f[7]));
    my = sub_r(add_r(sub_r(f[2], f[4]), add_r(f[5], f[6])), add_r(f[7], f[8]));
  }
  const N rho = add_r(one, drho);
  const N mark = finite_mark(phi, U, rho);
  const N ph = clamp1(phi);
  const N mask = mul_r(half, sub_r(one, ph));  // (1 - phi)/2 of Eq. 7 and q(phi) of Eq. 18
  o.usx = o.usy = o.Fx = o.Fy = splat<N>(S(0));
  if (FLOW) {
    // Eq. 6: F = b - K u, K = h tau_f (1+phi)^2 (1-phi) / (4 W0^2); the Guo
    // half-force velocity u = (m + F/2)/rho solved in closed form.
    const N ph1 = add_r(one, ph);
    const N K = mul_r(mul_r(mul_r(c.kdrag, ph1), ph1), sub_r(one, ph));
    const N inv = rcp_r(fma_r(half, K, rho));
    const N ux = mul_r(fma_r(half, c.body[0], mx), inv);
    const N uy = mul_r(fma_r(half, c.body[1], my), inv);
    o.Fx = fma_r(neg_r(K), ux, c.body[0]);
    o.Fy = fma_r(neg_r(K), uy, c.body[1]);
    o.usx = mul_r(mask, ux);  // u* (Eq. 7)
    o.usy = mul_r(mask, uy);
  }
  if constexpr (FLOW && CHM)
    chm_post_2d<N>(f, drho, rho, mx, my, o.usx, o.usy, o.Fx, o.Fy, c, fchm);
  const N omega_U = rcp_r(fma_r(c.tauU_slope, mask, half));  // Eq. 18
  const N dphidt = sub_r(dphi, dphi_prev);

  // ---- gradient, anisotropy, phase-field coefficients (Eqs. 3, 20, 21, 23) --
  // grad = 3 sum_a w_a c_a phi(x + c_a) over D2Q9
  const N third = splat<N>(S(1.0 / 3.0)), twelfth = splat<N>(S(1.0 / 12.0));
  const N gx = fma_r(third, sub_r(pE, pW),
                     mul_r(twelfth, sub_r(add_r(pNE, pSE), add_r(pNW, pSW))));
  const N gy = fma_r(third, sub_r(pN, pS),
                     mul_r(twelfth, sub_r(add_r(pNE, pNW), add_r(pSE, pSW))));
  N as, Nx, Ny;
  aniso_2d<N>(c, fold, gx, gy, as, Nx, Ny);
  const N a2 = mul_r(as, as);
  o.inv_a2 = rcp_r(a2);
  const N tpc = c.tpc;
  const N omega_phi = rcp_r(fma_r(a2, tpc, half));  // Eq. 23
  const N pp = mul_r(phi, phi);
  const N phi2m = sub_r(one, pp);
  // Eq. 20
  const N Qs = mul_r(fma_r(mul_r(mul_r(c.lambda, U), phi2m), phi2m,
                           fma_r(neg_r(pp), phi, phi)),
                     c.inv_tau0);
  if (FLOW && !CHM) {
    const N uu = fma_r(o.usx, o.usx, mul_r(o.usy, o.usy));
    const N uF = fma_r(o.usx, o.Fx, mul_r(o.usy, o.Fy));
    o.E0 = mul_r(c.omega_f, fma_r(neg_r(mul_r(splat<N>(S(1.5)), rho)), uu, drho));
    o.E1 = mul_r(c.wf3, rho);
    o.E2 = mul_r(c.wf45, rho);
    o.G0 = mul_r(splat<N>(S(-3)), uF);
    o.F_s = add_r(o.Fx, o.Fy);
    o.F_d = sub_r(o.Fx, o.Fy);
  }
  o.us_s = add_r(o.usx, o.usy);
  o.us_d = sub_r(o.usx, o.usy);
  o.keep_U = sub_r(one, omega_U);
  o.K0 = fma_r(omega_U, dU, neg_r(dphidt));
  o.K1 = mul_r(mul_r(splat<N>(S(3)), omega_U), U);
  o.keep_phi = sub_r(one, omega_phi);
  o.H0 = fma_r(omega_phi, dphi, Qs);
  const N wt = mul_r(omega_phi, tpc);
  o.Hx = mul_r(wt, Nx);
  o.Hy = mul_r(wt, Ny);
  o.H_s = add_r(o.Hx, o.Hy);
  o.H_d = sub_r(o.Hx, o.Hy);
  // Eq. 19: h_new = h* / a_s^2 + (1 - 1/a_s^2) h_old
  o.keep_old = sub_r(one, o.inv_a2);
  return mark;
}

// c_a . v from the components and their sum and difference (a a constant
// after unrolling; not for the rest direction)
template <typename N>
__device__ __forceinline__ N dir_dot(int a, N x, N y, N s, N d) {
  switch (a) {
    case 1: return x;
    case 2: return y;
    case 3: return neg_r(x);
    case 4: return neg_r(y);
    case 5: return s;
    case 6: return neg_r(d);
    case 7: return neg_r(s);
    default: return d;
  }
}

// Post-collision deviations of direction a at the node: f* (Eq. 4), g* (Eq.
// 13) and, before Eq. 19's division by a_s^2, h*.
template <typename N>
__device__ __forceinline__ N post_f_2d(const Coef<N>& c, const Node2D<N>& n, int a, N f) {
  using S = typename Lanes<N>::S;
  const N w = splat<N>(d2_w<S>(a));
  N feq = n.E0, gt = n.G0;
  if (a > 0) {
    const N cu = dir_dot(a, n.usx, n.usy, n.us_s, n.us_d);
    const N cF = dir_dot(a, n.Fx, n.Fy, n.F_s, n.F_d);
    feq = fma_r(cu, fma_r(n.E2, cu, n.E1), n.E0);
    gt = fma_r(cF, fma_r(splat<N>(S(9)), cu, splat<N>(S(3))), n.G0);
  }
  return fma_r(c.keep_f, f, mul_r(w, add_r(feq, prod_r(c.guo, gt, c.mzero))));
}
template <typename N>
__device__ __forceinline__ N post_g_2d(const Node2D<N>& n, int a, N g) {
  using S = typename Lanes<N>::S;
  const N w = splat<N>(d2_w<S>(a));
  N e = n.K0;
  if (a > 0) e = fma_r(n.K1, dir_dot(a, n.usx, n.usy, n.us_s, n.us_d), n.K0);
  return fma_r(n.keep_U, g, mul_r(w, e));
}
template <typename N>
__device__ __forceinline__ N post_h_2d(const Node2D<N>& n, int a, N h) {
  using S = typename Lanes<N>::S;
  const N w = splat<N>(d2_w<S>(a));
  N e = n.H0;
  if (a > 0) e = sub_r(n.H0, dir_dot(a, n.Hx, n.Hy, n.H_s, n.H_d));
  return fma_r(n.keep_phi, h, mul_r(w, e));
}
// Eq. 19 at the destination, whose old value is hold
template <typename N>
__device__ __forceinline__ N arrive_h_2d(const Node2D<N>& n, N hp, N hold) {
  return fma_r(n.inv_a2, hp, mul_r(n.keep_old, hold));
}

// Collide and push a thread's one or two nodes (N = float2: the second DY rows
// below the first).
//   own(q): stored deviation q of the node(s) (f, then g)
//   pc: phi + 1 of the first node in the tile (row pitch PROW); dphi,
//     dphi_prev: phi + 1 of the node(s) now and one step earlier
//   hold(a, dy, dx), uref(dy, dx): h_a and the encoding reference of g (UREL) at
//     that offset from the node(s)
//   sm[k]: bit a set where node k's neighbour in direction a (0: the node
//     itself) is solid, mapped like a gradient neighbour (MASK)
//   (x, y): the first node; tb: the tile's origin in array 0 of the
//     destination buffer (the same for the whole CTA, so that every array's
//     address is one uniform base plus the thread's offset); o0, o1: offsets
//     of the node(s) from it, in bytes
// EDGE = false: every destination is an ordinary node (the tile lies at least
// one node away from every domain edge and holds or borders no solid node), so
// the push needs no boundary logic.  EDGE = true: each destination goes through
// the boundary rules; nodes outside the domain (of a partial tile) and solid
// nodes push nothing.  MASK: the code for solid nodes is compiled in.  CHM: the
// flow collides by the central Hermite MRT.
template <typename T, typename N, bool FLOW, bool CHM, bool MASK, bool EDGE, bool UREL, int PROW,
          int DY, typename Own, typename Hold, typename Uref>
__device__ __forceinline__ void collide_push_2d(
    const Grid2D& gr, const Coef<N>& c, int x, int y, const Own& own, const N (&h)[9], N dphi,
    N dphi_prev, const typename Lanes<N>::S* pc, const Hold& hold, const Uref& uref,
    const unsigned (&sm)[Lanes<N>::V], N Rg, T* __restrict__ tb, unsigned o0, unsigned o1,
    unsigned* __restrict__ err, N& Unew) {
  using S = typename Lanes<N>::S;
  constexpr int V = Lanes<N>::V, QF = FLOW ? 9 : 0;
  const int nx = gr.nx, ny = gr.ny, px = gr.px;
  const long long P = gr.plane;
  N pn[9];  // the neighbours' phi + 1
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    const int off = D2_CY[a] * PROW + D2_CX[a];
    set_lane(pn[a], 0, pc[off]);
    if (V == 2) set_lane(pn[a], 1, pc[off + DY * PROW]);
  }
  if (MASK && EDGE) {
    // a solid neighbour counts as the first fluid node among (x + c_x, y),
    // (x, y + c_y) and (x, y): zero normal derivative at walls and obstacles
    const N centre = dphi;
#pragma unroll
    for (int k = 0; k < V; ++k) {
      if (sm[k] == 0) continue;
      auto is = [&](int a) { return (sm[k] >> a & 1u) != 0; };
      // the diagonals first: they look at the axis values as they are
#pragma unroll
      for (int a = 8; a > 0; --a) {
        if (!is(a)) continue;
        S v = lane(centre, k);
        if (a > 4) {
          const int ax = D2_CX[a] > 0 ? 1 : 3, ay = D2_CY[a] > 0 ? 2 : 4;
          if (!is(ax)) v = lane(pn[ax], k);
          else if (!is(ay)) v = lane(pn[ay], k);
        }
        set_lane(pn[a], k, v);
      }
    }
  }
  N f[9], g[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    if (FLOW) f[a] = own(a);
    g[a] = own(QF + a);
  }
  Node2D<N> nd;
  N fchm[9];
  const N mark = node_2d<N, FLOW, CHM>(c, gr.fold, f, g, dphi, dphi_prev, Rg, pn[1], pn[3], pn[2],
                                       pn[4], pn[5], pn[6], pn[8], pn[7], nd, fchm);
  if (!all_finite(mark)) {
    bool bad = !(MASK && EDGE);
    if (MASK && EDGE)  // whatever a solid node holds takes no part in the step
#pragma unroll
      for (int k = 0; k < V; ++k) bad = bad || (!(sm[k] & 1u) && !(lane(mark, k) == S(0)));
    if (bad) atomicOr(err, 1u);
  }
  Unew = nd.U;

  if constexpr (!EDGE) {
    auto put = [&](int q, int off, N v) {
      char* b = reinterpret_cast<char*>(tb + (q * P + off));
      Pop<T>::st(reinterpret_cast<T*>(b + o0), lane(v, 0));
      if (V == 2) Pop<T>::st(reinterpret_cast<T*>(b + o1), lane(v, 1));
    };
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int off = D2_CY[a] * px + D2_CX[a];
      if (FLOW) put(a, off, CHM ? fchm[a] : post_f_2d<N>(c, nd, a, f[a]));
      N gp = post_g_2d<N>(nd, a, g[a]);
      if (UREL) gp = fma_r(splat<N>(-d2_w<S>(a)), sub_r(uref(D2_CY[a], D2_CX[a]), Rg), gp);
      put(QF + a, off, gp);
      put(QF + 9 + a, off,
          arrive_h_2d<N>(nd, post_h_2d<N>(nd, a, h[a]), hold(a, D2_CY[a], D2_CX[a])));
    }
    return;
  } else {
    // Element steps to the neighbouring columns and rows (across a periodic
    // edge to the far side) and what lies there: a wall (the population comes
    // back to its node reversed, half-way bounce-back) or, in x, the inflow
    // or outflow ghost (nothing to push).
    const int bcx = gr.bcx, bcy = gr.bcy;
    const bool x_lo = x == 0, x_hi = x == nx - 1;
    const int sxm = x_lo ? nx - 1 : -1, sxp = x_hi ? 1 - nx : 1;
    const bool wxm = x_lo && bcx == BC_WALL, wxp = x_hi && bcx == BC_WALL;
    const bool gxm = x_lo && bcx == BC_INOUT, gxp = x_hi && bcx == BC_INOUT;
    const int wrap_y = (ny - 1) * px;
    int sym[V], syp[V];
    bool wym[V], wyp[V], on[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const int yk = y + k * DY;
      on[k] = x < nx && yk < ny;
      if (MASK) on[k] = on[k] && !(sm[k] & 1u);
      sym[k] = yk == 0 ? wrap_y : -px;
      syp[k] = yk == ny - 1 ? -wrap_y : px;
      wym[k] = yk == 0 && bcy == BC_WALL;
      wyp[k] = yk == ny - 1 && bcy == BC_WALL;
    }
    T* const n0 = reinterpret_cast<T*>(reinterpret_cast<char*>(tb) + o0);
    T* const n1 = reinterpret_cast<T*>(reinterpret_cast<char*>(tb) + o1);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const int cx = D2_CX[a], cy = D2_CY[a], b = D2_OPP[a];
      N fp = splat<N>(S(0));
      if (FLOW) fp = CHM ? fchm[a] : post_f_2d<N>(c, nd, a, f[a]);
      const N gp = post_g_2d<N>(nd, a, g[a]);
      const N hp = post_h_2d<N>(nd, a, h[a]);
      const N w = splat<N>(d2_w<S>(a));
      const N hfar = arrive_h_2d<N>(nd, hp, hold(a, cy, cx));    // at the destination
      const N hown = arrive_h_2d<N>(nd, hp, h[b]);               // reversed at the node
      N gfar = gp, gown = gp;
      if (UREL) {
        gfar = fma_r(neg_r(w), sub_r(uref(cy, cx), Rg), gp);
        gown = fma_r(neg_r(w), sub_r(uref(0, 0), Rg), gp);
      }
#pragma unroll
      for (int k = 0; k < V; ++k) {
        T* const node = k ? n1 : n0;
        bool back = (cy < 0 && wym[k]) || (cy > 0 && wyp[k]) || (cx < 0 && wxm) || (cx > 0 && wxp);
        const bool ghost = !back && ((cx < 0 && gxm) || (cx > 0 && gxp));
        const int step = (cx < 0 ? sxm : (cx > 0 ? sxp : 0)) +
                         (cy < 0 ? sym[k] : (cy > 0 ? syp[k] : 0));
        if (MASK) back = back || (!ghost && (sm[k] >> a & 1u));  // obstacle
        if (on[k] && !ghost) {
          T* const p = back ? node + b * P : node + (a * P + step);
          if (FLOW) Pop<T>::st(p, lane(fp, k));
          Pop<T>::st(p + QF * P, back ? lane(gown, k) : lane(gfar, k));
          Pop<T>::st(p + (QF + 9) * P, back ? lane(hown, k) : lane(hfar, k));
        }
      }
      if (cx != 0 && bcx == BC_INOUT) {
        if (cx < 0 && x_hi) {
          // outflow ghost x = nx repeats this column: its post-collision value
          // arrives at (nx - 1, y + c_y)
          const N hout = arrive_h_2d<N>(nd, hp, hold(a, cy, 0));
          N gout = gp;
          if (UREL) gout = fma_r(neg_r(w), sub_r(uref(cy, 0), Rg), gp);
#pragma unroll
          for (int k = 0; k < V; ++k) {
            if (!on[k] || (cy < 0 && wym[k]) || (cy > 0 && wyp[k])) continue;
            T* const p = (k ? n1 : n0) + (a * P + (cy < 0 ? sym[k] : (cy > 0 ? syp[k] : 0)));
            if (FLOW) Pop<T>::st(p, lane(fp, k));
            Pop<T>::st(p + QF * P, lane(gout, k));
            Pop<T>::st(p + (QF + 9) * P, lane(hout, k));
          }
        }
        if (cx > 0 && x_lo) {
          // inflow ghost x = -1: equilibrium at rho = 1, u = u_in e_x, U = U_in,
          // phi = -1 (a_s = 1; its h deviation is 0), unless behind a wall
          const S uin = lane(c.u_in, 0), Uin = lane(c.U_in, 0), ws = d2_w<S>(a), gu = FLOW ? uin : S(0);
          const S fin = ws * (S(3) * uin + S(4.5) * uin * uin - S(1.5) * uin * uin);
#pragma unroll
          for (int k = 0; k < V; ++k) {
            if (!on[k] || (cy > 0 && wym[k]) || (cy < 0 && wyp[k])) continue;
            T* const p = (k ? n1 : n0) + a * P;
            const S R0 = lane(Rg, k);
            S gin = ws * ((Uin - R0) + Uin * S(3) * gu);
            if (UREL) gin = fma_r(-ws, lane(uref(0, 0), k) - R0, gin);
            if (FLOW) Pop<T>::st(p, fin);
            Pop<T>::st(p + QF * P, gin);
            Pop<T>::st(p + (QF + 9) * P, S(0));
          }
        }
      }
    }
  }
}

}  // namespace lbk
