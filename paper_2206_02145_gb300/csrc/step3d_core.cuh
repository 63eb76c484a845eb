// Per-node part of the 3D coupled step, shared by the 3D step kernels:
// D3Q19 flow f (Eqs. 4-12), D3Q7 solute g (Eqs. 13-18) and D3Q7 phase field
// h (Eqs. 19-23, cubic anisotropy of Eq. 3), push streaming.  The caller has
// the node's own population deviations, phi + 1 and the h deviations around
// the node (one node in x, y and z) in shared memory.  As in 2D every
// operation of the BGK collision, the solute and the phase field is written with its
// rounding (the central Hermite MRT and the inflow's constants are plain
// expressions, to FP32 and FP64 accuracy); a thread holds one node (two, on
// the packed FP32 instructions, measured slower: 831 against 690 us per step of
// 256^3 in FP16, the code of both paths no longer fits the instruction cache).
#pragma once

#include "lbpf_device.cuh"

namespace lbk {

// ---- central Hermite MRT of the D3Q19 flow lattice (Sec. 2.2 after Eq. 9) ----
// The nineteen moments are the products H_i(X) H_j(Y) H_k(Z) (H_0 = 1,
// H_1 = X, H_2 = X^2 - 1/3; i, j, k <= 2, at most two non-zero) about u*.
// Every one involves at most two axes, and the weights' moments over an axis
// pair are those of D2Q9 (1, 1/3, 1/3, 1/9), so each pair (p, q) takes the
// 2D transform of its nine raw moments; the pairs share the moments of one
// axis.  Raw moments of the stored deviations -> central Hermite moments ->
// relaxation by order -> raw moments -> populations through the inverse of
// the D3Q19 raw-moment matrix (rest, faces and each pair's four edges in
// closed form).

// central Hermite moments XY, X^2 Y, X Y^2, X^2 Y^2 of the pair (p, q) from
// the raw deviation moments e_ij of p^i q^j
template <typename R>
struct ChmPair {
  R hpq, hppq, hpqq, hppqq;
};

template <typename R>
__device__ __forceinline__ ChmPair<R> chm_pair_central(R e00, R e10, R e01, R e20, R e02, R e11,
                                                      R e21, R e12, R e22, R vp, R vq, R rho) {
  const R t3 = R(1.0 / 3.0), t9 = R(1.0 / 9.0);
  const R vpp = vp * vp, vqq = vq * vq, vpq = vp * vq;
  ChmPair<R> h;
  h.hpq = e11 - vp * e01 - vq * e10 + vpq * rho;
  h.hppq = e21 - R(2) * vp * e11 + vpp * e01 - vq * e20 + R(2) * vpq * e10 - vpp * vq * rho -
           t3 * e01 + t3 * vq * e00;
  h.hpqq = e12 - R(2) * vq * e11 + vqq * e10 - vp * e02 + R(2) * vpq * e01 - vp * vqq * rho -
           t3 * e10 + t3 * vp * e00;
  h.hppqq = e22 - R(2) * vp * e12 - R(2) * vq * e21 + vpp * e02 + vqq * e20 + R(4) * vpq * e11 -
            R(2) * vpq * vq * e10 - R(2) * vpq * vp * e01 + vpp * vqq * rho -
            t3 * (e20 + e02) + R(2) * t3 * (vp * e10 + vq * e01) - t3 * (vpp + vqq) * e00 +
            t9 * e00;
  return h;
}

// raw deviation moments f11, f21 (p^2 q), f12 (p q^2), f22 of the pair after
// collision, from its relaxed central Hermite moments (s: first and
// diagonal second order of p and q, m: the pair's own)
template <typename R>
__device__ __forceinline__ void chm_pair_raw(const ChmPair<R>& m, R hp, R hq, R hpp, R hqq, R vp,
                                             R vq, R rho, R e00, R& f11, R& f21, R& f12,
                                             R& f22) {
  const R t3 = R(1.0 / 3.0), t9 = R(1.0 / 9.0);
  const R vpp = vp * vp, vqq = vq * vq, vpq = vp * vq;
  const R kpp = hpp + t3 * rho, kqq = hqq + t3 * rho;
  const R k21 = m.hppq + t3 * hq, k12 = m.hpqq + t3 * hp;
  f11 = m.hpq + vp * hq + vq * hp + vpq * rho;
  f21 = k21 + R(2) * vp * m.hpq + vpp * hq + vq * kpp + R(2) * vpq * hp + vpp * vq * rho;
  f12 = k12 + R(2) * vq * m.hpq + vqq * hp + vp * kqq + R(2) * vpq * hq + vp * vqq * rho;
  f22 = m.hppqq + t3 * (hpp + hqq) + t9 * e00 + R(2) * vp * k12 + R(2) * vq * k21 + vpp * kqq +
        vqq * kpp + R(4) * vpq * m.hpq + R(2) * vpq * vq * hp + R(2) * vpq * vp * hq +
        vpp * vqq * rho;
}

// d: the node's f deviations (D3Q19 order: rest, +x, -x, +y, -y, +z, -z, then
// the pairs xy, xz, yz with four edges each, (+,+), (-,-), (+,-), (-,+));
// mo: their first moments; v: u*; F: the force.  out: post-collision
// deviations.
template <typename R>
__device__ __forceinline__ void chm_post_3d(const R (&d)[19], R drho, R rho, const R (&mo)[3],
                                            const R (&v)[3], const R (&F)[3], R wf, R wb, R wh,
                                            R (&out)[19]) {
  const R t3 = R(1.0 / 3.0);
  const R e00 = drho;
  // raw moments of each pair: p^2 q^2, p q, p^2 q, p q^2
  R e22[3], e11[3], e21[3], e12[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int b = 7 + 4 * k;
    e22[k] = (d[b] + d[b + 1]) + (d[b + 2] + d[b + 3]);
    e11[k] = (d[b] + d[b + 1]) - (d[b + 2] + d[b + 3]);
    e21[k] = (d[b] - d[b + 1]) - (d[b + 2] - d[b + 3]);
    e12[k] = (d[b] - d[b + 1]) + (d[b + 2] - d[b + 3]);
  }
  // pairs: 0 = (x, y), 1 = (x, z), 2 = (y, z)
  const R e2[3] = {(d[1] + d[2]) + (e22[0] + e22[1]), (d[3] + d[4]) + (e22[0] + e22[2]),
                   (d[5] + d[6]) + (e22[1] + e22[2])};
  // central Hermite moments, first and diagonal second order
  R h1[3], h2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    h1[a] = mo[a] - v[a] * rho;
    h2[a] = e2[a] - t3 * e00 - R(2) * v[a] * mo[a] + v[a] * v[a] * rho;
  }
  constexpr int PP[3] = {0, 0, 1}, QQ[3] = {1, 2, 2};
  ChmPair<R> hp[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int p = PP[k], q = QQ[k];
    hp[k] = chm_pair_central<R>(e00, mo[p], mo[q], e2[p], e2[q], e11[k], e21[k], e12[k], e22[k],
                                v[p], v[q], rho);
  }
  // relaxation towards rho and zeros; the force in the first order; the
  // trace of the second order at wb, its deviatoric part and the mixed
  // moments at wf, third and fourth order at wh
  const R kf = R(1) - wf, gf = R(1) - R(0.5) * wf, kh = R(1) - wh;
  const R mean = (h2[0] + h2[1] + h2[2]) * t3;
  const R kb = (R(1) - wb) * mean;
  R s1[3], s2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    s1[a] = kf * h1[a] + gf * F[a];
    s2[a] = kb + kf * (h2[a] - mean);
  }
  R f11[3], f21[3], f12[3], f22[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int p = PP[k], q = QQ[k];
    ChmPair<R> m;
    m.hpq = kf * hp[k].hpq;
    m.hppq = kh * hp[k].hppq;
    m.hpqq = kh * hp[k].hpqq;
    m.hppqq = kh * hp[k].hppqq;
    chm_pair_raw<R>(m, s1[p], s1[q], s2[p], s2[q], v[p], v[q], rho, e00, f11[k], f21[k], f12[k],
                    f22[k]);
  }
  // raw moments of one axis after collision
  R f1[3], f2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f1[a] = s1[a] + v[a] * rho;
    f2[a] = s2[a] + t3 * e00 + R(2) * v[a] * s1[a] + v[a] * v[a] * rho;
  }
  // populations: rest, faces, edges
  out[0] = e00 - (f2[0] + f2[1] + f2[2]) + (f22[0] + f22[1] + f22[2]);
  {
    // faces of x: x y^2 and x z^2 are the p q^2 of pairs xy and xz; of y:
    // x^2 y (pair xy, p^2 q) and y z^2 (pair yz, p q^2); of z: x^2 z and y^2 z
    const R sx = f2[0] - f22[0] - f22[1], ax = f1[0] - f12[0] - f12[1];
    const R sy = f2[1] - f22[0] - f22[2], ay = f1[1] - f21[0] - f12[2];
    const R sz = f2[2] - f22[1] - f22[2], az = f1[2] - f21[1] - f21[2];
    out[1] = R(0.5) * (sx + ax);
    out[2] = R(0.5) * (sx - ax);
    out[3] = R(0.5) * (sy + ay);
    out[4] = R(0.5) * (sy - ay);
    out[5] = R(0.5) * (sz + az);
    out[6] = R(0.5) * (sz - az);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int b = 7 + 4 * k;
    out[b] = R(0.25) * (f22[k] + f12[k] + f21[k] + f11[k]);
    out[b + 1] = R(0.25) * (f22[k] - f12[k] - f21[k] + f11[k]);
    out[b + 2] = R(0.25) * (f22[k] + f12[k] - f21[k] - f11[k]);
    out[b + 3] = R(0.25) * (f22[k] - f12[k] + f21[k] - f11[k]);
  }
}

// Solid nodes (3D mask): is the node at (x, y, z), mapped like a gradient
// neighbour (periodic wrap, else nearest node), solid?
__device__ __forceinline__ bool solid_mapped3(const Model& m, int x, int y, int z) {
  x = grad_coord(x, m.nx, m.bc[0]);
  y = grad_coord(y, m.ny, m.bc[1]);
  z = grad_coord(z, m.nz, m.bc[2]);
  return m.solid[(size_t(z) * m.ny + y) * m.px + x] != 0;
}

// What the collisions need, so that each direction costs a few FMAs (see the
// 2D core; D3Q7 has c_s^2 = 1/4).
template <typename N>
struct Node3D {
  N U;
  N us[3], F[3], E0, E1, E2, G0;
  N keep_U, K0, K1, keep_phi, H0, H[3], inv_a2, keep_old;
};

// Moments, gradient, anisotropy and coefficients of a node; pn: the eighteen
// neighbours' phi + 1.  Returns the finite_mark of phi, U and rho.
template <typename N, bool FLOW, bool CHM>
__device__ __forceinline__ N node_3d(const Coef<N>& c, const N (&f)[19], const N (&g)[7], N dphi,
                                     N dphi_prev, N Rg, const N (&pn)[19], bool y_first,
                                     Node3D<N>& o, N (&fchm)[19]) {
  using S = typename Lanes<N>::S;
  const N one = splat<N>(S(1)), half = splat<N>(S(0.5));
  // ---- local moments (Eqs. 11, 12, 17, 22) ----------------------------------
  const N phi = sub_r(dphi, one);
  N dU = g[0];
#pragma unroll
  for (int a = 1; a < 7; ++a) dU = add_r(dU, g[a]);
  // g deviations are taken from w_a Rg; the collision (Eqs. 13-16) is linear
  // in them, so any per-node Rg gives the same populations
  const N U = o.U = add_r(Rg, dU);
  N drho = splat<N>(S(0)), mo[3] = {drho, drho, drho};
  if (FLOW) {
    drho = f[0];
    mo[0] = f[1];
    mo[1] = f[3];
    mo[2] = f[5];
#pragma unroll
    for (int a = 1; a < 19; ++a) {
      drho = add_r(drho, f[a]);
      const int cv[3] = {D3_CX[a], D3_CY[a], D3_CZ[a]};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (cv[d] == 0 || a == 1 + 2 * d) continue;
        mo[d] = cv[d] > 0 ? add_r(mo[d], f[a]) : sub_r(mo[d], f[a]);
      }
    }
  }
  const N rho = add_r(one, drho);
  const N mark = finite_mark(phi, U, rho);
  const N ph = clamp1(phi);
  const N mask = mul_r(half, sub_r(one, ph));  // (1 - phi)/2 of Eq. 7 and q(phi) of Eq. 18
#pragma unroll
  for (int d = 0; d < 3; ++d) o.us[d] = o.F[d] = splat<N>(S(0));
  if (FLOW) {
    const N ph1 = add_r(one, ph);
    const N K = mul_r(mul_r(mul_r(c.kdrag, ph1), ph1), sub_r(one, ph));  // Eq. 6
    const N inv = rcp_r(fma_r(half, K, rho));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const N u = mul_r(fma_r(half, c.body[d], mo[d]), inv);
      o.F[d] = fma_r(neg_r(K), u, c.body[d]);
      o.us[d] = mul_r(mask, u);  // Eq. 7
    }
  }
  if constexpr (FLOW && CHM) {
#pragma unroll
    for (int k = 0; k < Lanes<N>::V; ++k) {
      S d[19], post[19], m3[3], v3[3], F3[3];
#pragma unroll
      for (int a = 0; a < 19; ++a) d[a] = lane(f[a], k);
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        m3[e] = lane(mo[e], k);
        v3[e] = lane(o.us[e], k);
        F3[e] = lane(o.F[e], k);
      }
      chm_post_3d<S>(d, lane(drho, k), lane(rho, k), m3, v3, F3, lane(c.omega_f, 0),
                     lane(c.chm_wb, 0), lane(c.chm_wh, 0), post);
#pragma unroll
      for (int a = 0; a < 19; ++a) set_lane(fchm[a], k, post[a]);
    }
  }
  const N omega_U = rcp_r(fma_r(c.tauU_slope, mask, half));  // Eq. 18
  const N dphidt = sub_r(dphi, dphi_prev);

  // ---- grad = 3 sum_a w_a c_a phi(x + c_a) over D3Q19 ---------------------------
  N gr[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) gr[d] = mul_r(pn[1 + 2 * d], splat<N>(S(1.0 / 6.0)));
#pragma unroll
  for (int a = 2; a < 19; ++a) {
    const N w = splat<N>(a < 7 ? S(1.0 / 6.0) : S(1.0 / 12.0));
    const int cv[3] = {D3_CX[a], D3_CY[a], D3_CZ[a]};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (cv[d] == 0 || a == 1 + 2 * d) continue;
      gr[d] = fma_r(cv[d] > 0 ? pn[a] : neg_r(pn[a]), w, gr[d]);
    }
  }
  N as, Nv[3];
  aniso_3d<N>(c, gr, y_first, as, Nv);
  const N a2 = mul_r(as, as);
  o.inv_a2 = rcp_r(a2);
  const N omega_phi = rcp_r(fma_r(a2, c.tpc, half));  // Eq. 23
  const N pp = mul_r(phi, phi);
  const N phi2m = sub_r(one, pp);
  // Eq. 20
  const N Qs = mul_r(fma_r(mul_r(mul_r(c.lambda, U), phi2m), phi2m, fma_r(neg_r(pp), phi, phi)),
                     c.inv_tau0);
  if (FLOW && !CHM) {
    const N uu = fma_r(o.us[2], o.us[2], fma_r(o.us[0], o.us[0], mul_r(o.us[1], o.us[1])));
    const N uF = fma_r(o.us[2], o.F[2], fma_r(o.us[0], o.F[0], mul_r(o.us[1], o.F[1])));
    o.E0 = mul_r(c.omega_f, fma_r(neg_r(mul_r(splat<N>(S(1.5)), rho)), uu, drho));
    o.E1 = mul_r(c.wf3, rho);
    o.E2 = mul_r(c.wf45, rho);
    o.G0 = mul_r(splat<N>(S(-3)), uF);
  }
  o.keep_U = sub_r(one, omega_U);
  o.K0 = fma_r(omega_U, dU, neg_r(dphidt));
  o.K1 = mul_r(mul_r(splat<N>(S(4)), omega_U), U);
  o.keep_phi = sub_r(one, omega_phi);
  o.H0 = fma_r(omega_phi, dphi, Qs);
  const N wt = mul_r(omega_phi, c.tpc);
#pragma unroll
  for (int d = 0; d < 3; ++d) o.H[d] = mul_r(wt, Nv[d]);
  // Eq. 19: h_new = h* / a_s^2 + (1 - 1/a_s^2) h_old
  o.keep_old = sub_r(one, o.inv_a2);
  return mark;
}

// c_a . v (a a constant after unrolling; not the rest direction)
template <typename N>
__device__ __forceinline__ N dir_dot3(int a, const N (&v)[3]) {
  const int cv[3] = {D3_CX[a], D3_CY[a], D3_CZ[a]};
  N r = v[0];
  bool first = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (cv[d] == 0) continue;
    const N t = cv[d] > 0 ? v[d] : neg_r(v[d]);
    r = first ? t : add_r(r, t);
    first = false;
  }
  return r;
}

// Post-collision deviations of direction a at the node: f* (Eq. 4), g* (Eq.
// 13) and, before Eq. 19's division by a_s^2, h*.
template <typename N>
__device__ __forceinline__ N post_f_3d(const Coef<N>& c, const Node3D<N>& n, int a, N f) {
  using S = typename Lanes<N>::S;
  N feq = n.E0, gt = n.G0;
  if (a > 0) {
    const N cu = dir_dot3(a, n.us), cF = dir_dot3(a, n.F);
    feq = fma_r(cu, fma_r(n.E2, cu, n.E1), n.E0);
    gt = fma_r(cF, fma_r(splat<N>(S(9)), cu, splat<N>(S(3))), n.G0);
  }
  return fma_r(c.keep_f, f,
               mul_r(splat<N>(d3q19_w<S>(a)), add_r(feq, prod_r(c.guo, gt, c.mzero))));
}
template <typename N>
__device__ __forceinline__ N post_g_3d(const Node3D<N>& n, int a, N g) {
  using S = typename Lanes<N>::S;
  N e = n.K0;
  if (a > 0) e = fma_r(n.K1, dir_dot3(a, n.us), n.K0);
  return fma_r(n.keep_U, g, mul_r(splat<N>(d3q7_w<S>(a)), e));
}
template <typename N>
__device__ __forceinline__ N post_h_3d(const Node3D<N>& n, int a, N h) {
  using S = typename Lanes<N>::S;
  N e = n.H0;
  if (a > 0) e = sub_r(n.H0, dir_dot3(a, n.H));
  return fma_r(n.keep_phi, h, mul_r(splat<N>(d3q7_w<S>(a)), e));
}
// Eq. 19 at the destination, whose old value is hold
template <typename N>
__device__ __forceinline__ N arrive_h_3d(const Node3D<N>& n, N hp, N hold) {
  return fma_r(n.inv_a2, hp, mul_r(n.keep_old, hold));
}

// the D3Q19 directions (bit a) whose component d is v
constexpr unsigned dirs3(int d, int v) {
  unsigned m = 0;
  for (int a = 0; a < 19; ++a)
    if ((d == 0 ? D3_CX[a] : (d == 1 ? D3_CY[a] : D3_CZ[a])) == v) m |= 1u << a;
  return m;
}

// What the 3D step needs of a grid besides the model constants.
struct Grid3D {
  int nx, ny, nz, px, slab, bc[3];
  long long plane;
  __device__ __forceinline__ explicit Grid3D(const Model& m)
      : nx(m.nx), ny(m.ny), nz(m.nz), px(m.px), slab(m.ny * m.px),
        bc{m.bc[0], m.bc[1], m.bc[2]}, plane(m.plane) {}
};

// Collide the node (x, y, z) and push its populations.
//   own(q): stored deviation q of the node (f, then g); h: its own h
//   dphi, dphi_prev: phi + 1 now and one step earlier
//   phi(dz, dy, dx), hold(a, dz, dy, dx), uref(dz, dy, dx): phi + 1, h_a and the
//     encoding reference of g (UREL) at that offset from the node
//   sm: bit a set where the D3Q19 neighbour a (0: the node itself) is solid (MASK)
//   tb: the tile's first node in its plane in array 0 of the destination
//     buffer (the same for the whole CTA, so that every array's address is one
//     uniform base plus the thread's offset); o0: the node's byte offset from it
//   y_first: as of aniso_3d
// EDGE = false: interior nodes with no solid node near: all neighbours at fixed
// offsets, no tests.  EDGE = true: any node; one outside the domain (of a partial
// column) or solid pushes nothing.  Which populations go where is then a few
// bit masks over the directions: 25 % of the warps of a 256^3 grid touch a
// boundary in x (871 us per step against 891 with a test per direction).
template <typename T, typename R, bool FLOW, bool CHM, bool MASK, bool EDGE, bool UREL,
          typename Own, typename Phi, typename Hold, typename Uref>
__device__ __forceinline__ void collide_push_3d(
    const Grid3D& gr, const Coef<R>& c, int x, int y, int z, const Own& own, const R (&h)[7],
    R dphi, R dphi_prev, const Phi& phi, const Hold& hold, const Uref& uref, unsigned sm, R Rg,
    T* __restrict__ tb, unsigned o0, bool y_first, unsigned* __restrict__ err, R& Unew) {
  constexpr int QF = FLOW ? 19 : 0;
  const long long P = gr.plane;
  const int px = gr.px, slab = gr.slab;
  R pn[19];  // the neighbours' phi + 1
#pragma unroll
  for (int a = 1; a < 19; ++a) pn[a] = phi(D3_CZ[a], D3_CY[a], D3_CX[a]);
  if (MASK && EDGE && sm != 0) {
    // a solid neighbour counts as the first fluid node among the single-axis
    // steps of its direction (x, y, z order) and the node itself: zero normal
    // derivative at walls and obstacles
    auto is = [&](int a) { return (sm >> a & 1u) != 0; };
#pragma unroll
    for (int a = 18; a > 0; --a) {  // the axis values last: the others look at them
      if (!is(a)) continue;
      R v = dphi;
      if (a > 6) {
        const int ax = D3_CX[a] > 0 ? 1 : 2, ay = D3_CY[a] > 0 ? 3 : 4, az = D3_CZ[a] > 0 ? 5 : 6;
        if (D3_CX[a] != 0 && !is(ax)) v = pn[ax];
        else if (D3_CY[a] != 0 && !is(ay)) v = pn[ay];
        else if (D3_CZ[a] != 0 && !is(az)) v = pn[az];
      }
      pn[a] = v;
    }
  }
  R f[19], g[7];
  if (FLOW) {
#pragma unroll
    for (int a = 0; a < 19; ++a) f[a] = own(a);
  }
#pragma unroll
  for (int a = 0; a < 7; ++a) g[a] = own(QF + a);
  Node3D<R> nd;
  R fchm[19];
  const R mark = node_3d<R, FLOW, CHM>(c, f, g, dphi, dphi_prev, Rg, pn, y_first, nd, fchm);
  // (whatever a solid node holds takes no part in the step)
  if (!all_finite(mark) && !(MASK && EDGE && (sm & 1u))) atomicOr(err, 1u);
  Unew = nd.U;

  if constexpr (!EDGE) {
    auto put = [&](int q, int off, R v) {
      Pop<T>::st(reinterpret_cast<T*>(reinterpret_cast<char*>(tb + (q * P + off)) + o0), v);
    };
#pragma unroll
    for (int a = 0; a < 19; ++a) {
      if (!FLOW && a >= 7) break;
      const int cx = D3_CX[a], cy = D3_CY[a], cz = D3_CZ[a];
      const int off = cz * slab + cy * px + cx;
      if (FLOW) put(a, off, CHM ? fchm[a] : post_f_3d<R>(c, nd, a, f[a]));
      if (a < 7) {
        R gp = post_g_3d<R>(nd, a, g[a]);
        if (UREL) gp = fma_r(-d3q7_w<R>(a), sub_r(uref(cz, cy, cx), Rg), gp);
        put(QF + a, off, gp);
        put(QF + 7 + a, off, arrive_h_3d<R>(nd, post_h_3d<R>(nd, a, h[a]), hold(a, cz, cy, cx)));
      }
    }
  } else {
    // Element steps to the neighbouring columns, rows and planes (across a
    // periodic edge to the far side), and the directions (bit a) in which the
    // node's push meets a wall or solid node (the population comes back to it
    // reversed, half-way bounce-back) or, in x, the inflow or outflow ghost
    // (nothing to push); those whose outflow repeats at the last column and
    // those that arrive from the inflow ghost.
    constexpr unsigned XM = dirs3(0, -1), XP = dirs3(0, 1), YM = dirs3(1, -1), YP = dirs3(1, 1),
                       ZM = dirs3(2, -1), ZP = dirs3(2, 1);
    const int nx = gr.nx, ny = gr.ny, nz = gr.nz;
    const bool x_lo = x == 0, x_hi = x == nx - 1, y_lo = y == 0, y_hi = y == ny - 1;
    const bool z_lo = z == 0, z_hi = z == nz - 1;
    const int sx[3] = {x_lo ? nx - 1 : -1, 0, x_hi ? 1 - nx : 1};
    const int sy[3] = {y_lo ? (ny - 1) * px : -px, 0, y_hi ? -(ny - 1) * px : px};
    const int sz[3] = {z_lo ? (nz - 1) * slab : -slab, 0, z_hi ? -(nz - 1) * slab : slab};
    const bool io = gr.bc[0] == BC_INOUT, wy = gr.bc[1] == BC_WALL, wz = gr.bc[2] == BC_WALL;
    const unsigned x_out = (x_lo ? XM : 0u) | (x_hi ? XP : 0u);
    const unsigned wall = (wy && y_lo ? YM : 0u) | (wy && y_hi ? YP : 0u) |
                          (wz && z_lo ? ZM : 0u) | (wz && z_hi ? ZP : 0u);
    const unsigned behind = (wy && y_lo ? YP : 0u) | (wy && y_hi ? YM : 0u) |
                            (wz && z_lo ? ZP : 0u) | (wz && z_hi ? ZM : 0u);
    unsigned back = wall | (gr.bc[0] == BC_WALL ? x_out : 0u);
    const unsigned ghost = io ? x_out & ~back : 0u;
    if (MASK) back |= sm & ~ghost;  // obstacles
    unsigned go = ~(back | ghost);
    unsigned outf = io && x_hi ? XM & ~wall : 0u;
    unsigned inf = io && x_lo ? XP & ~behind : 0u;
    if (!(x < nx && y < ny) || (MASK && (sm & 1u))) go = back = outf = inf = 0u;
    const unsigned odd = back | outf | inf;
    T* const node = reinterpret_cast<T*>(reinterpret_cast<char*>(tb) + o0);
#pragma unroll
    for (int a = 0; a < 19; ++a) {
      if (!FLOW && a >= 7) break;
      const int cx = D3_CX[a], cy = D3_CY[a], cz = D3_CZ[a], b = D3_OPP[a];
      const bool sc = a < 7;  // also a direction of the D3Q7 lattices
      R fp = R(0), gp = R(0), hp = R(0), hd = R(0), gd = R(0);
      if (FLOW) fp = CHM ? fchm[a] : post_f_3d<R>(c, nd, a, f[a]);
      const R w = sc ? d3q7_w<R>(a) : R(0);
      if (sc) {
        gp = post_g_3d<R>(nd, a, g[a]);
        hp = post_h_3d<R>(nd, a, h[a]);
        hd = arrive_h_3d<R>(nd, hp, hold(a, cz, cy, cx));
        gd = UREL ? fma_r(-w, sub_r(uref(cz, cy, cx), Rg), gp) : gp;
      }
      auto store = [&](T* p, R fv, R gv, R hv) {
        if (FLOW) Pop<T>::st(p, fv);
        if (sc) {
          Pop<T>::st(p + QF * P, gv);
          Pop<T>::st(p + (QF + 7) * P, hv);
        }
      };
      if (go >> a & 1u) store(node + (a * P + sx[cx + 1] + sy[cy + 1] + sz[cz + 1]), fp, gd, hd);
      if (a > 0 && (odd >> a & 1u)) {
        if (sc) {  // reversed at the node
          hd = arrive_h_3d<R>(nd, hp, h[b < 7 ? b : 0]);
          if (UREL) gd = fma_r(-w, sub_r(uref(0, 0, 0), Rg), gp);
        }
        if (back >> a & 1u) store(node + b * P, fp, gd, hd);
        if (cx < 0) {
          // outflow ghost x = nx repeats this column
          if (sc) {
            hd = arrive_h_3d<R>(nd, hp, hold(a, cz, cy, 0));
            if (UREL) gd = fma_r(-w, sub_r(uref(cz, cy, 0), Rg), gp);
          }
          if (outf >> a & 1u) store(node + (a * P + sy[cy + 1] + sz[cz + 1]), fp, gd, hd);
        }
        if (cx > 0 && (inf >> a & 1u)) {
          // inflow ghost x = -1 (equilibrium, phi = -1: zero h deviation), unless
          // behind a wall
          const R uin = c.u_in, Uin = c.U_in, gu = FLOW ? uin : R(0);
          const R fin = d3q19_w<R>(a) * (R(3) * uin + R(4.5) * uin * uin - R(1.5) * uin * uin);
          R gin = w * ((Uin - Rg) + Uin * R(4) * gu);
          if (UREL) gin = fma_r(-w, uref(0, 0, 0) - Rg, gin);
          store(node + a * P, fin, gin, R(0));
        }
      }
    }
  }
}

}  // namespace lbk
