// Device helpers of liblbpf.so: lattice constants, population storage
// codecs and the anisotropy function.  Internal to the CUDA library.
#pragma once

#include "lbpf_internal.cuh"

namespace lbk {

// ---- lattices (direction order of the exported state) ----------------------
// D2Q9: (0,0) (1,0) (0,1) (-1,0) (0,-1) (1,1) (-1,1) (-1,-1) (1,-1)
__device__ constexpr int D2_CX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__device__ constexpr int D2_CY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
__device__ constexpr int D2_OPP[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
// Weights.  In FP32 the three values are chosen so that their exact sum
// (w0 + 4 w1 + 4 w2, resp. w0 + 6 w1 + 12 w2) is 1: with the rounded 4/9, 1/9,
// 1/36 the sum is 1 + 7.4e-9, which biases every zeroth moment by that much
// per collision (sum of U + phi(t-1) drifts; phi drifts by ~1e-8 per step).
// FP64 uses the plain fractions.
template <typename R>
__device__ __forceinline__ R d2_w(int a);
template <>
__device__ __forceinline__ double d2_w<double>(int a) {
  return a == 0 ? 4.0 / 9.0 : (a < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
}
template <>
__device__ __forceinline__ float d2_w<float>(int a) {
  return a == 0 ? 0x1.c71c72p-2f : (a < 5 ? 0x1.c71c72p-4f : 0x1.c71c70p-6f);
}

// D3Q19: rest, +x, -x, +y, -y, +z, -z, then the 12 edge links; D3Q7 is the
// first seven of these.
__device__ constexpr int D3_CX[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
__device__ constexpr int D3_CY[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
__device__ constexpr int D3_CZ[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
__device__ constexpr int D3_OPP[19] = {0, 2, 1, 4, 3, 6, 5, 8, 7, 10, 9, 12, 11, 14, 13, 16, 15, 18, 17};
template <typename R>
__device__ __forceinline__ R d3q19_w(int a);
template <>
__device__ __forceinline__ double d3q19_w<double>(int a) {
  return a == 0 ? 1.0 / 3.0 : (a < 7 ? 1.0 / 18.0 : 1.0 / 36.0);
}
template <>
__device__ __forceinline__ float d3q19_w<float>(int a) {
  return a == 0 ? 0x1.555558p-2f : (a < 7 ? 0x1.c71c72p-5f : 0x1.c71c6ep-6f);
}
template <typename R>
__device__ __forceinline__ R d3q7_w(int a) {
  return a == 0 ? R(0.25) : R(0.125);
}

// ---- arithmetic helpers -------------------------------------------------------
// Reciprocal of the per-node relaxation and velocity denominators (all in
// [0.5, ~10]) and reciprocal root of |grad phi|^2 (> 1e-12 where it is used):
// in FP32 the hardware approximations (2 ulp), one instruction each in the
// form without denormal handling (denormal arguments do not occur; the forms
// with it scale and compare around each, 40 issue slots per two nodes); in
// FP64 the exact division and root.
__device__ __forceinline__ float rcp_r(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float rsqrt_r(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ double rcp_r(double v) { return 1.0 / v; }
__device__ __forceinline__ double rsqrt_r(double v) { return rsqrt(v); }
// clamp to [-1, 1]; NaN stays NaN
__device__ __forceinline__ double clamp1(double v) {
  return v < -1.0 ? -1.0 : (v > 1.0 ? 1.0 : v);
}
__device__ __forceinline__ float clamp1(float v) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "f"(-1.0f));
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(r), "f"(1.0f));
  return r;
}
__device__ __forceinline__ bool finite_r(float v) { return isfinite(v); }

// Explicitly rounded multiply / add / fused multiply-add.  The values a node
// pushes are written with these so that the compiler cannot fuse them
// differently in different code paths (interior vs edge tiles, single vs
// batched kernels): every path then rounds identically and a node's result
// does not depend on how the grid was tiled.  Two exceptions in 3D: 16-bit grids
// keep an order of one sum that follows their blocks (aniso_3d), and the central
// Hermite MRT there is written as plain expressions.
__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_r(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_r(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ bool finite_r(double v) { return isfinite(v); }

// ---- population storage ---------------------------------------------------------
// Every lattice stores and updates the deviation of its populations from the
// weights times a reference moment, d_a = p_a - w_a M_ref (M_ref = 1 for f,
// U_ref for g, -1 for h), so that rounding acts on small numbers: the moments
// are M = M_ref + sum d and the equilibria are written as deviations too.
// FP32/FP64 store d as is; the 16-bit modes store d rounded to binary16 or
// bfloat16 and compute in FP32.
template <typename T>
struct Pop;
template <>
struct Pop<float> {
  template <typename R>
  __device__ static __forceinline__ R ld(const float* p) { return R(*p); }
  template <typename R>
  __device__ static __forceinline__ void st(float* p, R v) { *p = float(v); }
};
template <>
struct Pop<double> {
  template <typename R>
  __device__ static __forceinline__ R ld(const double* p) { return R(*p); }
  template <typename R>
  __device__ static __forceinline__ void st(double* p, R v) { *p = double(v); }
};
template <>
struct Pop<__half> {
  template <typename R>
  __device__ static __forceinline__ R ld(const __half* p) { return R(__half2float(*p)); }
  template <typename R>
  __device__ static __forceinline__ void st(__half* p, R v) { *p = __float2half_rn(float(v)); }
};
template <>
struct Pop<__nv_bfloat16> {
  template <typename R>
  __device__ static __forceinline__ R ld(const __nv_bfloat16* p) {
    return R(__bfloat162float(*p));
  }
  template <typename R>
  __device__ static __forceinline__ void st(__nv_bfloat16* p, R v) {
    *p = __float2bfloat16_rn(float(v));
  }
};

// ---- one or two nodes per thread ------------------------------------------------
// The per-node arithmetic is written once over a number type N: float or
// double (one node) or float2 (two nodes of a thread, one per lane, on the
// packed FP32 instructions of sm_100 and later: one issue slot for both).
// Every lane rounds exactly like the scalar form, so a node's result does not
// depend on how many nodes its thread holds.
template <typename N>
struct Lanes {
  using S = N;
  static constexpr int V = 1;
};
template <>
struct Lanes<float2> {
  using S = float;
  static constexpr int V = 2;
};
__device__ __forceinline__ float2 fma_r(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul_r(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add_r(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a b for a product whose only use is a sum: the assembler fuses such a packed
// multiply and add into one rounding (the scalar ones it does not, and neither
// a packed product with several uses), so the packed form takes a -0 that the
// compiler does not know to be one as its addend
__device__ __forceinline__ float prod_r(float a, float b, float) { return mul_r(a, b); }
__device__ __forceinline__ double prod_r(double a, double b, double) { return mul_r(a, b); }
__device__ __forceinline__ float2 prod_r(float2 a, float2 b, float2 mzero) {
  return __ffma2_rn(a, b, mzero);
}
__device__ __forceinline__ float neg_r(float a) { return -a; }
__device__ __forceinline__ double neg_r(double a) { return -a; }
__device__ __forceinline__ float2 neg_r(float2 a) { return make_float2(-a.x, -a.y); }
template <typename N>
__device__ __forceinline__ N sub_r(N a, N b) { return add_r(a, neg_r(b)); }
__device__ __forceinline__ float2 rcp_r(float2 v) { return make_float2(rcp_r(v.x), rcp_r(v.y)); }
__device__ __forceinline__ float2 rsqrt_r(float2 v) {
  return make_float2(rsqrt_r(v.x), rsqrt_r(v.y));
}
__device__ __forceinline__ float2 clamp1(float2 v) { return make_float2(clamp1(v.x), clamp1(v.y)); }
template <typename N>
__device__ __forceinline__ N splat(typename Lanes<N>::S v) {
  if constexpr (Lanes<N>::V == 2) return make_float2(v, v);
  else return v;
}
// lane k of a number of one or two nodes
template <typename N>
__device__ __forceinline__ typename Lanes<N>::S lane(const N& v, int k) {
  if constexpr (Lanes<N>::V == 2) return k ? v.y : v.x;
  else return v;
}
template <typename N>
__device__ __forceinline__ void set_lane(N& v, int k, typename Lanes<N>::S s) {
  if constexpr (Lanes<N>::V == 2) (k ? v.y : v.x) = s;
  else v = s;
}
// 0 in every lane where a, b and c are finite, elsewhere NaN
template <typename N>
__device__ __forceinline__ N finite_mark(N a, N b, N c) {
  const N z = splat<N>(typename Lanes<N>::S(0));
  return fma_r(c, z, fma_r(b, z, mul_r(a, z)));
}
// is the mark 0 in every lane?
template <typename N>
__device__ __forceinline__ bool all_finite(N mark) {
  if constexpr (Lanes<N>::V == 2) return mark.x + mark.y == 0.f;
  else return mark == typename Lanes<N>::S(0);
}
// v where |grad phi|^2 = g2 > 1e-12, elsewhere w
__device__ __forceinline__ float where_steep(float g2, float v, float w) {
  return g2 > 1e-12f ? v : w;
}
__device__ __forceinline__ double where_steep(double g2, double v, double w) {
  return g2 > 1e-12 ? v : w;
}
__device__ __forceinline__ float2 where_steep(float2 g2, float2 v, float2 w) {
  return make_float2(where_steep(g2.x, v.x, w.x), where_steep(g2.y, v.y, w.y));
}
__device__ __forceinline__ bool any_steep(float g2) { return g2 > 1e-12f; }
__device__ __forceinline__ bool any_steep(double g2) { return g2 > 1e-12; }
__device__ __forceinline__ bool any_steep(float2 g2) { return g2.x > 1e-12f || g2.y > 1e-12f; }

// ---- anisotropy (Eq. 3) and flux vector N (Eq. 21) ----------------------------
// n = -grad/|grad| (solid -> liquid); a_s = 1 and N = 0 where |grad|^2 <= 1e-12.
// k-fold: cos/sin(k theta) are the real and imaginary parts of (n_x + i
// n_y)^k, rotated by k theta0, so no atan2 is needed.
// N = fac |grad|^2 a_s d(a_s)/d(grad):
//   k-fold: N = fac k eps a_s sin(k(theta - theta0)) (g_y, -g_x)
//   cubic : N_i = fac 16 eps a_s |grad| (n_i S - n_i^3), S = sum n_j^4
template <typename N>
__device__ __forceinline__ void aniso_cubic(const Coef<N>& c, const N* n, N g2, N ig, int dim,
                                            N& a, N* out) {
  N n2[3];
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (d < dim) n2[d] = mul_r(n[d], n[d]);
  N S = fma_r(n2[0], n2[0], mul_r(n2[1], n2[1]));
  if (dim == 3) S = fma_r(n2[2], n2[2], S);
  a = fma_r(c.eps4, S, c.cub0);
  const N amp = mul_r(mul_r(c.amp_c, a), mul_r(g2, ig));
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (d < dim) out[d] = mul_r(mul_r(amp, n[d]), sub_r(S, n2[d]));
}

template <typename N>
__device__ __forceinline__ void aniso_2d(const Coef<N>& c, int fold, N gx, N gy, N& as, N& Nx,
                                         N& Ny) {
  using S1 = typename Lanes<N>::S;
  as = splat<N>(S1(1));
  Nx = Ny = splat<N>(S1(0));
  const N g2 = fma_r(gx, gx, mul_r(gy, gy));
  if (!any_steep(g2) || lane(c.eps, 0) == S1(0)) return;
  // (n = 0 on a flat lane: the k-fold form then gives a_s = 1, N = 0 by itself)
  const N ig = where_steep(g2, rsqrt_r(g2), splat<N>(S1(0)));
  const N n[2] = {mul_r(neg_r(gx), ig), mul_r(neg_r(gy), ig)};
  if (fold > 0) {
    N ck = n[0], sk = n[1];
    for (int j = 1; j < fold; ++j) {
      const N c2 = fma_r(ck, n[0], neg_r(mul_r(sk, n[1])));
      sk = fma_r(ck, n[1], mul_r(sk, n[0]));
      ck = c2;
    }
    const N cosd = fma_r(ck, c.ck0, mul_r(sk, c.sk0));
    const N sind = fma_r(sk, c.ck0, neg_r(mul_r(ck, c.sk0)));
    as = fma_r(c.eps, cosd, splat<N>(S1(1)));
    const N amp = mul_r(mul_r(c.amp_k, as), sind);
    Nx = mul_r(amp, gy);
    Ny = mul_r(neg_r(amp), gx);
  } else {
    N a, out[2];
    aniso_cubic<N>(c, n, g2, ig, 2, a, out);
    as = where_steep(g2, a, as);
    Nx = out[0];
    Ny = out[1];
  }
}

// y_first: |grad|^2 takes x's square rounded and adds y's exactly, else the other
// way round.  An FP32 rounding apart, but with 16-bit storage it turns over a
// stored value here and there, which spreads over the run; results keep to the
// order that each part of a 16-bit grid has always had: y first in the blocks of
// 32 x 4 nodes that touch no face and, of 32 x 4 x 8, hold and border no solid node.
// Neither order is the more exact; a state moved by a node along a periodic axis may
// differ by such roundings.
template <typename N>
__device__ __forceinline__ void aniso_3d(const Coef<N>& c, const N (&g)[3], bool y_first, N& as,
                                         N (&Nv)[3]) {
  using S1 = typename Lanes<N>::S;
  as = splat<N>(S1(1));
#pragma unroll
  for (int d = 0; d < 3; ++d) Nv[d] = splat<N>(S1(0));
  const N ga = y_first ? g[1] : g[0], gb = y_first ? g[0] : g[1];
  const N g2 = fma_r(g[2], g[2], fma_r(ga, ga, mul_r(gb, gb)));
  if (!any_steep(g2) || lane(c.eps, 0) == S1(0)) return;
  // (n = 0 on a flat lane, so N = 0 there by itself)
  const N ig = where_steep(g2, rsqrt_r(g2), splat<N>(S1(0)));
  N n[3], a;
#pragma unroll
  for (int d = 0; d < 3; ++d) n[d] = mul_r(neg_r(g[d]), ig);
  aniso_cubic<N>(c, n, g2, ig, 3, a, Nv);
  as = where_steep(g2, a, as);
}

// periodic wrap of a coordinate that is at most one period out of range
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
// neighbour coordinate for the gradient stencil: periodic wrap, else copy the
// nearest node (zero normal derivative)
__device__ __forceinline__ int grad_coord(int v, int n, int bc) {
  if (bc == BC_PERIODIC) return wrap1(v, n);
  return v < 0 ? 0 : (v >= n ? n - 1 : v);
}

}  // namespace lbk
