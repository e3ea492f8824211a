// stage_kernels.cuh -- interface fluxes (Tables SM3 / SM4), the walk along a
// grid line that the stage kernels share, and the Laplacian terms.
#pragma once
#include "mr_internal.cuh"

namespace mr {

// ---------------------------------------------------------------------------
// Interface flux F_{i+1/2} (Tables SM3 / SM4) in difference form.  With point
// fluxes f_{i-2..i+3}, halved (w = f/2: an exact scaling that turns the 1/4
// and 13/12 of the smoothness indicators into 1 and 13/3), first differences
// h_j = w_{j+1} - w_j and c = w_i, the reconstruction biased to the left is
//   F/2 = c + sum_k a_k N_k / sum_k a_k g_k / 0.1,
//   N_0 = 5/6 e2 - 1/3 e1, N_1 = e2 + 2 e3, N_2 = 2 e3 - e4/2
// with e1..e4 = h_{i-2..i+1} (the ideal weights 1 : 6 : 3 folded into N_k)
// and, for WENO-Z, beta_k + eps = t_k^2 + V_k,
//   t_0 = 3 e2 - e1, t_1 = e2 + e3, t_2 = 3 e3 - e4,
//   V_j = 13/3 (h_j - h_{j-1})^2 + eps at the points j = i-1, i, i+1.
// The reconstruction biased to the right is the mirror image: e1..e4 =
// h_{i+2..i-1}, V at i+2, i+1, i, c = w_{i+1}, and the sum subtracted, so the
// upwind choice only selects inputs.  h and V belong to one point each, so a
// thread that walks a grid line evaluates them once per point and shares them
// between neighbouring interfaces.
// WENO-Z weights: a_k = 1 + r_k^2, r_k = min(tau / (beta_k + eps), rcap),
// tau = |beta_0 - beta_2|, eps = 1e-30, rcap = 1e15 (r_k^2 finite in FP32).
// ---------------------------------------------------------------------------
template <typename T>
struct WenoC {
  static constexpr double eps = 1e-30;
  static constexpr double rcap = 1e15;
};

// V_j of the point between the differences hm = h_{j-1} and hp = h_j
template <typename T>
__device__ __forceinline__ T weno_v(T hm, T hp) {
  const T g = hp - hm;
  return fma(T(13.0 / 3) * g, g, T(WenoC<T>::eps));
}

// FP32: approximate reciprocals (1 ulp) times the numerator.  The operands are
// normal numbers (c >= 1e-30, weight sum >= 10), so the form that flushes
// denormals needs none of the scaling around __fdividef; where c exceeds 2^126
// either gives 0.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float weno_corr(float c0, float c1, float c2, float n0, float n1, float n2) {
  const float tau = fabsf(c0 - c2), cap = float(WenoC<float>::rcap);
  const float r0 = fminf(tau * rcp_approx(c0), cap), r1 = fminf(tau * rcp_approx(c1), cap),
              r2 = fminf(tau * rcp_approx(c2), cap);
  const float a0 = fmaf(r0, r0, 1.f), a1 = fmaf(r1, r1, 1.f), a2 = fmaf(r2, r2, 1.f);
  const float den = fmaf(6.f, a1, fmaf(3.f, a2, a0));
  return fmaf(a2, n2, fmaf(a1, n1, a0 * n0)) * rcp_approx(den);
}
// FP64: the pipe is narrow here (2 fused multiply-adds per clock and SM), so
// the four divisions become one: a_k times (c_0 c_1 c_2)^2 is
// (c_0 c_1 c_2)^2 + (tau c_i c_j)^2.  Where that product could leave the
// exponent range (c above 1e45, infinities, NaN) or the cap could act (tau
// above 2^49 c, checked on the exponent words), the quotients are taken one by
// one.
__device__ __forceinline__ double weno_corr(double c0, double c1, double c2, double n0, double n1, double n2) {
  const double tau = fabs(c0 - c2);
  const unsigned k0 = (unsigned)__double2hiint(c0), k1 = (unsigned)__double2hiint(c1),
                 k2 = (unsigned)__double2hiint(c2);
  const unsigned hi = max(max(k0, k1), k2), lo = min(min(k0, k1), k2);
  double a0, a1, a2;
  if (hi > 0x49466bb7u || (int)lo <= __double2hiint(tau) - (49 << 20)) {
    const double cap = WenoC<double>::rcap;
    double r0 = tau / c0, r1 = tau / c1, r2 = tau / c2;
    r0 = r0 > cap ? cap : r0;
    r1 = r1 > cap ? cap : r1;
    r2 = r2 > cap ? cap : r2;
    a0 = fma(r0, r0, 1.0), a1 = fma(r1, r1, 1.0), a2 = fma(r2, r2, 1.0);
  } else {
    const double q0 = c1 * c2, q1 = c0 * c2, q2 = c0 * c1, pr = q0 * c0, p2 = pr * pr;
    const double e0 = tau * q0, e1 = tau * q1, e2 = tau * q2;
    a0 = fma(e0, e0, p2), a1 = fma(e1, e1, p2), a2 = fma(e2, e2, p2);
  }
  const double den = fma(6.0, a1, fma(3.0, a2, a0));
  return fma(a2, n2, fma(a1, n1, a0 * n0)) / den;
}

// F/2 at the interface behind point i: w2 = w_i, w3 = w_{i+1}, h0..h4 =
// h_{i-2..i+2}, v0..v3 = V_{i-1..i+2} (v: WENO-Z only, h0 / h4: not CONS-3).
template <typename T, int SCHEME>
__device__ __forceinline__ T half_flux(T w2, T w3, T h0, T h1, T h2, T h3, T h4, T v0, T v1, T v2, T v3, bool left) {
  const T c = left ? w2 : w3, e2 = left ? h1 : h3;
  if (SCHEME == MR_CONS3) {
    const T s = fma(T(1.0 / 3), h2, T(1.0 / 6) * e2);
    return left ? c + s : c - s;
  }
  const T e1 = left ? h0 : h4, e4 = left ? h3 : h1;
  if (SCHEME == MR_CONS5) {
    const T s = fma(T(11.0 / 60), e2, fma(T(-1.0 / 30), e1, fma(T(2.0 / 5), h2, T(-1.0 / 20) * e4)));
    return left ? c + s : c - s;
  }
  const T t0 = fma(T(3), e2, -e1), t1 = e2 + h2, t2 = fma(T(3), h2, -e4);
  const T c0 = fma(t0, t0, left ? v0 : v3), c1 = fma(t1, t1, left ? v1 : v2), c2 = fma(t2, t2, left ? v2 : v1);
  const T n0 = fma(T(5.0 / 6), e2, T(-1.0 / 3) * e1), n1 = fma(T(2), h2, e2), n2 = fma(T(2), h2, T(-0.5) * e4);
  const T s = weno_corr(c0, c1, c2, n0, n1, n2);
  return left ? c + s : c - s;
}

// F/2 from the six halved point fluxes w_{i-2..i+3} alone
template <typename T, int SCHEME>
__device__ __forceinline__ T half_flux6(const T *w, bool left) {
  const T h0 = w[1] - w[0], h1 = w[2] - w[1], h2 = w[3] - w[2], h3 = w[4] - w[3], h4 = w[5] - w[4];
  T va = T(0), vb = T(0), vc = T(0);
  if (SCHEME == MR_WENOZ5) {  // V of the three points that the upwind side reads
    const T e1 = left ? h0 : h4, e2 = left ? h1 : h3, e4 = left ? h3 : h1;
    va = weno_v(e1, e2), vb = weno_v(e2, h2), vc = weno_v(h2, e4);
  }
  return half_flux<T, SCHEME>(w[2], w[3], h0, h1, h2, h3, h4, left ? va : T(0), left ? vb : vc, left ? vc : vb,
                              left ? T(0) : va, left);
}

// One direction's term of the central Laplacian (Sec. 4.3, DIFF-2 / DIFF-4),
// unscaled by 1/h^2, from the values at offsets -2..2 along it.
template <typename T>
__device__ __forceinline__ T lap_term(T m2, T m1, T c, T p1, T p2, int diff) {
  if (diff == 2) return (m1 + p1) - T(2) * c;
  return (T(16) * (m1 + p1) - (m2 + p2) - T(30) * c) * T(1.0 / 12);
}

// State of a walk along one grid line: step() moves one cell on and hands
// emit(m, dF, c, lap) the halved flux difference F_{m+1/2}/2 - F_{m-1/2}/2 of
// cell m, its value c = phi(m) and (LAP) its Laplacian term along the line.  The
// velocities of the two points of an interface pick its upwind side, or (LEFT: a
// constant velocity along the walk) it is the left one throughout.  The point
// fluxes are rounded products (never contracted into a sum), so a flux does not
// depend on where its line starts.
template <typename T, int SCHEME, bool LAP, bool LEFT>
struct Walk {
  T am, a0, a1, a2, a3, va, vb, vc;  // phi(m-2 .. m+2), half velocities at m .. m+2
  T w2, w3, w4, w5, h0, h1, h2, h3, h4, v0, v1, v2, v3, Fm;
  // phi(m), hv(m): value and half velocity at cells -3 .. 2
  template <typename FP, typename FV>
  __device__ __forceinline__ void start(FP phi, FV hv) {
    const T wa = rmul(hv(-3), phi(-3));
    am = phi(-2);
    const T wb = rmul(hv(-2), am), vl = hv(-1);
    a0 = phi(-1), w2 = rmul(vl, a0);
    va = hv(0), a1 = phi(0), w3 = rmul(va, a1);
    vb = hv(1), a2 = phi(1), w4 = rmul(vb, a2);
    vc = hv(2), a3 = phi(2), w5 = rmul(vc, a3);
    h0 = wb - wa, h1 = w2 - wb, h2 = w3 - w2, h3 = w4 - w3, h4 = w5 - w4;
    v0 = v1 = v2 = v3 = T(0);
    if (SCHEME == MR_WENOZ5) v0 = weno_v(h0, h1), v1 = weno_v(h1, h2), v2 = weno_v(h2, h3), v3 = weno_v(h3, h4);
    Fm = half_flux<T, SCHEME>(w2, w3, h0, h1, h2, h3, h4, v0, v1, v2, v3, LEFT || vl + va >= T(0));
  }
  // an, vn: value and half velocity at cell m + 3
  template <typename FE>
  __device__ __forceinline__ void step(int m, int diff, T an, T vn, FE emit) {
    const T wn = rmul(vn, an);
    w2 = w3, w3 = w4, w4 = w5;
    h0 = h1, h1 = h2, h2 = h3, h3 = h4, h4 = wn - w5;
    w5 = wn;
    if (SCHEME == MR_WENOZ5) v0 = v1, v1 = v2, v2 = v3, v3 = weno_v(h3, h4);
    const T Fp = half_flux<T, SCHEME>(w2, w3, h0, h1, h2, h3, h4, v0, v1, v2, v3, LEFT || va + vb >= T(0));
    emit(m, Fp - Fm, a1, LAP ? lap_term<T>(am, a0, a1, a2, a3, diff) : T(0));
    Fm = Fp;
    va = vb, vb = vc, vc = vn;
    if (LAP) am = a0, a0 = a1;
    a1 = a2, a2 = a3, a3 = an;
  }
};

// Walks the n cells of one line.  phi(m), hv(m): value and half velocity at cell
// m (-3 <= m < n + 3, called once each in ascending order).
template <typename T, int SCHEME, bool LAP, bool LEFT, typename FP, typename FV, typename FE>
__device__ __forceinline__ void walk_line(int n, int diff, FP phi, FV hv, FE emit) {
  Walk<T, SCHEME, LAP, LEFT> w;
  w.start(phi, hv);
#pragma unroll(sizeof(T) == 4 ? 4 : 2)
  for (int m = 0; m < n; ++m) {
    const T vn = hv(m + 3), an = phi(m + 3);
    w.step(m, diff, an, vn, emit);
  }
}

// Central Laplacian at *c: sum over the three directions of lap_term.
template <typename T>
__device__ __forceinline__ T lap_at(const T *c, const int *stride, int diff) {
  T s = T(0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int st = stride[d];
    s += lap_term<T>(c[-2 * st], c[-st], c[0], c[st], c[2 * st], diff);
  }
  return s;
}

}  // namespace mr
