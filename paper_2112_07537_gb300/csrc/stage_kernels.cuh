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
// above 2^49 c), the quotients are taken one by one.  Where tau is below 2^-26
// of every c, r_k^2 < 2^-53 and each a_k is 1 to rounding: it is taken as 1, for
// the scaled weights of a field so small that every c is eps are 1e-180 and their
// products with N_k would underflow (from differences of 1e-128 down).  All
// three tests are on the exponent words, whose difference is at most 0.1 off the
// logarithm of the ratio.
__device__ __forceinline__ double weno_corr(double c0, double c1, double c2, double n0, double n1, double n2) {
  const double tau = fabs(c0 - c2);
  const unsigned k0 = (unsigned)__double2hiint(c0), k1 = (unsigned)__double2hiint(c1),
                 k2 = (unsigned)__double2hiint(c2);
  const unsigned hi = max(max(k0, k1), k2), lo = min(min(k0, k1), k2);
  const int above = (int)lo - __double2hiint(tau);  // c over tau, in exponent words
  double a0 = 1.0, a1 = 1.0, a2 = 1.0;
  if (hi > 0x49466bb7u || above <= -(49 << 20)) {
    const double cap = WenoC<double>::rcap;
    double r0 = tau / c0, r1 = tau / c1, r2 = tau / c2;
    r0 = r0 > cap ? cap : r0;
    r1 = r1 > cap ? cap : r1;
    r2 = r2 > cap ? cap : r2;
    a0 = fma(r0, r0, 1.0), a1 = fma(r1, r1, 1.0), a2 = fma(r2, r2, 1.0);
  } else if (above < (27 << 20)) {
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

// Walks n cells of one grid line and hands emit(m, dF, c) the halved flux
// difference F_{m+1/2}/2 - F_{m-1/2}/2 of every cell m and its value c = phi(m).
// phi(m), hv(m): value and half velocity at cell m (-3 <= m < n + 3, called once
// each in ascending order); the velocities of the two points of an interface pick
// its upwind side.  The point fluxes are rounded products (never contracted into
// a sum), so a flux does not depend on where its line starts.
template <typename T, int SCHEME, typename FP, typename FV, typename FE>
__device__ __forceinline__ void walk_line(int n, FP phi, FV hv, FE emit) {
  const T wa = rmul(hv(-3), phi(-3)), wb = rmul(hv(-2), phi(-2));
  T vl = hv(-1), w2 = rmul(vl, phi(-1));
  T va = hv(0), a1 = phi(0), w3 = rmul(va, a1);
  T vb = hv(1), a2 = phi(1), w4 = rmul(vb, a2);
  T vc = hv(2), a3 = phi(2), w5 = rmul(vc, a3);
  T h0 = wb - wa, h1 = w2 - wb, h2 = w3 - w2, h3 = w4 - w3, h4 = w5 - w4;
  T v0 = T(0), v1 = T(0), v2 = T(0), v3 = T(0);
  if (SCHEME == MR_WENOZ5) v0 = weno_v(h0, h1), v1 = weno_v(h1, h2), v2 = weno_v(h2, h3), v3 = weno_v(h3, h4);
  T Fm = half_flux<T, SCHEME>(w2, w3, h0, h1, h2, h3, h4, v0, v1, v2, v3, vl + va >= T(0));
#pragma unroll(sizeof(T) == 4 ? 4 : 2)
  for (int m = 0; m < n; ++m) {
    const T vn = hv(m + 3), an = phi(m + 3), wn = rmul(vn, an);
    w2 = w3, w3 = w4, w4 = w5;
    h0 = h1, h1 = h2, h2 = h3, h3 = h4, h4 = wn - w5;
    w5 = wn;
    if (SCHEME == MR_WENOZ5) v0 = v1, v1 = v2, v2 = v3, v3 = weno_v(h3, h4);
    const T Fp = half_flux<T, SCHEME>(w2, w3, h0, h1, h2, h3, h4, v0, v1, v2, v3, va + vb >= T(0));
    emit(m, Fp - Fm, a1);
    Fm = Fp;
    va = vb, vb = vc, vc = vn;
    a1 = a2, a2 = a3, a3 = an;
  }
}

// ---------------------------------------------------------------------------
// Two FP32 lines at once.  A thread walks a pair of lines in lockstep with packed
// arithmetic (one instruction per pair of sums, products or fused multiply-adds,
// each half rounded like the scalar instruction), so a kernel bound by issued
// instructions issues about half of them; selects, minima and reciprocals have
// no packed form.  Operation for operation the values of the scalar code above.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pfma(float a, float2 b, float2 c) { return __ffma2_rn(both(a), b, c); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(both(-1.f), b, a); }

__device__ __forceinline__ float2 weno_v(float2 hm, float2 hp) {
  const float2 g = psub(hp, hm);
  return pfma(pmul(both(13.0f / 3), g), g, both((float)WenoC<float>::eps));
}

__device__ __forceinline__ float2 weno_corr(float2 c0, float2 c1, float2 c2, float2 n0, float2 n1, float2 n2) {
  const float cap = float(WenoC<float>::rcap);
  const float2 tau = psub(c0, c2);
  auto ratio = [&](float2 c) {
    const float2 r = pmul(tau, make_float2(rcp_approx(c.x), rcp_approx(c.y)));
    return make_float2(fminf(fabsf(r.x), cap), fminf(fabsf(r.y), cap));
  };
  const float2 r0 = ratio(c0), r1 = ratio(c1), r2 = ratio(c2), one = both(1.f);
  const float2 a0 = pfma(r0, r0, one), a1 = pfma(r1, r1, one), a2 = pfma(r2, r2, one);
  const float2 den = pfma(6.f, a1, pfma(3.f, a2, a0));
  return pmul(pfma(a2, n2, pfma(a1, n1, pmul(a0, n0))), make_float2(rcp_approx(den.x), rcp_approx(den.y)));
}

// half_flux of a pair; lx, ly: the side of either line (LEFT: left of both)
template <int SCHEME, bool LEFT>
__device__ __forceinline__ float2 half_flux2(float2 w2, float2 w3, float2 h0, float2 h1, float2 h2, float2 h3,
                                             float2 h4, float2 v0, float2 v1, float2 v2, float2 v3, bool lx, bool ly) {
  auto up = [&](float2 l, float2 r) { return LEFT ? l : make_float2(lx ? l.x : r.x, ly ? l.y : r.y); };
  const float2 c = up(w2, w3), e2 = up(h1, h3);
  float2 s;
  if (SCHEME == MR_CONS3) {
    s = pfma(1.0f / 3, h2, pmul(both(1.0f / 6), e2));
  } else {
    const float2 e1 = up(h0, h4), e4 = up(h3, h1);
    if (SCHEME == MR_CONS5) {
      s = pfma(11.0f / 60, e2, pfma(-1.0f / 30, e1, pfma(2.0f / 5, h2, pmul(both(-1.0f / 20), e4))));
    } else {
      // (t_0, t_2 with the sign changed: they are squared)
      const float2 t0 = pfma(-3.f, e2, e1), t1 = padd(e2, h2), t2 = pfma(-3.f, h2, e4);
      const float2 c0 = pfma(t0, t0, up(v0, v3)), c1 = pfma(t1, t1, up(v1, v2)), c2 = pfma(t2, t2, up(v2, v1));
      const float2 n0 = pfma(5.0f / 6, e2, pmul(both(-1.0f / 3), e1)), n1 = pfma(2.f, h2, e2),
                   n2 = pfma(2.f, h2, pmul(both(-0.5f), e4));
      s = weno_corr(c0, c1, c2, n0, n1, n2);
    }
  }
  return LEFT ? padd(c, s) : pfma(make_float2(lx ? 1.f : -1.f, ly ? 1.f : -1.f), s, c);
}

// Walk of a pair of lines: walk_line a cell at a time, with (LAP) the Laplacian
// term along the line and (LEFT: a constant velocity along the walk) the left side
// throughout.
template <int SCHEME, bool LAP, bool LEFT>
struct Walk2 {
  float2 am, a0, a1, a2, a3, va, vb, vc;  // phi(m-2 .. m+2), half velocities at m .. m+2
  float2 w2, w3, w4, w5, h0, h1, h2, h3, h4, v0, v1, v2, v3, Fm;
  __device__ __forceinline__ float2 flux(float2 ul, float2 ur) {
    const float2 u = LEFT ? ul : padd(ul, ur);
    return half_flux2<SCHEME, LEFT>(w2, w3, h0, h1, h2, h3, h4, v0, v1, v2, v3, u.x >= 0.f, u.y >= 0.f);
  }
  // phi(m), hv(m): values and half velocities at cells -3 .. 2
  template <typename FP, typename FV>
  __device__ __forceinline__ void start(FP phi, FV hv) {
    const float2 wa = pmul(hv(-3), phi(-3));
    am = phi(-2);
    const float2 wb = pmul(hv(-2), am), vl = hv(-1);
    a0 = phi(-1), w2 = pmul(vl, a0);
    va = hv(0), a1 = phi(0), w3 = pmul(va, a1);
    vb = hv(1), a2 = phi(1), w4 = pmul(vb, a2);
    vc = hv(2), a3 = phi(2), w5 = pmul(vc, a3);
    h0 = psub(wb, wa), h1 = psub(w2, wb), h2 = psub(w3, w2), h3 = psub(w4, w3), h4 = psub(w5, w4);
    v0 = v1 = v2 = v3 = both(0.f);
    if (SCHEME == MR_WENOZ5) v0 = weno_v(h0, h1), v1 = weno_v(h1, h2), v2 = weno_v(h2, h3), v3 = weno_v(h3, h4);
    Fm = flux(vl, va);
  }
  // an, vn: values and half velocities at cell m + 3; emit(dF, c, lap)
  template <typename FE>
  __device__ __forceinline__ void step(int diff, float2 an, float2 vn, FE emit) {
    const float2 wn = pmul(vn, an);
    w2 = w3, w3 = w4, w4 = w5;
    h0 = h1, h1 = h2, h2 = h3, h3 = h4, h4 = psub(wn, w5);
    w5 = wn;
    if (SCHEME == MR_WENOZ5) v0 = v1, v1 = v2, v2 = v3, v3 = weno_v(h3, h4);
    const float2 Fp = flux(va, vb);
    emit(psub(Fp, Fm), a1,
         LAP ? make_float2(lap_term<float>(am.x, a0.x, a1.x, a2.x, a3.x, diff),
                           lap_term<float>(am.y, a0.y, a1.y, a2.y, a3.y, diff))
             : both(0.f));
    Fm = Fp;
    va = vb, vb = vc, vc = vn;
    if (LAP) am = a0, a0 = a1;
    a1 = a2, a2 = a3, a3 = an;
  }
};

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
