// wavelet_runs.cuh -- separable refinement and coarsening along lines: a thread
// keeps a window of inputs in registers and produces a run of outputs, so a
// run's taps are loaded together and shared.
#pragma once
#include "mr_internal.cuh"

namespace mr {

// Partial-sum type of the refinement: the block's, or float pairs for an FP32
// field in an FP64 block (the K^s weights are dyadic, exact in FP32).
template <typename TI, typename TP>
struct RefSum {
  using U = TP;
  static __device__ __forceinline__ U zero() { return TP(0); }
  static __device__ __forceinline__ U from(TI v) { return Cvt<TP>::f(v); }
  static __device__ __forceinline__ U acc(U s, double w, U v) { return racc(s, TP(w), v); }
  static __device__ __forceinline__ U norm(U s) { return s; }
  static __device__ __forceinline__ TP value(U s) { return s; }
};
template <>
struct RefSum<float, double> {
  using U = F2;
  static __device__ __forceinline__ U zero() { return f2_of(0.f); }
  static __device__ __forceinline__ U from(float v) { return f2_of(v); }
  static __device__ __forceinline__ U acc(U s, double w, U v) { return f2_acc(s, float(w), v); }
  static __device__ __forceinline__ U norm(U s) { return f2_norm(s); }
  static __device__ __forceinline__ double value(U s) { return f2_dbl(s); }
};

// Zero-detail refinement along one line: fine points f0 .. f0 + n - 1 (n <= 16)
// from the coarse values at(q) (q: coarse index, each called once); put(m, v)
// receives point f0 + m.  A register window of N coarse values moves along the
// line and yields an even (coincident) and an odd (K^s) point per step.
template <int N, int NT, typename RS, typename A, typename F>
__device__ __forceinline__ void refine_run(A at, int f0, int n, F put) {
  using W = Wav<N, NT>;
  using U = typename RS::U;
  constexpr int ko = N - 1, h = N / 2;
  // window w[0..N-1] = coarse q-h+1 .. q+h around the odd point 2q + 1
  const int q0 = f0 >> 1;
  U w[N];
#pragma unroll
  for (int x = 0; x + 1 < N; ++x) w[x] = at(q0 - h + 1 + x);
  const int par = f0 & 1;
  // (the last value of a window is read only where its odd point exists)
  w[N - 1] = par || n > 1 ? at(q0 + h) : w[0];
  for (int m = -par; m < n; m += 2) {  // even point m, odd point m + 1
    if (m >= 0) put(m, w[h - 1]);
    if (m + 1 < n) {
      U s = RS::acc(RS::zero(), W::K(-ko), w[0]);
#pragma unroll
      for (int x = 1; x < N; ++x) s = RS::acc(s, W::K(2 * x - ko), w[x]);
      put(m + 1, s);
    }
    if (m + 2 < n) {
#pragma unroll
      for (int x = 0; x + 1 < N; ++x) w[x] = w[x + 1];
      if (m + 3 < n) w[N - 1] = at(q0 + (m + par) / 2 + 1 + h);
    }
  }
}
// the same from the coarse values src[q * st]
template <int N, int NT, typename RS, typename U, typename F>
__device__ __forceinline__ void refine_run(const U *src, int st, int f0, int n, F put) {
  refine_run<N, NT, RS>([&](int q) { return src[q * st]; }, f0, n, put);
}

// tensor H^a along one line: sum_t H^a(t) src[(2 m + t) st], m = 0 .. n - 1 <= M,
// from one window of fine values; put(m, sum)
template <int N, int NT, int M, typename TP, typename F>
__device__ __forceinline__ void coarsen_run(const TP *src, int st, int n, F put) {
  constexpr int hH = Wav<N, NT>::hwH, len = 2 * M - 1 + 2 * hH;
  TP v[len];
#pragma unroll
  for (int x = 0; x < len; ++x) {
    // (points that no sum with m < n reads are not loaded)
    bool used = false;
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (x - hH - 2 * m >= -hH && x - hH - 2 * m <= hH && Wav<N, NT>::H(x - hH - 2 * m) != 0.0) used |= m < n;
    v[x] = used ? src[(x - hH) * st] : TP(0);
  }
#pragma unroll
  for (int m = 0; m < M; ++m) {
    if (m >= n) break;
    TP s = TP(0);
    for_taps<N, NT, FK_H>([&](int t, double w) { s = racc(s, TP(w), v[2 * m + hH + t]); });
    put(m, s);
  }
}

// H^a coarsening of the coarse points [lo, hi)^3 of a block (fine value of coarse
// point p at F[2 p0 + Wd (2 p1 + Wd 2 p2)]), put(p0, p1, p2, value): thinnest axis a
// first (then b, c), up to four layers of a at a time: one thread loads a fine
// column along a and sums every layer from it; along b and c a thread sums four
// points from one window.  buf: cap elements of shared memory (at least one
// layer's sums); the whole CTA takes part.
template <int N, int NT, typename TP, typename F>
__device__ __forceinline__ void coarsen_box(const TP *F0, int Wd, const int *lo, const int *hi, TP *buf, int cap,
                                            F put) {
  constexpr int hH = Wav<N, NT>::hwH, LAYERS = 4;
  const int W2 = Wd * Wd, tid = threadIdx.x, bd = blockDim.x;
  const int e0 = hi[0] - lo[0], e1 = hi[1] - lo[1], e2 = hi[2] - lo[2];
  const int a = e0 < e1 && e0 < e2 ? 0 : e1 < e2 ? 1 : 2, bx = a == 0 ? 1 : 0, c = 3 - a - bx;
  const int na = hi[a] - lo[a], nbb = hi[bx] - lo[bx], nc = hi[c] - lo[c];
  const int fb = 2 * nbb - 1 + 2 * hH, fc = 2 * nc - 1 + 2 * hH;
  const int sA = a == 0 ? 1 : a == 1 ? Wd : W2, sB = bx == 0 ? 1 : Wd, sC = c == 1 ? Wd : W2;
  const int layers = max(1, min(min(na, LAYERS), cap / (fc * (fb + nbb))));
  const int rb = (nbb + 3) >> 2, rc = (nc + 3) >> 2;  // runs of four points along b, c
  const DivM dfb = divm(fb), drb = divm(rb), dnb = divm(nbb), drc = divm(rc);
  for (int l0 = 0; l0 < na; l0 += layers) {
    const int nl = min(layers, na - l0);
    TP *A = buf, *B = A + nl * fc * fb;  // [l][fc][fb], [l][fc][nbb]
    const TP *src0 = F0 + 2 * (lo[a] + l0) * sA + (2 * lo[bx] - hH) * sB + (2 * lo[c] - hH) * sC;
    for (int idx = tid; idx < fc * fb; idx += bd) {
      const int ic = divq(idx, dfb), ib = idx - ic * fb;
      coarsen_run<N, NT, LAYERS>(src0 + ib * sB + ic * sC, sA, nl, [&](int l, TP v) { A[l * fc * fb + idx] = v; });
    }
    __syncthreads();
    for (int idx = tid; idx < nl * fc * rb; idx += bd) {
      const int r = divq(idx, drb), ib = 4 * (idx - r * rb);
      TP *d = B + r * nbb + ib;
      coarsen_run<N, NT, 4>(A + r * fb + 2 * ib + hH, 1, min(4, nbb - ib), [&](int m, TP v) { d[m] = v; });
    }
    __syncthreads();
    for (int idx = tid; idx < nl * rc * nbb; idx += bd) {
      const int r = divq(idx, dnb), l = divq(r, drc), ib = idx - r * nbb, ic = 4 * (r - l * rc);
      coarsen_run<N, NT, 4>(B + (l * fc + 2 * ic + hH) * nbb + ib, nbb, min(4, nc - ic), [&](int m, TP sv) {
        const int va = lo[a] + l0 + l, vb = lo[bx] + ib, vc = lo[c] + ic + m;
        put(a == 0 ? va : vb, a == 0 ? vb : a == 1 ? va : vc, a == 2 ? va : vc, sv);
      });
    }
    __syncthreads();
  }
}

}  // namespace mr
