// adapt.cu -- block criterion and grid adaptation (Alg. SM3) on the device.
//
// One iteration: FP64 ghost fill with the adaptation shell -> per-leaf max
// |detail| (criterion) -> status -> policy (Jacobi iteration to the least
// fixed point) -> new leaves in Morton order (scan + emit) -> owner map of
// the new tree -> per field: ghost fill, refinement / coarsening / copy into
// the second pool, update step next to newly coarsened leaves.
#include <algorithm>

#include "wavelet_runs.cuh"

namespace mr {

enum { KIND_COPY = 0, KIND_CHILD = 1, KIND_PARENT = 2 };
enum { ST_COARSER = -1, ST_SAME = 0, ST_FINER = 1 };

// ------------------------------------------------------------- criterion
// Arithmetic of the details: the block's type TP, or float pairs (about 48
// significant bits on the FP32 pipe) from FP64 blocks.
template <typename TP, bool PAIRS>
struct DetOps {
  using E = TP;
  static __device__ __forceinline__ E zero() { return TP(0); }
  static __device__ __forceinline__ E load(TP v) { return v; }
  static __device__ __forceinline__ E acc(E s, double w, E v) { return racc(s, TP(w), v); }
  static __device__ __forceinline__ E norm(E s) { return s; }
  static __device__ __forceinline__ E lift(E v, E a, E b) { return racc(v, TP(0.25), a + b); }
  static __device__ __forceinline__ TP value(E s) { return s; }
};
template <>
struct DetOps<double, true> {
  using E = F2;
  static __device__ __forceinline__ E zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ E load(double v) { return f2_split(v); }
  static __device__ __forceinline__ E acc(E s, double w, E v) { return f2_acc(s, float(w), v); }
  static __device__ __forceinline__ E norm(E s) { return f2_norm(s); }
  static __device__ __forceinline__ E lift(E v, E a, E b) { return f2_norm(f2_acc(v, 0.25f, f2_add(a, b))); }
  static __device__ __forceinline__ double value(E s) { return f2_dbl(s); }
};

// Details gamma over a box of the extended region [-ext_f, nb-1+ext_b]^3 of one
// padded block: 1D filters x, then y, then z, G^a on odd and H^a on even
// coordinates; points with only even coordinates carry no detail and get 0.  Each 1D pass uses the lifting form of the pair:
// the G^a output at an odd point is the point minus the K^s-weighted prediction
// from its even neighbours (odd taps only), and the H^a output at an even point
// is the point plus 1/4 of the two neighbouring G^a outputs (N.2; H^a is the
// identity for N.0) -- the same filters, about half the multiply-adds.
// Planes march along z: the y-pass results live in a ring of 2(N-1)+1 planes,
// the z-details of the last two odd planes in a second ring (written and read
// by the same thread).  Four barriers per plane; the next plane is staged while
// the y pass runs.  A block is cut into column tiles so that two or three CTAs
// share an SM and one computes while another waits at a barrier.  Bound by issued
// instructions of the FP32 pipe (float pairs) and by the barriers: 2 080 leaves
// of 24^3, 6.2, took 2.79 ms whole (163 KB, one CTA per SM), 2.23 ms in tiles.
// emit(i, j, k, gamma) is called once per point of the box (gamma unconverted).
struct DetBox {  // inclusive
  int lo[3], hi[3];
};
struct DetTile {  // computed points [c0, c0 + w) of one axis: the lift of an even edge point reads one more
  int c0, w;
};
template <int NT>
__host__ __device__ __forceinline__ DetTile det_tile(int i0, int i1) {
  const int c0 = NT && !(i0 & 1) ? i0 - 1 : i0, c1 = NT && !(i1 & 1) ? i1 + 1 : i1;
  return {c0, c1 - c0 + 1};
}
// elements of shared memory for w computed columns and nR computed rows
template <int N>
__host__ __device__ __forceinline__ size_t det_elems(int nR, int w) {
  const int ko = N - 1, nA = nR + 2 * ko;
  return (size_t)(2 * ko + 3) * nR * w + (size_t)nA * w + (size_t)nA * (w + 2 * ko);
}

// Threads of a CTA, and items per thread and pass (det_tiles cuts accordingly):
// with KEEP the index arithmetic of a pass is done once, not once per plane (see
// criterion_impl).
constexpr int DET_THREADS = 512, DET_ITEMS = 2;
constexpr size_t DET_BYTES = 110 * 1024;  // shared memory: two CTAs on an SM

template <int N, int NT, bool PAIRS, bool KEEP, typename TP, typename F>
__device__ __forceinline__ void detail_planes(const TP *__restrict__ Pb, int nb, int Gi, const DetBox &B,
                                              typename DetOps<TP, PAIRS>::E *sm, F emit) {
  using W = Wav<N, NT>;
  using D = DetOps<TP, PAIRS>;
  using E = typename D::E;
  constexpr int ko = N - 1, R = 2 * ko + 1, K = DET_ITEMS;
  const int Wd = nb + 2 * Gi, tid = threadIdx.x, bd = blockDim.x;
  const DetTile tx = det_tile<NT>(B.lo[0], B.hi[0]), ty = det_tile<NT>(B.lo[1], B.hi[1]),
                tz = det_tile<NT>(B.lo[2], B.hi[2]);
  const int c0 = tx.c0, w = tx.w, wS = w + 2 * ko;               // columns
  const int r0 = ty.c0, nR = ty.w, r1 = r0 + nR - 1, nA = nR + 2 * ko;  // rows
  const int z0 = tz.c0, z1 = z0 + tz.w - 1, pl = nR * w;          // planes
  const int lo = -Gi, hi = nb - 1 + Gi;  // stored padded range
  E *ring = sm;             // [R][nR][w]     y-pass planes
  E *dz = sm + R * pl;      // [2][nR][w]     z-details of odd planes
  E *A = dz + 2 * pl;       // [nA][w]        x-pass of one plane
  E *S = A + nA * w;        // [nA][wS]       the staged plane
  // Beyond the region a pass reads even points only (the K^s taps of odd points):
  // rows and planes there with odd coordinates are left out.  Row jr of the
  // nE rows in use: the region's, then the even ones below and above it.
  const int eb = ko / 2 + 1, nE = nR + 2 * eb;
  auto row = [&](int q) {
    return q < nR ? ko + q : q < nR + eb ? (r0 & 1 ? ko - 1 : ko - 2) - 2 * (q - nR)
                                         : ko + nR + (r1 & 1 ? 0 : 1) + 2 * (q - nR - eb);
  };
  // items of the passes, the same on all planes.  x passes: (row, column) of A,
  // packed (-1: a row that is left out); y and z passes: offset in a plane
  const int fz = par_first(z0, 1);  // first odd plane
  const int fo = par_first(c0, 1), nxo = par_count(c0, c0 + w, 1);
  // even columns: those whose odd neighbours are computed (N.0: all)
  const int fe = NT && par_first(c0, 0) == c0 ? c0 + 2 : par_first(c0, 0);
  const int nxe = par_count(fe, NT ? c0 + w - 1 : c0 + w, 0);
  const int fy = par_first(r0, 1), ge = par_first(r0, 0), nyo = par_count(r0, r1 + 1, 1), nye = nR - nyo;
  const DivM dxo = divm(nxo > 0 ? nxo : 1), dxe = divm(nxe > 0 ? nxe : 1), dw = divm(w);
  auto at_x = [&](int idx, DivM d, int n, int first) {
    const int q = divq(idx, d), r = row(q);
    return r >= 0 && r < nA ? r << 16 | (first - c0 + 2 * (idx - q * n)) : -1;
  };
  auto at_xo = [&](int idx) { return at_x(idx, dxo, nxo, fo); };
  auto at_xe = [&](int idx) { return at_x(idx, dxe, nxe, fe); };
  auto at_yo = [&](int idx) { const int q = divq(idx, dw); return idx - q * w + w * (fy - r0 + 2 * q); };
  auto at_ye = [&](int idx) { const int q = divq(idx, dw); return idx - q * w + w * (ge - r0 + 2 * q); };
  int xo[K], xe[K], yo[K], ye[K];
  if constexpr (KEEP) {
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const int idx = tid + u * bd;
      xo[u] = idx < nxo * nE ? at_xo(idx) : -1, xe[u] = idx < nxe * nE ? at_xe(idx) : -1;
      yo[u] = idx < w * nyo ? at_yo(idx) : -1, ye[u] = idx < w * nye ? at_ye(idx) : -1;
    }
  }
  auto each = [&](const int *kept, int n, auto at, auto f) {
    if constexpr (KEEP) {
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (kept[u] >= 0) f(kept[u]);
    } else {
      for (int idx = tid; idx < n; idx += bd) {
        const int o = at(idx);
        if (o >= 0) f(o);
      }
    }
  };
  // G^a output: v[0] - sum_{t odd} K(t) v[t*stride]
  auto gsum = [](const E *v, int stride) {
    E s = v[0];
#pragma unroll
    for (int t = -ko; t <= ko; t += 2) s = D::acc(s, -W::K(t), v[t * stride]);
    return D::norm(s);
  };
  // rows r0-ko .. r1+ko of plane kk, columns c0-ko .. c0+w-1+ko, one row per warp
  auto stage = [&](int kk) {
    const bool kin = kk >= lo && kk <= hi;
    const TP *pk = Pb + (ptrdiff_t)(kk + Gi) * Wd * Wd + Gi;
    for (int x = tid & 31; x < wS; x += 32) {
      const int ii = c0 - ko + x;
      const bool cin = kin && ii >= lo && ii <= hi;
      for (int q = tid >> 5; q < nE; q += bd >> 5) {
        const int jr = row(q), jj = r0 - ko + jr;
        if (jr < 0 || jr >= nA) continue;
        S[jr * wS + x] = cin && jj >= lo && jj <= hi ? D::load(__ldg(pk + (jj + Gi) * Wd + ii)) : D::zero();
      }
    }
  };
  auto used = [&](int kk) { return kk <= z1 + ko && ((kk >= z0 && kk <= z1) || !(kk & 1)); };
  if (used(z0 - ko)) stage(z0 - ko);
  __syncthreads();
  int slot = 0;
  for (int kk = z0 - ko; kk <= z1 + ko + 1; ++kk, slot = slot + 1 == R ? 0 : slot + 1) {
    const bool in = used(kk);
    // x pass: odd columns, then even columns
    if (in) {
      each(xo, nxo * nE, at_xo, [&](int o) {
        const int jr = o >> 16, x = o & 0xffff;
        A[x + w * jr] = gsum(S + jr * wS + x + ko, 1);
      });
      __syncthreads();
      each(xe, nxe * nE, at_xe, [&](int o) {
        const int jr = o >> 16, x = o & 0xffff;
        E *a = A + x + w * jr;
        const E v = S[jr * wS + x + ko];
        if constexpr (NT != 0) *a = D::lift(v, a[-1], a[1]);
        else *a = v;
      });
      __syncthreads();
      // y pass into ring plane kk: odd rows, then even rows
      E *rp = ring + slot * pl;
      const E *Ay = A + w * ko;
      each(yo, w * nyo, at_yo, [&](int o) { rp[o] = gsum(Ay + o, w); });
      if (used(kk + 1)) stage(kk + 1);
      __syncthreads();
      each(ye, w * nye, at_ye, [&](int o) {
        E *r = rp + o;
        const E v = Ay[o];
        if constexpr (NT != 0) *r = D::lift(v, r[-w], r[w]);
        else *r = v;
      });
      __syncthreads();
    } else {
      if (used(kk + 1)) stage(kk + 1);
      __syncthreads();
    }
    // z: odd plane k1 = kk - ko (planes k1-ko .. k1+ko are in the ring), then
    // the even plane k1 - 1 from its ring plane and the odd planes around it
    const int k1 = kk - ko;
    if ((k1 & 1) && k1 >= z0 && k1 <= z1 + 1) {
      const int s1 = slot + ko + 1 >= R ? slot + ko + 1 - R : slot + ko + 1;  // ring slot of plane k1
      const int s0 = s1 == 0 ? R - 1 : s1 - 1, k0 = k1 - 1, par = ((k1 - fz) >> 1) & 1;
      E *d1 = dz + par * pl, *d0 = dz + (par ^ 1) * pl;
      int so[N];  // offsets of the N even planes around k1
#pragma unroll
      for (int x = 0; x < N; ++x) {
        int sl = s1 + 2 * x - ko;
        sl += sl < 0 ? R : 0;
        sl -= sl >= R ? R : 0;
        so[x] = sl * pl;
      }
      for (int idx = tid; idx < pl; idx += bd) {
        const int q = divq(idx, dw), i = c0 + idx - q * w, j = r0 + q;
        const bool mine = i >= B.lo[0] && i <= B.hi[0] && j >= B.lo[1] && j <= B.hi[1];
        const E *c = ring + idx;
        E v1 = D::zero();
        if (k1 <= z1) {
          v1 = c[s1 * pl];
#pragma unroll
          for (int x = 0; x < N; ++x) v1 = D::acc(v1, -W::K(2 * x - ko), c[so[x]]);
          v1 = D::norm(v1);
          if (NT) d1[idx] = v1;
          if (mine && k1 >= B.lo[2] && k1 <= B.hi[2]) emit(i, j, k1, v1);
        } else if (NT) {
          v1 = d1[idx];
        }
        if (k0 >= B.lo[2] && k0 <= B.hi[2] && mine) {
          E v = D::zero();
          if ((i | j) & 1) {
            v = c[s0 * pl];
            if constexpr (NT != 0) v = D::lift(v, d0[idx], v1);
          }
          emit(i, j, k0, v);
        }
      }
    }
  }
}

// column tiles of the extended region: tile q of nt is [i0, i1], cut before an
// odd column
__host__ __device__ __forceinline__ void det_cut(int r0, int r1, int q, int nt, int *i0, int *i1) {
  auto at = [&](int x) {
    const int c = r0 + x * (r1 - r0 + 1) / nt;
    return x == 0 ? r0 : x == nt ? r1 + 1 : c | 1;
  };
  *i0 = at(q), *i1 = at(q + 1) - 1;
}

// fewest tiles whose shared memory leaves room for two CTAs on an SM and whose
// passes (KEEP) have at most DET_ITEMS items per thread (24^3 with 6.2 in float pairs:
// 72 KB and 384 threads 2.64 ms, 110 KB and 512 threads 2.25 ms)
template <int N, int NT, bool KEEP>
static int det_tiles(int nb, size_t es, size_t *bytes) {
  const int r0 = -Wav<N, NT>::ext_f, r1 = nb - 1 + Wav<N, NT>::ext_b;
  for (int nt = 1;; ++nt) {
    int w = 0;
    for (int q = 0; q < nt; ++q) {
      int i0, i1;
      det_cut(r0, r1, q, nt, &i0, &i1);
      w = std::max(w, det_tile<NT>(i0, i1).w);
    }
    const int nR = r1 - r0 + 1, items = std::max(w * nR, (w + 1) / 2 * (nR + 2 * (N - 1)));
    *bytes = es * det_elems<N>(nR, w);
    if (*bytes <= DET_BYTES && (!KEEP || items <= DET_ITEMS * DET_THREADS)) return nt;
  }
}

// Per leaf: max |gamma| over the extended region (Sec. 2.3, the block norm
// that drives refinement and coarsening).  One CTA per column tile; the norms
// start at zero and take the maximum of the tiles' integer keys.
template <int N, int NT, bool PAIRS, bool KEEP>
__global__ void __launch_bounds__(1024, KEEP ? 1 : 2) k_criterion(int nb, const double *__restrict__ P, int Gi,
                                                                unsigned long long *__restrict__ maxdet, int ntile) {
  using E = typename DetOps<double, PAIRS>::E;
  const int b = blockIdx.x / ntile, Wd = nb + 2 * Gi;
  extern __shared__ double sm[];
  unsigned long long mx = 0;  // max |gamma| as an integer key (integer pipe)
  const int r0 = -Wav<N, NT>::ext_f, r1 = nb - 1 + Wav<N, NT>::ext_b;
  DetBox B{{r0, r0, r0}, {r1, r1, r1}};
  det_cut(r0, r1, blockIdx.x - b * ntile, ntile, &B.lo[0], &B.hi[0]);
  const double *Pb = P + (size_t)b * Wd * Wd * Wd;
  if constexpr (PAIRS) {
    // the largest pair by its high part's bits (a NaN above all), then its low
    // part; one conversion at the end
    unsigned kh = 0;
    float kl = 0.f;
    detail_planes<N, NT, PAIRS, KEEP, double>(Pb, nb, Gi, B, reinterpret_cast<E *>(sm), [&](int, int, int, F2 g) {
      const unsigned h = __float_as_uint(g.h) & 0x7fffffffu;
      const float l = g.h < 0.f ? -g.l : g.l;
      if (h > kh || (h == kh && l > kl)) kh = h, kl = l;
    });
    mx = abs_key(f2_dbl({__uint_as_float(kh), kl}));
  } else {
    detail_planes<N, NT, PAIRS, KEEP, double>(Pb, nb, Gi, B, reinterpret_cast<E *>(sm),
                                              [&](int, int, int, double g) { mx = max(mx, abs_key(g)); });
  }
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(maxdet + b, mx);
}

template <int N, int NT, bool PAIRS, bool KEEP>
static int criterion_launch(mr_grid *g, const double *P, int Gi, double *maxdet) {
  const int nb = g->desc.nb, n = g->nleaf;
  size_t sm;
  const int nt = det_tiles<N, NT, KEEP>(nb, sizeof(double), &sm);
  // (accepted are the block sizes whose untiled planes would fit an SM: of all,
  // 32^3 with 6.2 in float pairs is refused, although its tiles would fit)
  const int nR = nb + Wav<N, NT>::ext_f + Wav<N, NT>::ext_b, nA = nR + 2 * (N - 1);
  if (8 * ((size_t)(2 * N + 1) * nR * nR + (size_t)nR * nA + (PAIRS ? (size_t)nA * nA : 0)) > 227 * 1024)
    return MR_ERR_UNSUPPORTED;
  const auto kc = k_criterion<N, NT, PAIRS, KEEP>;
  if (smem_limit(kc, DET_BYTES, "criterion smem") ||
      check_cuda(cudaMemsetAsync(maxdet, 0, sizeof(double) * (size_t)n, g->stream), "criterion norms"))
    return MR_ERR_CUDA;
  unsigned long long *md = reinterpret_cast<unsigned long long *>(maxdet);
  // FP64: issue is limited by its own pipe, more warps hide its latency
  static const int cc[2] = {PAIRS ? DET_THREADS : 2 * DET_THREADS, PAIRS ? 2 * DET_THREADS : DET_THREADS};
  const int th = tune_threads(g, TuneKey{2, N, NT, nb, PAIRS ? 5 : 8, Gi, KEEP ? 0 : 4}, cc, 2, [&](int thr) {
    kc<<<n * nt, thr, sm, g->stream>>>(nb, P, Gi, md, nt);
  });
  MR_LAUNCH(g, MRK_CRITERION, kc<<<n * nt, th, sm, g->stream>>>(nb, P, Gi, md, nt));
  return check_cuda(cudaGetLastError(), "k_criterion") ? MR_ERR_CUDA : MR_OK;
}

template <int N, int NT>
static int criterion_impl(mr_grid *g, const double *P, int Gi, double *maxdet) {
  // FP32 grids evaluate the details in float pairs (FP32 pipe), FP64 grids in FP64.
  // There the kept indices cost 62 registers, one CTA of 1 024 threads to an SM: they
  // pay where every tile has an SM to itself (55 leaves of 24^3 with 6.2: 177 us
  // against 192), and two CTAs of 32 registers elsewhere (576 leaves: 1 451 against
  // 1 080 us; of 16^3 with 4.2 342 and 258; of 32^3 with 2.0, which the kept indices cut
  // into two tiles, 655 and 317).
  if (g->desc.precision == MR_F32) return criterion_launch<N, NT, true, true>(g, P, Gi, maxdet);
  size_t sm;
  return g->nleaf * det_tiles<N, NT, true>(g->desc.nb, sizeof(double), &sm) <= 152
             ? criterion_launch<N, NT, false, true>(g, P, Gi, maxdet)
             : criterion_launch<N, NT, false, false>(g, P, Gi, maxdet);
}

int launch_criterion(mr_grid *g, const double *P, int Gi, double *maxdet) {
  const int N = g->desc.wav_N, Nt = g->desc.wav_Nt;
#define MR_CCASE(n_, nt_) \
  if (N == n_ && Nt == nt_) return criterion_impl<n_, nt_>(g, P, Gi, maxdet);
  MR_CCASE(2, 0) MR_CCASE(2, 2) MR_CCASE(4, 0) MR_CCASE(4, 2) MR_CCASE(6, 0) MR_CCASE(6, 2)
#undef MR_CCASE
  return MR_ERR_UNSUPPORTED;
}

// --------------------------------------------------------- status, policy
__global__ void k_status(int n, const double *maxdet, double er, double ec, int flags, const int *lev,
                         const int *refined, int lmin, int lmax, int8_t *st) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const double m = maxdet[b];
  int s = m >= er ? ST_FINER : (m <= ec ? ST_COARSER : ST_SAME);
  if (s == ST_FINER && !(flags & MR_ADAPT_REFINE)) s = ST_SAME;
  if (s == ST_COARSER && !(flags & MR_ADAPT_COARSEN)) s = ST_SAME;
  const int L = lev[b];
  if (s == ST_FINER && L >= lmax) s = ST_SAME;
  if (s == ST_COARSER && (L <= lmin || L == 0 || refined[b])) s = ST_SAME;
  st[b] = (int8_t)s;
}

// One Jacobi sweep of the policy rules (monotone: statuses only rise, so the
// sweeps converge to the same least fixed point as any other order).
__global__ void k_policy(Tree t, const int8_t *__restrict__ sin, int8_t *__restrict__ sout, int *changed) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= t.nleaf) return;
  const int L = __ldg(t.lev + b), nb = t.nb;
  const int s = sin[b];
  int ns = s;
  const bool fin = L < t.M;
  const int Ls = fin ? L + 1 : L, span = fin ? 2 * nb : nb;
  int base[3];
  for (int d = 0; d < 3; ++d) base[d] = __ldg(t.anc + 3 * b + d) * span;
  bool raise = false, cancel = false;
  for (int m = 0; m < 27; ++m) {
    if (m == 13) continue;
    const int dd[3] = {m % 3 - 1, (m / 3) % 3 - 1, m / 9 - 1};
    const int c0 = dd[0] ? 1 : 2, c1 = dd[1] ? 1 : 2, c2 = dd[2] ? 1 : 2;
    for (int cz = 0; cz < c2; ++cz)
      for (int cy = 0; cy < c1; ++cy)
        for (int cx = 0; cx < c0; ++cx) {
          const int cc[3] = {cx, cy, cz};
          int g[3];
          for (int d = 0; d < 3; ++d)
            g[d] = dd[d] < 0 ? base[d] - 1 : dd[d] > 0 ? base[d] + span : base[d] + cc[d] * (span / 2);
          if (beyond3(t, Ls, g)) continue;  // no neighbour beyond a physical boundary
          const int o = owner(t, Ls, g[0], g[1], g[2], b);
          if (o == b) continue;
          const int Lo = __ldg(t.lev + o), so = sin[o];
          if (Lo > L && so == ST_FINER) raise = true;
          if (Lo > L || (Lo == L && so == ST_FINER)) cancel = true;
        }
  }
  if (s != ST_FINER && raise) ns = ST_FINER;
  if (ns == ST_COARSER) {
    if (cancel) ns = ST_SAME;
    for (int c = 0; c < 8 && ns == ST_COARSER; ++c) {
      int a[3];
      for (int d = 0; d < 3; ++d) a[d] = (__ldg(t.anc + 3 * b + d) & ~1) + ((c >> d) & 1);
      const int o = owner(t, L, a[0] * nb, a[1] * nb, a[2] * nb, b);
      const bool leaf = __ldg(t.lev + o) == L && __ldg(t.anc + 3 * o) == a[0] &&
                        __ldg(t.anc + 3 * o + 1) == a[1] && __ldg(t.anc + 3 * o + 2) == a[2];
      if (!leaf || sin[o] != ST_COARSER) ns = ST_SAME;
    }
  }
  sout[b] = (int8_t)ns;
  if (ns != s) atomicAdd(changed, 1);
}

// ------------------------------------------------------------ new tree
__global__ void k_count(int n, const int8_t *st, const int *anc, int *cnt, int *changed) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const int s = st[b];
  int c = 1;
  if (s == ST_FINER) c = 8;
  if (s == ST_COARSER) c = ((anc[3 * b] | anc[3 * b + 1] | anc[3 * b + 2]) & 1) ? 0 : 1;
  cnt[b] = c;
  if (s != ST_SAME) atomicAdd(changed, 1);
}

// exclusive scan of cnt[0..n) in place, total in cnt[n]; one CTA of 1024
__global__ void __launch_bounds__(1024) k_scan(int *cnt, int n) {
  __shared__ int part[1024];
  const int chunk = (n + 1023) / 1024;
  const int beg = threadIdx.x * chunk, end = min(n, beg + chunk);
  int s = 0;
  for (int i = beg; i < end; ++i) s += cnt[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int run = part[threadIdx.x] - s;
  for (int i = beg; i < end; ++i) {
    const int c = cnt[i];
    cnt[i] = run;
    run += c;
  }
  if (threadIdx.x == 1023) cnt[n] = part[1023];
}

__device__ unsigned long long morton_key_dev(int lev, int ax, int ay, int az, int M) {
  const unsigned long long x = (unsigned long long)ax << (M - lev), y = (unsigned long long)ay << (M - lev),
                           z = (unsigned long long)az << (M - lev);
  unsigned long long key = 0;
  for (int bit = 0; bit < 19; ++bit) {
    key |= ((x >> bit) & 1ULL) << (3 * bit);
    key |= ((y >> bit) & 1ULL) << (3 * bit + 1);
    key |= ((z >> bit) & 1ULL) << (3 * bit + 2);
  }
  return (key << 5) | (unsigned long long)lev;
}

__global__ void k_emit(int n, int M, const int8_t *st, const int *pos, const int *lev, const int *anc,
                       const int *refined, int *nlev, int *nanc, unsigned long long *nkey, int *nref,
                       int *src) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  const int s = st[b], p = pos[b], L = lev[b];
  const int a0 = anc[3 * b], a1 = anc[3 * b + 1], a2 = anc[3 * b + 2];
  if (s == ST_FINER) {
    for (int c = 0; c < 8; ++c) {
      const int q = p + c;
      const int x = 2 * a0 + (c & 1), y = 2 * a1 + ((c >> 1) & 1), z = 2 * a2 + (c >> 2);
      nlev[q] = L + 1;
      nanc[3 * q] = x, nanc[3 * q + 1] = y, nanc[3 * q + 2] = z;
      nkey[q] = morton_key_dev(L + 1, x, y, z, M);
      nref[q] = 1;
      src[2 * q] = KIND_CHILD;
      src[2 * q + 1] = (b << 3) | c;
    }
  } else if (s == ST_COARSER) {
    if ((a0 | a1 | a2) & 1) return;
    nlev[p] = L - 1;
    nanc[3 * p] = a0 / 2, nanc[3 * p + 1] = a1 / 2, nanc[3 * p + 2] = a2 / 2;
    nkey[p] = morton_key_dev(L - 1, a0 / 2, a1 / 2, a2 / 2, M);
    nref[p] = 0;
    src[2 * p] = KIND_PARENT;
    src[2 * p + 1] = b;
  } else {
    nlev[p] = L;
    nanc[3 * p] = a0, nanc[3 * p + 1] = a1, nanc[3 * p + 2] = a2;
    nkey[p] = morton_key_dev(L, a0, a1, a2, M);
    nref[p] = refined[b];
    src[2 * p] = KIND_COPY;
    src[2 * p + 1] = b;
  }
}

// ------------------------------------------------------ interpolation
// New leaf values: copy, zero-detail refinement of the parent's padded block
// (J^s / K^s), or tensor H^a coarsening of the 8 children's padded blocks, in
// the padded blocks' precision TP.  Both sums are separable and run along
// lines (wavelet_runs.cuh): 3 x 6 taps per child point at most instead of up
// to 216 (43 on average with 6.x), 3 x 9 per parent point instead of 729.
// Bound by shared-memory and issue slots; remeshing about 6 000 leaves of 24^3
// with 6.2 and four fields spent 36 ms here with tensor sums per point, 4.3 ms now.

// z-planes of a child per step, and the shared memory of its two passes
constexpr int INTERP_Z = 8;
static size_t interp_smem(int N, int nb, size_t es) {
  const size_t m = nb / 2 + N - 1;
  return es * INTERP_Z * (m * (m | 1) + (size_t)nb * (m | 1));
}
// sums of four layers of a new parent's octant (fine extent: a child's and the H^a half-widths)
static size_t parent_smem(int hH, int nb, size_t es) {
  const size_t fw = nb - 1 + 2 * hH;
  return es * 4 * fw * (fw + nb / 2);
}

template <typename TO, typename TP, int N, int NT>
__global__ void __launch_bounds__(256) k_interp(int nb, const int *__restrict__ src, const TP *__restrict__ P, int Gi,
                                                const TO *__restrict__ fold, TO *__restrict__ fnew) {
  using RS = RefSum<TP, TP>;
  constexpr int h = N / 2;
  const int q = blockIdx.x, Wd = nb + 2 * Gi, W2 = Wd * Wd, hb = nb / 2, tid = threadIdx.x, bd = blockDim.x;
  const size_t nb3 = (size_t)nb * nb * nb, np = (size_t)Wd * W2;
  const int kind = src[2 * q], s = src[2 * q + 1];
  TO *out = fnew + (size_t)q * nb3;
  if (kind == KIND_COPY) {
    const float4 *f4 = reinterpret_cast<const float4 *>(fold + (size_t)s * nb3);  // nb^3 is a multiple of 8
    float4 *o4 = reinterpret_cast<float4 *>(out);
    const int n4 = (int)(nb3 * sizeof(TO) / 16);
#pragma unroll 4
    for (int p = tid; p < n4; p += bd) o4[p] = __ldg(f4 + p);
    return;
  }
  if (kind != KIND_CHILD) return;  // parents: k_interp_parent
  const int ch = s & 7;
  const int cx = (ch & 1) * hb, cy = ((ch >> 1) & 1) * hb, cz = (ch >> 2) * hb;  // child's first coarse point
  const TP *Pp = P + (size_t)(s >> 3) * np + Gi * (1 + Wd + (size_t)W2);
  extern __shared__ double smi[];
  const int m = hb + N - 1, mp = m | 1;        // coarse points per axis the child reads; pitch
  TP *U1 = reinterpret_cast<TP *>(smi);        // [z][m][mp]: refined along z
  TP *U2 = U1 + INTERP_Z * m * mp;             // [z][nb][mp]: and along y
  const DivM dm = divm(m), dh = divm(hb), dnb = divm(nb);
  const int nseg = (nb + 15) >> 4;
  const DivM dl = divm(INTERP_Z * m);
  for (int z0 = 0; z0 < nb; z0 += INTERP_Z) {
    const int nz = min(INTERP_Z, nb - z0);
    for (int idx = tid; idx < m * m; idx += bd) {
      const int jy = divq(idx, dm), jx = idx - jy * m;
      TP *d = U1 + jx + mp * jy;
      refine_run<N, NT, RS>(Pp + (cx - h + 1 + jx) + Wd * (cy - h + 1 + jy), W2, 2 * cz + z0, nz,
                            [&](int z, TP v) { d[z * m * mp] = v; });
    }
    __syncthreads();
    for (int idx = tid; idx < INTERP_Z * m * nseg; idx += bd) {
      const int sg = divq(idx, dl), l = idx - sg * INTERP_Z * m, z = divq(l, dm), jx = l - z * m;
      if (z >= nz) continue;
      // (U1's row jy holds coarse point cy - h + 1 + jy)
      const TP *r = U1 + z * m * mp + jx - (ptrdiff_t)(cy - h + 1) * mp;
      TP *d = U2 + z * nb * mp + 16 * sg * mp + jx;
      refine_run<N, NT, RS>(r, mp, 2 * cy + 16 * sg, min(16, nb - 16 * sg), [&](int y, TP v) { d[y * mp] = v; });
    }
    __syncthreads();
    // along x: one thread per (even, odd) pair, neighbouring threads write
    // neighbouring points
    for (int idx = tid; idx < nz * nb * hb; idx += bd) {
      const int r = divq(idx, dh), px = idx - r * hb;  // r = y + nb z
      const TP *w = U2 + r * mp + px;
      TP v = TP(0);
#pragma unroll
      for (int x = 0; x < N; ++x) v = racc(v, TP(Wav<N, NT>::K(2 * x - (N - 1))), w[x]);
      TO *o = out + (size_t)(z0 * nb + r) * nb + 2 * px;
      o[0] = TO(w[h - 1]);
      o[1] = TO(v);
    }
    __syncthreads();
  }
}

// One CTA per octant of a new parent: the child leaf's block coarsened.
template <typename TO, typename TP, int N, int NT>
__global__ void __launch_bounds__(256) k_interp_parent(Tree to, const int *__restrict__ src, const TP *__restrict__ P,
                                                       int Gi, TO *__restrict__ fnew, int cap) {
  const int q = blockIdx.x >> 3, c = blockIdx.x & 7, nb = to.nb, Wd = nb + 2 * Gi, hb = nb / 2;
  if (src[2 * q] != KIND_PARENT) return;
  // s: the new parent's first child in the old tree (level L = parent level + 1)
  const int s = src[2 * q + 1], L = __ldg(to.lev + s);
  int a[3];
  for (int d = 0; d < 3; ++d) a[d] = (__ldg(to.anc + 3 * s + d) + ((c >> d) & 1)) * nb;
  const int o = owner(to, L, a[0], a[1], a[2], s);
  TO *out = fnew + (size_t)q * nb * nb * nb + hb * ((c & 1) + nb * (((c >> 1) & 1) + (size_t)nb * (c >> 2)));
  extern __shared__ double smi[];
  const int lo[3] = {0, 0, 0}, hi[3] = {hb, hb, hb};
  coarsen_box<N, NT, TP>(P + (size_t)o * Wd * Wd * Wd + Gi * (1 + Wd + (size_t)Wd * Wd), Wd, lo, hi,
                         reinterpret_cast<TP *>(smi), cap,
                         [&](int x, int y, int z, TP v) { out[x + nb * (y + nb * z)] = TO(v); });
}

// ------------------------------------------------------------- update

// Directions of newly coarsened neighbours (one level coarser) of unchanged
// new leaves; 0 for other leaves.
__global__ void k_newmask(Tree tn, const int *src, int *nmask) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= tn.nleaf) return;
  int mask = 0;
  if (src[2 * q] == KIND_COPY) {
    const int L = __ldg(tn.lev + q), nb = tn.nb;
    for (int m = 0; m < 27; ++m) {
      if (m == 13) continue;
      const int dd[3] = {m % 3 - 1, (m / 3) % 3 - 1, m / 9 - 1};
      int g[3];
      for (int d = 0; d < 3; ++d) g[d] = __ldg(tn.anc + 3 * q + d) * nb + (dd[d] < 0 ? -1 : dd[d] > 0 ? nb : 0);
      if (beyond3(tn, L, g)) continue;
      const int o = owner(tn, L, g[0], g[1], g[2], q);
      if (__ldg(tn.lev + o) == L - 1 && src[2 * o] == KIND_PARENT) mask |= 1 << m;
    }
  }
  nmask[q] = mask;
}

// A leaf's box of discarded details, packed: per axis the first and last pair of
// points of the extended region (5 bits each; 43 points at most), bit 30 set.
__device__ __forceinline__ int box_pack(const int *lo, const int *hi, int r0) {
  int p = 1 << 30;
  for (int d = 0; d < 3; ++d) p |= ((lo[d] - r0) >> 1) << (10 * d) | ((hi[d] - r0) >> 1) << (10 * d + 5);
  return p;
}
__device__ __forceinline__ DetBox box_unpack(int p, int r0, int r1) {
  DetBox B;
  for (int d = 0; d < 3; ++d)
    B.lo[d] = r0 + 2 * ((p >> (10 * d)) & 31), B.hi[d] = min(r0 + 2 * ((p >> (10 * d + 5)) & 31) + 1, r1);
  return B;
}

// gamma for the details the coarsening discarded (in newly coarsened leaves, or
// in the new bands of F or of its unchanged same-level neighbours) of every
// unchanged leaf F, over the box of the extended region that holds them; 0 at
// the box's other points.  Q is indexed by F's old slot in the padded layout.
// The 27 block-sized regions around F are classified once: a newly coarsened
// leaf one level coarser owns all of D in its region, an unchanged same-level
// leaf with newly coarsened neighbours owns the part of its band next to them,
// finer leaves none.  Most leaves discard next to one face, so the box is a
// third of the region or less (the two update kernels together: 40.4 ms over
// the whole region, 12.3 ms over the boxes, in that remeshing); the box goes to
// hasD (0: nothing discarded).
template <typename TP, int N, int NT>
__global__ void __launch_bounds__(DET_THREADS, sizeof(TP) == 4 ? 3 : 2) k_update_gamma(
    Tree tn, const int *__restrict__ src, const int *__restrict__ nmask, const TP *__restrict__ P, int Gi,
    TP *__restrict__ Q, int *hasD, int cap) {
  using W = Wav<N, NT>;
  const int q = blockIdx.x;
  if (src[2 * q] != KIND_COPY) return;
  const int s = src[2 * q + 1], L = __ldg(tn.lev + q), nb = tn.nb, Wd = nb + 2 * Gi;
  const int ef = W::ext_f, eb = W::ext_b, r0 = -ef, r1 = nb - 1 + eb;
  const size_t np = (size_t)Wd * Wd * Wd;
  __shared__ int rD[27], blo[3], bhi[3];
  if (threadIdx.x < 3) blo[threadIdx.x] = 1 << 20, bhi[threadIdx.x] = -(1 << 20);
  __syncthreads();
  if (threadIdx.x < 27) {
    const int r = threadIdx.x;
    const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
    int g[3];
    for (int d = 0; d < 3; ++d) g[d] = __ldg(tn.anc + 3 * q + d) * nb + (dd[d] < 0 ? -1 : dd[d] > 0 ? nb : 0);
    int v = 0;  // regions beyond a physical boundary hold no details
    if (!beyond3(tn, L, g)) {
      const int o = owner(tn, L, g[0], g[1], g[2], q);
      const int Lo = __ldg(tn.lev + o), ko = src[2 * o];
      if (Lo == L - 1 && ko == KIND_PARENT) v = -1;
      else if (Lo == L && ko == KIND_COPY) v = nmask[o];
    }
    rD[r] = v;
    // box of D in this region: all of it, or the band next to each new neighbour m
    for (int m = v == -1 ? 13 : 0; v && m < (v == -1 ? 14 : 27); ++m) {
      if (v > 0 && !((v >> m) & 1)) continue;
      const int md[3] = {m % 3 - 1, (m / 3) % 3 - 1, m / 9 - 1};
      int lo[3], hi[3];
      bool some = true;
      for (int d = 0; d < 3; ++d) {
        lo[d] = max(dd[d] * nb + (md[d] > 0 ? nb - ef : 0), r0);
        hi[d] = min(dd[d] * nb + (md[d] < 0 ? eb : nb) - 1, r1);
        some &= lo[d] <= hi[d];
      }
      if (some)
        for (int d = 0; d < 3; ++d) atomicMin(&blo[d], lo[d]), atomicMax(&bhi[d], hi[d]);
    }
  }
  __syncthreads();
  if (blo[0] > bhi[0]) {
    if (threadIdx.x == 0) hasD[q] = 0;
    return;
  }
  const int packed = box_pack(blo, bhi, r0);
  if (threadIdx.x == 0) hasD[q] = packed;
  TP *Qb = Q + (size_t)s * np;
  extern __shared__ double smd[];
  const DetBox B = box_unpack(packed, r0, r1);
  // column tiles whose passes fit in shared memory and the threads' items
  const int nR = det_tile<NT>(B.lo[1], B.hi[1]).w;
  int wm = min(DET_ITEMS * DET_THREADS / nR, 2 * DET_ITEMS * DET_THREADS / (nR + 2 * (N - 1)) - 1);
  while ((int)det_elems<N>(nR, wm) > cap) --wm;
  const int step = max((wm - 1) & ~1, 2);  // (even: tiles start at the box's parity; one column more is computed)
  for (int c = B.lo[0]; c <= B.hi[0]; c += step) {
    DetBox T = B;
    T.lo[0] = c, T.hi[0] = min(c + step - 1, B.hi[0]);
    if (c != B.lo[0]) __syncthreads();
    detail_planes<N, NT, false, true, TP>(P + (size_t)s * np, nb, Gi, T, reinterpret_cast<TP *>(smd),
                                    [&](int i, int j, int k, TP g) {
      if ((i | j | k) & 1) {
        const int r = region_of(i, j, k, nb), v = rD[r];
        bool inD = v == -1;
        if (v > 0) {
          const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
          inD = in_band_dev(v, i - dd[0] * nb, j - dd[1] * nb, k - dd[2] * nb, nb, ef, eb);
        }
        if (!inD) g = TP(0);
      }
      Qb[(size_t)(i + Gi) + Wd * ((size_t)(j + Gi) + (size_t)Wd * (k + Gi))] = g;
    });
  }
}

// Subtract the synthesis of the discarded details (the J^s / K^s tensor taps
// of the zero-detail refinement's complement) from the unchanged leaf, over the
// points within reach of its box of details: separable, x then y then z, with
// the y-pass planes in a ring of 2*hw(K^s)+1 shared-memory planes.  gamma is
// zero outside the box.
template <typename TO, typename TP, int N, int NT>
__global__ void __launch_bounds__(256) k_update_apply(int nb, const int *__restrict__ src,
                                                      const int *__restrict__ hasD,
                                                      const TP *__restrict__ Q, int Gi,
                                                      TO *__restrict__ fnew) {
  using W = Wav<N, NT>;
  constexpr int hk = W::hwK, R = 2 * hk + 1;
  const int q = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  if (src[2 * q] != KIND_COPY || !hasD[q]) return;
  const int s = src[2 * q + 1], Wd = nb + 2 * Gi;
  const DetBox B = box_unpack(hasD[q], -W::ext_f, nb - 1 + W::ext_b);
  int o0[3], on[3];  // output points
  for (int d = 0; d < 3; ++d) {
    o0[d] = max(B.lo[d] - hk, 0);
    on[d] = min(B.hi[d] + hk, nb - 1) - o0[d] + 1;
  }
  if (on[0] <= 0 || on[1] <= 0 || on[2] <= 0) return;
  const int bx0 = B.lo[0], bx1 = B.hi[0], by0 = B.lo[1], by1 = B.hi[1], bz0 = B.lo[2], bz1 = B.hi[2];
  const int nx = on[0], pl = nx * on[1], ny = by1 - by0 + 1;
  const TP *Qb = Q + (size_t)s * Wd * Wd * Wd;
  TO *v = fnew + (size_t)q * nb * nb * nb;
  extern __shared__ double smd[];
  TP *ring = reinterpret_cast<TP *>(smd);  // [R][on1][nx]
  TP *X = ring + (size_t)R * pl;           // [ny][nx]: x pass of one plane
  const int xo = par_first(o0[0], 1), xe = par_first(o0[0], 0), nxo = par_count(o0[0], o0[0] + nx, 1), nxe = nx - nxo;
  const DivM dxo = divm(max(nxo, 1)), dxe = divm(max(nxe, 1)), dx = divm(nx);
  int slot = 0;
  for (int kk = bz0; kk <= min(bz1 + hk, nb - 1) + hk; ++kk, slot = slot + 1 == R ? 0 : slot + 1) {
    if (kk <= bz1) {
      // odd columns (K^s) first, then even ones (J^s): one filter per warp
      for (int idx = tid; idx < nx * ny; idx += bd) {
        const bool od = idx < nxo * ny;
        const int p0 = od ? idx : idx - nxo * ny, r = divq(p0, od ? dxo : dxe);
        const int i = (od ? xo : xe) + 2 * (p0 - r * (od ? nxo : nxe)), jj = by0 + r;
        const TP *p = Qb + (i + Gi) + Wd * ((jj + Gi) + (size_t)Wd * (kk + Gi));
        auto at = [&](int t) { return (i + t >= bx0 && i + t <= bx1) ? p[t] : TP(0); };
        TP a = TP(0);
        if (od)
          for_taps<N, NT, FK_K>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        else
          for_taps<N, NT, FK_J>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        X[i - o0[0] + nx * r] = a;
      }
      __syncthreads();
      for (int idx = tid; idx < pl; idx += bd) {
        const int r = divq(idx, dx), x = idx - r * nx, j = o0[1] + r;
        auto at = [&](int t) { return (j + t >= by0 && j + t <= by1) ? X[x + nx * (j + t - by0)] : TP(0); };
        TP a = TP(0);
        if (j & 1)
          for_taps<N, NT, FK_K>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        else
          for_taps<N, NT, FK_J>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        ring[slot * pl + idx] = a;
      }
    }
    __syncthreads();
    // output plane k = kk - hk: its taps k+t with t in [-hk, hk] are planes
    // kk-2hk .. kk, all in the ring (planes outside the box read as 0)
    const int k = kk - hk;
    if (k >= 0 && k < nb) {
      const int sk = slot + hk + 1 >= R ? slot + hk + 1 - R : slot + hk + 1;
      for (int idx = tid; idx < pl; idx += bd) {
        auto at = [&](int t) {
          if (k + t < bz0 || k + t > bz1) return TP(0);
          int sl = sk + t;
          sl += sl < 0 ? R : 0;
          sl -= sl >= R ? R : 0;
          return ring[sl * pl + idx];
        };
        TP a = TP(0);
        if (k & 1)
          for_taps<N, NT, FK_K>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        else
          for_taps<N, NT, FK_J>([&](int t, double w) { a = racc(a, TP(w), at(t)); });
        const int r = divq(idx, dx);
        const size_t p = (size_t)(o0[0] + idx - r * nx) + nb * (o0[1] + r + (size_t)nb * k);
        if (a != TP(0)) v[p] = TO(Cvt<TP>::f(v[p]) - a);
      }
    }
    __syncthreads();
  }
}

template <int N, int NT>
static size_t apply_smem(int nb, size_t es) {
  using W = Wav<N, NT>;
  const int nR = nb + W::ext_f + W::ext_b;
  return es * ((size_t)(2 * W::hwK + 1) * nb * nb + (size_t)nR * nb);
}

// ------------------------------------------------- fields needing ghosts
// Leaves touching b across a face, edge or corner (one probe per adjacent
// level-(L+1) cell; finer neighbours are at most one level finer).
template <typename F>
__device__ __forceinline__ void for_each_nbr(const Tree &t, int b, F f) {
  const int L = __ldg(t.lev + b), nb = t.nb;
  const bool fin = L < t.M;
  const int Ls = fin ? L + 1 : L, span = fin ? 2 * nb : nb;
  int base[3];
  for (int d = 0; d < 3; ++d) base[d] = __ldg(t.anc + 3 * b + d) * span;
  for (int m = 0; m < 27; ++m) {
    if (m == 13) continue;
    const int dd[3] = {m % 3 - 1, (m / 3) % 3 - 1, m / 9 - 1};
    const int c0 = dd[0] ? 1 : 2, c1 = dd[1] ? 1 : 2, c2 = dd[2] ? 1 : 2;
    for (int cz = 0; cz < c2; ++cz)
      for (int cy = 0; cy < c1; ++cy)
        for (int cx = 0; cx < c0; ++cx) {
          const int cc[3] = {cx, cy, cz};
          int g[3];
          for (int d = 0; d < 3; ++d)
            g[d] = dd[d] < 0 ? base[d] - 1 : dd[d] > 0 ? base[d] + span : base[d] + cc[d] * (span / 2);
          if (beyond3(t, Ls, g)) continue;
          const int o = owner(t, Ls, g[0], g[1], g[2], b);
          if (o != b) f(o);
        }
  }
}

// ring 1: a neighbour changes level
__global__ void k_need1(Tree t, const int8_t *st, int *nb1) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= t.nleaf) return;
  int any = 0;
  for_each_nbr(t, b, [&](int o) { any |= st[o] != ST_SAME; });
  nb1[b] = any;
}

// ring 2: the leaf changes, or a neighbour does, or a neighbour's neighbour
// (whose new substitution band can lie within this leaf's update reach)
__global__ void k_need2(Tree t, const int8_t *st, const int *nb1, int *need) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= t.nleaf) return;
  int any = st[b] != ST_SAME || nb1[b];
  if (!any) for_each_nbr(t, b, [&](int o) { any |= nb1[o]; });
  need[b] = any;
}

// finer neighbours of needed leaves push the fine-to-coarse ghost values the
// needed leaves read: the needed leaves and those finer neighbours
__global__ void k_need3(Tree t, const int *need, int *need2) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= t.nleaf) return;
  const int L = __ldg(t.lev + b);
  int any = need[b];
  if (!any) for_each_nbr(t, b, [&](int o) { any |= __ldg(t.lev + o) < L && need[o]; });
  need2[b] = any;
}

// ------------------------------------------------------------- driver
static Tree next_view(const mr_grid *g, int nleaf) {
  Tree t = tree_view(g);
  const int nx = g->cur ^ 1;
  t.lev = g->lev[nx];
  t.anc = g->anc[nx];
  t.map = g->maps[nx];
  t.nleaf = nleaf;
  return t;
}

// interpolation and update of field fid from its padded blocks P (type TP;
// the update's details go to the FP64 side buffer's memory in type TP)
template <typename TO, typename TP, int N, int NT>
static int interp_update(mr_grid *g, const Tree &to, const Tree &tn, const TP *P, int Gi, int fid,
                         int *nmask, int *hasD) {
  const int *src = g->newsrc;
  TP *Q = reinterpret_cast<TP *>(g->padQ64);
  const int tp = sizeof(TP) == 4 ? 4 : sizeof(TO) == 4 ? 5 : 8;
  const int nb = g->desc.nb;
  const size_t smi = interp_smem(N, nb, sizeof(TP));
  constexpr int hH = Wav<N, NT>::hwH;
  const size_t smp = parent_smem(hH, nb, sizeof(TP));
  const auto ki = k_interp<TO, TP, N, NT>;
  const auto kp = k_interp_parent<TO, TP, N, NT>;
  if (smem_limit(ki, interp_smem(N, MAX_NB, sizeof(TP)), "interp smem") ||
      smem_limit(kp, parent_smem(hH, MAX_NB, sizeof(TP)), "interp smem"))
    return MR_ERR_CUDA;
  const TO *fo = (const TO *)field_ptr(g, fid);
  TO *fn = (TO *)next_field_ptr(g, fid);
  static const int ci[2] = {256, 128};
  const int thi = tune_threads(g, TuneKey{4, N, NT, nb, tp, Gi, 0}, ci, 2, [&](int th) {
    ki<<<tn.nleaf, th, smi, g->stream>>>(nb, src, P, Gi, fo, fn);
  });
  MR_LAUNCH(g, MRK_INTERP, ki<<<tn.nleaf, thi, smi, g->stream>>>(nb, src, P, Gi, fo, fn));
  MR_LAUNCH(g, MRK_INTERP, kp<<<8 * tn.nleaf, 256, smp, g->stream>>>(to, src, P, Gi, fn, (int)(smp / sizeof(TP))));
  const size_t smg = sizeof(TP) == 4 ? 72 * 1024 : 110 * 1024;  // three / two CTAs of 512 threads per SM
  const size_t sma = apply_smem<N, NT>(nb, sizeof(TP));
  if (sma > MAX_SMEM) return MR_ERR_UNSUPPORTED;
  if (smem_limit(k_update_gamma<TP, N, NT>, smg, "update smem") ||
      smem_limit(k_update_apply<TO, TP, N, NT>, std::min(apply_smem<N, NT>(MAX_NB, sizeof(TP)), MAX_SMEM),
                 "update smem"))
    return MR_ERR_CUDA;
  MR_LAUNCH(g, MRK_UPDATE, k_update_gamma<TP, N, NT><<<tn.nleaf, DET_THREADS, smg, g->stream>>>(
                               tn, src, nmask, P, Gi, Q, hasD, (int)(smg / sizeof(TP))));
  MR_LAUNCH(g, MRK_UPDATE, k_update_apply<TO, TP, N, NT><<<tn.nleaf, 256, sma, g->stream>>>(
                               nb, src, hasD, Q, Gi, fn));
  return check_cuda(cudaGetLastError(), "interp/update") ? MR_ERR_CUDA : MR_OK;
}

template <typename TO, typename TP>
static int interp_dispatch(mr_grid *g, const Tree &to, const Tree &tn, const TP *P, int Gi, int fid,
                           int *nmask, int *hasD) {
  const int N = g->desc.wav_N, Nt = g->desc.wav_Nt;
#define MR_ICASE(n_, nt_) \
  if (N == n_ && Nt == nt_) return interp_update<TO, TP, n_, nt_>(g, to, tn, P, Gi, fid, nmask, hasD);
  MR_ICASE(2, 0) MR_ICASE(2, 2) MR_ICASE(4, 0) MR_ICASE(4, 2) MR_ICASE(6, 0) MR_ICASE(6, 2)
#undef MR_ICASE
  return MR_ERR_UNSUPPORTED;
}

static int read_ints(mr_grid *g, const int *dev, int *host, int n) {
  if (check_cuda(cudaMemcpyAsync(host, dev, sizeof(int) * n, cudaMemcpyDeviceToHost, g->stream), "readback"))
    return MR_ERR_CUDA;
  return check_cuda(cudaStreamSynchronize(g->stream), "readback sync") ? MR_ERR_CUDA : MR_OK;
}

int adapt_iteration(mr_grid *g, int crit, double er, double ec, int flags, int *nch) {
  *nch = 0;
  const int n = g->nleaf, G = adapt_shell(g->desc.wav_N, g->desc.wav_Nt);
  cudaStream_t st = g->stream;
  void *Pv;
  int Gi;
  // 1-2: ghosts of the criterion field, block criterion
  int e = launch_ghost(g, field_ptr(g, crit), field_ptr(g, crit), G, true, &Pv, &Gi);
  if (e) return e;
  const double *P = (const double *)Pv;
  // grids with physical boundaries take the bounded criterion, and full ghost
  // fills (with write-back) of every field
  const bool bnd = grid_bounded(g);
  e = bnd ? launch_criterion_bounded(g, P, Gi, g->maxdet) : launch_criterion(g, P, Gi, g->maxdet);
  if (e) return e;
  // the norms this iteration decides with (mr_last_block_norms)
  if (check_cuda(cudaMemcpyAsync(g->mdlast, g->maxdet, sizeof(double) * (size_t)n, cudaMemcpyDeviceToDevice, st),
                 "block norms copy"))
    return MR_ERR_CUDA;
  g->nleaf_last = n;
  // 3-4: status and policy
  Tree t = tree_view(g);
  const int tb = 128, nblk = (n + tb - 1) / tb;
  MR_LAUNCH(g, MRK_STATUS, k_status<<<nblk, tb, 0, st>>>(n, g->maxdet, er, ec, flags, g->lev[g->cur], g->refined,
                                                         g->desc.lmin, g->desc.lmax, g->status));
  int8_t *sa = g->status, *sb = (int8_t *)g->newsrc;
  int it = 0;
  for (;; ++it) {
    if (it >= g->max_policy_sweeps) {
      set_error("policy did not reach a fixed point within the sweep limit");
      return MR_ERR_TIMEOUT;
    }
    if (check_cuda(cudaMemsetAsync(g->counter, 0, sizeof(int), st), "memset")) return MR_ERR_CUDA;
    MR_LAUNCH(g, MRK_POLICY, k_policy<<<nblk, tb, 0, st>>>(t, sa, sb, g->counter));
    int changed;
    e = read_ints(g, g->counter, &changed, 1);
    if (e) return e;
    int8_t *tmp = sa;
    sa = sb, sb = tmp;
    if (!changed) break;
  }
  if (sa != g->status &&
      check_cuda(cudaMemcpyAsync(g->status, sa, n, cudaMemcpyDeviceToDevice, st), "status copy"))
    return MR_ERR_CUDA;
  // 5: new tree
  if (check_cuda(cudaMemsetAsync(g->counter, 0, sizeof(int), st), "memset")) return MR_ERR_CUDA;
  MR_LAUNCH(g, MRK_SCAN, k_count<<<nblk, tb, 0, st>>>(n, g->status, g->anc[g->cur], g->scan, g->counter));
  MR_LAUNCH(g, MRK_SCAN, k_scan<<<1, 1024, 0, st>>>(g->scan, n));
  int hc[2];
  e = read_ints(g, g->counter, &hc[0], 1);
  if (!e) e = read_ints(g, g->scan + n, &hc[1], 1);
  if (e) return e;
  const int changed = hc[0], nn = hc[1];
  if (check_cuda(cudaGetLastError(), "policy")) return MR_ERR_CUDA;
  // the other fields of an FP32 grid adapt in FP32 unless asked otherwise
  const bool f32 = g->desc.precision == MR_F32, o32 = f32 && !bnd && !(flags & MR_ADAPT_OTHERS_FP64);
  if (changed == 0) {
    // Alg. SM3 step 1 ghost-fills every field in every iteration; with no
    // leaf changing, what remains of it for the other fields is the
    // substitution next to coarser leaves, which overwrites their values
    for (int fid = 0; fid < g->desc.nfields; ++fid) {
      if (fid == crit) continue;
      e = bnd ? launch_ghost(g, field_ptr(g, fid), field_ptr(g, fid), G, true, &Pv, &Gi)
              : launch_substitute(g, field_ptr(g, fid), nullptr, false, o32);
      if (e) return e;
    }
    return MR_OK;
  }
  if (nn > g->desc.capacity) {
    set_error("adaptation exceeds the leaf capacity");
    return MR_ERR_NOMEM;
  }
  const int nx = g->cur ^ 1;
  MR_LAUNCH(g, MRK_EMIT, k_emit<<<nblk, tb, 0, st>>>(n, g->M, g->status, g->scan, g->lev[g->cur],
                                                     g->anc[g->cur], g->refined, g->lev[nx], g->anc[nx],
                                                     g->keys[nx], g->refined2, g->newsrc));
  // owner map of the new tree
  Tree tn = next_view(g, nn);
  {
    const int saved_cur = g->cur, saved_n = g->nleaf;
    g->cur = nx, g->nleaf = nn;
    e = build_map(g);
    g->cur = saved_cur, g->nleaf = saved_n;
    if (e) return e;
  }
  int *nmask = g->cmask + g->desc.capacity;  // second half of the mask buffer
  int *hasD = g->hasD;
  // leaves whose ghosts the other fields need (statuses are final; maxdet and
  // scan are free from here on)
  int *nb1 = reinterpret_cast<int *>(g->maxdet), *need2 = nb1 + g->desc.capacity, *need = g->scan;
  MR_LAUNCH(g, MRK_MISC, k_need1<<<nblk, tb, 0, st>>>(t, g->status, nb1));
  MR_LAUNCH(g, MRK_MISC, k_need2<<<nblk, tb, 0, st>>>(t, g->status, nb1, need));
  MR_LAUNCH(g, MRK_MISC, k_need3<<<nblk, tb, 0, st>>>(t, need, need2));
  MR_LAUNCH(g, MRK_UPDATE, k_newmask<<<(nn + tb - 1) / tb, tb, 0, st>>>(tn, g->newsrc, nmask));
  // 6-9: every field: ghosts (criterion field first: P is current), interpolate, update.
  // Alg. SM3 step 1 ghost-fills every field, so the substitution next to
  // coarser leaves overwrites every field; the padded blocks themselves are
  // read only by the interpolation and update of the leaves in need2.  The
  // other fields therefore take (A) the adaptation-shell fill of the need2
  // leaves, without writing substituted values back, and (B) the
  // substitution-only pass of every leaf next to a coarser leaf (its padded
  // blocks in the side buffer, free here), which writes them back; both read
  // the field as it was, like one full ghost fill.  In FP32 (o32) both run
  // with FP32 padded blocks, and so do the interpolation and update.
  for (int pass = 0; pass < g->desc.nfields; ++pass) {
    const int fid = pass == 0 ? crit : (pass <= crit ? pass - 1 : pass);
    if (pass > 0 && o32) {
      e = launch_ghost_adapt32(g, (const float *)field_ptr(g, fid), G, need2, &Pv, &Gi);
      if (!e) e = launch_substitute(g, field_ptr(g, fid), nullptr, true, true);
      if (!e) e = interp_dispatch<float, float>(g, t, tn, (const float *)Pv, Gi, fid, nmask, hasD);
      if (e) return e;
      continue;
    }
    if (pass > 0 && bnd) {
      e = launch_ghost(g, field_ptr(g, fid), field_ptr(g, fid), G, true, &Pv, &Gi);
      if (e) return e;
      P = (const double *)Pv;
    } else if (pass > 0) {
      e = launch_ghost(g, field_ptr(g, fid), nullptr, G, true, &Pv, &Gi, nullptr, need2);
      if (!e) e = launch_substitute(g, field_ptr(g, fid), nullptr, true);
      if (e) return e;
      P = (const double *)Pv;
    }
    e = f32 ? interp_dispatch<float, double>(g, t, tn, P, Gi, fid, nmask, hasD)
            : interp_dispatch<double, double>(g, t, tn, P, Gi, fid, nmask, hasD);
    if (e) return e;
  }
  // swap to the new tree and pool
  g->cur = nx;
  g->map = g->maps[nx];
  g->pool_cur ^= 1;
  g->nleaf = nn;
  g->tree_version++;
  int *tmp = g->refined;
  g->refined = g->refined2;
  g->refined2 = tmp;
  *nch = changed;
  return check_cuda(cudaGetLastError(), "adapt") ? MR_ERR_CUDA : MR_OK;
}

}  // namespace mr
