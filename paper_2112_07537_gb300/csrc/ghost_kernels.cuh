// ghost_kernels.cuh -- the ghost-reconstruction kernels and their launch
// logic, templated on the field type TI and the padded-block type TP.  The
// instantiations of ghost_impl live in one small translation unit per
// (field type, block type, interpolation order) -- ghost_i_*.cu -- so that
// they compile in parallel; ghost.cu holds the dispatch and the untemplated
// launchers.
#pragma once
// Ghost-point reconstruction on the device (Alg. SM1 / SM2).
//
// Two kernels, one CTA per leaf:
//   prep:  padded block = interior + same-level copies + zero-detail
//          refinement of the coarse-level values where a coarser leaf owns
//          the point + the coincident value where a finer leaf owns it; then
//          the degree-ordered substitution of the band next to coarser
//          leaves (Sec. 2.2.4, eqs 2.27-2.29) on the padded block; then the
//          tensor H^a coarsening of the block at every ghost point of a
//          coarser neighbour that it owns, pushed to a side buffer (Part 2);
//   merge: side buffer -> padded block; substituted interior -> field.
// The wavelet sums are fused multiply-adds evaluated separably where that
// saves work (refinement per coarse region box, substitution per band box,
// Part-2 coarsening), so they agree with a plain nested-loop evaluation to
// rounding, not bit for bit; each is deterministic (one writer per value, a
// fixed order of terms).
#include <algorithm>
#include <cstdio>

#include "wavelet_runs.cuh"

namespace mr {

template <typename T>
__device__ __forceinline__ T ld(const T *p) { return __ldg(p); }

// Value stored by leaf o (level Lo >= L or a coarse grid point) at level-L
// point g; flags a balance error through *err when g is not on o's grid.
template <typename TI>
__device__ __forceinline__ TI leaf_value(const Tree &t, const TI *phi, int o, int L, int gx,
                                         int gy, int gz, int *err) {
  const int Lo = __ldg(t.lev + o);
  const int lx = local_index(t, o, Lo, L, gx, 0);
  const int ly = local_index(t, o, Lo, L, gy, 1);
  const int lz = local_index(t, o, Lo, L, gz, 2);
  const int nb = t.nb;
  if (lx < 0 || ly < 0 || lz < 0 || lx >= nb || ly >= nb || lz >= nb) {
    atomicOr(err, 1);
    return TI(0);
  }
  return ld(phi + (size_t)o * nb * nb * nb + lx + nb * (ly + nb * lz));
}

// ---------------------------------------------------------------------------
// Physical boundaries (Sec. 2.4).  Along a bounded axis, points beyond the
// domain take the polynomial of degree < N through grid values next to the
// boundary (or zeros); along several bounded axes the one-axis polynomials
// multiply.  The regions of a block's neighbourhood beyond the domain count as
// the block's own (level L, its own slot) in the region tables of the kernels
// below: they are filled with in-range values first, and bc_box then
// overwrites every point beyond the domain -- in the coarse tile before
// refinement (Alg. SM1), in the block before substitution and coarsening
// (Alg. SM2), and once more when every ghost is known.
// ---------------------------------------------------------------------------

// Nodes and weights of the boundary polynomial for the point r relative to the
// boundary (lower: r < 0, domain points 0, 1, ...; upper: r >= 0, domain points
// -1, -2, ...): value = sum_j w[j] f(node[j]).  Returns the node count, 0 for
// plain zeros.  Zero value: 0 at position 0 and the N-1 nearest points off it.
template <int N>
__device__ int bc_weights(int bc, int r, bool lower, int *node, double *w) {
  if (bc == MR_BC_ZERO) return 0;
  const int first = bc == MR_BC_DIRICHLET0 ? 1 : 0, m = N - first;
  double xs[N];
  for (int i = 0; i < N; ++i) xs[i] = lower ? (double)i : bc == MR_BC_DIRICHLET0 ? (double)-i : (double)(-1 - i);
  for (int j = 0; j < m; ++j) {
    const int jj = j + first;
    double wj = 1.0;
    for (int k = 0; k < N; ++k)
      if (k != jj) wj *= ((double)r - xs[k]) / (xs[jj] - xs[k]);
    w[j] = wj;
    node[j] = (int)xs[jj];
  }
  return m;
}

// first index inside the domain and one past the last along axis d, local to a
// block whose first point is a at level L (no limit along a periodic axis)
__device__ __forceinline__ int bc_first(const Tree &t, int a, int d) { return (t.bnd >> d) & 1 ? -a : -(1 << 28); }
__device__ __forceinline__ int bc_end(const Tree &t, int L, int a, int d) {
  return (t.bnd >> d) & 1 ? npts(t, L, d) - a : 1 << 28;
}
// the cube [lo, hi)^3 around that block reaches beyond the domain
__device__ __forceinline__ bool bc_touches(const Tree &t, int L, int ax, int ay, int az, int lo, int hi) {
  return lo < bc_first(t, ax, 0) || hi > bc_end(t, L, ax, 0) || lo < bc_first(t, ay, 1) || hi > bc_end(t, L, ay, 1) ||
         lo < bc_first(t, az, 2) || hi > bc_end(t, L, az, 2);
}

// Every point of the box [lo, lo + n) beyond the domain, axis by axis: A[x +
// s1 y + s2 z], indices local to the block whose first level-L point is (ax,
// ay, az).  The whole CTA takes part; the nodes lie inside the box.  Out of
// line: only blocks at a boundary call it.
template <int N, typename TP>
__device__ __noinline__ void bc_box(const Tree &t, int L, int ax, int ay, int az, TP *A, int s1, int s2, int lx, int ly,
                                    int lz, int ex, int ey, int ez) {
  __shared__ double wt[MR_MAX_SHELL + 4][N];
  __shared__ int nd[N], nn;
  const int st[3] = {1, s1, s2}, lo[3] = {lx, ly, lz}, hi[3] = {lx + ex, ly + ey, lz + ez}, a[3] = {ax, ay, az};
  const int bc = t.bc;
  for (int d = 0; d < 3; ++d)
    for (int side = 0; side < 2; ++side) {
      const int org = side ? bc_end(t, L, a[d], d) : bc_first(t, a[d], d);
      const int l0 = side ? max(org, lo[d]) : lo[d], l1 = side ? hi[d] : min(org, hi[d]), n = l1 - l0;
      if (n <= 0) continue;
      __syncthreads();  // the values this side reads; the tables of the last one
      if ((int)threadIdx.x < n) {
        double w[N];
        int node[N];
        const int c = bc_weights<N>(bc, l0 + (int)threadIdx.x - org, !side, node, w);
        for (int j = 0; j < c; ++j) wt[threadIdx.x][j] = w[j];
        if (threadIdx.x == 0) {
          nn = c;
          for (int j = 0; j < c; ++j) nd[j] = node[j] + org;
        }
      }
      __syncthreads();
      const int e1 = d == 0 ? 1 : 0, e2 = d == 2 ? 1 : 2, n1 = hi[e1] - lo[e1], n2 = hi[e2] - lo[e2];
      const DivM dn = divm(n), d1 = divm(n1);
      for (int p = threadIdx.x; p < n * n1 * n2; p += blockDim.x) {
        const int r = divq(p, dn), l = p - r * n, q2 = divq(r, d1), q1 = r - q2 * n1;
        TP *c = A + st[e1] * (lo[e1] + q1) + st[e2] * (lo[e2] + q2);
        TP v = TP(0);
        for (int j = 0; j < nn; ++j) v += TP(wt[l][j]) * c[st[d] * nd[j]];
        c[st[d] * (l0 + l)] = v;
      }
    }
  __syncthreads();
}

// Coarse value of Alg. SM1 at level-Lq point q next to leaf hb: the stored
// value inside the domain, the tensor of the boundary polynomials beyond it.
// One point at a time, for coarse tiles that do not fit in shared memory.
template <typename TI, typename TP, int N>
__device__ __noinline__ TP coarse_bc(const Tree &t, int Lq, int qx, int qy, int qz, const TI *phi, int hb, int *err) {
  const int q[3] = {qx, qy, qz};
  int m[3], idx[3][N];
  double w[3][N];
  for (int d = 0; d < 3; ++d) {
    m[d] = 1, idx[d][0] = q[d], w[d][0] = 1.0;
    if (!beyond(t, Lq, q[d], d)) continue;
    const int org = q[d] < 0 ? 0 : npts(t, Lq, d);
    m[d] = bc_weights<N>(t.bc, q[d] - org, q[d] < 0, idx[d], w[d]);
    for (int j = 0; j < m[d]; ++j) idx[d][j] += org;
  }
  TP s = TP(0);
  for (int c = 0; c < m[2]; ++c)
    for (int b = 0; b < m[1]; ++b)
      for (int a = 0; a < m[0]; ++a) {
        const int o = owner(t, Lq, idx[0][a], idx[1][b], idx[2][c], hb);
        if (__ldg(t.lev + o) < Lq) {
          atomicOr(err, 2);
          return TP(0);
        }
        s += TP(w[0][a] * w[1][b] * w[2][c]) *
             Cvt<TP>::f(leaf_value(t, phi, o, Lq, idx[0][a], idx[1][b], idx[2][c], err));
      }
  return s;
}

// Zero-detail refinement at level-L point g from the level-(L-1) values
// (J^s on even, K^s on odd coordinates; taps landing on details skipped).
template <typename TI, typename TP, int N, int NT>
__device__ TP refine_point(const Tree &t, const TI *phi, int L, int gx, int gy, int gz, int *err, int hb) {
  return refine_dispatch<N, NT, TP>(gx & 1, gy & 1, gz & 1, [&](int ox, int oy, int oz) -> TP {
    const int qx = floordiv2(gx + ox), qy = floordiv2(gy + oy), qz = floordiv2(gz + oz);
    if (t.bnd) return coarse_bc<TI, TP, N>(t, L - 1, qx, qy, qz, phi, hb, err);
    const int o = owner(t, L - 1, qx, qy, qz, hb);
    if (__ldg(t.lev + o) < L - 1) {
      atomicOr(err, 2);
      return TP(0);
    }
    return Cvt<TP>::f(leaf_value(t, phi, o, L - 1, qx, qy, qz, err));
  });
}

// ---------------------------------------------------------------------------
// The padded block of a leaf: the gather, and next to coarser leaves the
// zero-detail refinement of their regions (Part 1), the substitution of the band
// next to them, and Part 2 pushed to the coarser neighbours.  A block is read
// and written by its own CTA only, so the copy-bound gather of some leaves
// overlaps the latency-bound phases of others.
//
// Coarser neighbours by parent: a leaf's coarser neighbours touch its parent
// from outside, so they lie in the (up to) seven directions e = 1..7 of the
// parent's outward sides (bit d of e: across axis d, on the side of the
// leaf's own half), and the neighbour in direction e owns one box of the
// padded block: the shell along the axes of e, the block and its inward ghosts
// along the others.  Refinement boxes, band boxes and push boxes are therefore
// intervals per axis, cut into disjoint boxes by at most one clip each.
//
// Every phase is a flat list of items over all boxes (or as many as the
// shared-memory sums allow), so the CTA meets a handful of barriers per leaf
// instead of one per box and pass, and the index tables of a phase are built
// by one thread each and read by all.  What bounds the kernel is issued
// instructions (index arithmetic, 42 % issue) and the latency of its ~20 dependent
// phases at 32 warps per SM.  3 424 leaves of 24^3 with 6.2, FP32: 1 028 us for a
// gather and a pre-pass of boxes in turn, 433 us with flat phases in two kernels,
// 376 us so, of which region tables 23, gather 98, refinement 76, substitution 130,
// push 48.
// ---------------------------------------------------------------------------
struct PrepTab {
  int rslot[27], rlev[27], ranc[27][3], rsub[27][8];
  // level-(L-1) values of a region held by one leaf: index rbase + rmul *
  // (q0 + nb q1 + nb^2 q2) of the block-local coarse point q (rmul 0: finer)
  long long rbase[27];
  int rmul[27];
  int cmask, ce;  // coarser directions (bit region), coarser neighbours (bit e)
  int s[3], odd[3];  // outward side per axis (+-1), anchor parity
  int miss;          // bounded grids: prep_fetch met a point that no leaf holds
};

// up to 7 disjoint boxes over [0, n) per axis, the layers (dlo on the - side,
// dhi on the + side) next to the coarser neighbours ce
struct Boxes {
  int n, lo[7][3], hi[7][3];
  int flat[7];  // axes along which the neighbour does not lie across a side (bit per axis)
};
// (by one warp, a lane per direction; faces first, then edges, then the corner)
__device__ __forceinline__ void outward_boxes(Boxes &B, int ce, const int *s, int n, int dlo, int dhi) {
  const int q = threadIdx.x & 31;
  auto dir = [](int rank) { return (0x7653421 >> (4 * rank)) & 7; };
  const int e = q < 7 ? dir(q) : 0;
  bool keep = (ce >> e) & 1;  // not inside the box of a coarser neighbour across fewer axes
  for (int f = 1; f < 7; ++f) keep = keep && !(((ce >> f) & 1) && f != e && (f & e) == f);
  const unsigned kept = __ballot_sync(0xffffffffu, keep);
  int lo[3], hi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const bool on = (e >> d) & 1;
    lo[d] = on && s[d] > 0 ? n - dhi : 0, hi[d] = on && s[d] < 0 ? dlo : n;
    // an earlier box (across the axes of f) covers this one along every axis
    // but the one of f that e does not have
    for (int r = 0; r < 6; ++r)
      if (r < q && ((kept >> r) & 1) && (((dir(r) & ~e) >> d) & 1)) {
        if (s[d] > 0) hi[d] = min(hi[d], n - dhi);
        else lo[d] = max(lo[d], dlo);
      }
  }
  keep = keep && lo[0] < hi[0] && lo[1] < hi[1] && lo[2] < hi[2];
  const unsigned have = __ballot_sync(0xffffffffu, keep);
  if (keep) {
    const int at = __popc(have & ((1u << q) - 1u));
    for (int d = 0; d < 3; ++d) B.lo[at][d] = lo[d], B.hi[at][d] = hi[d];
    B.flat[at] = 7 & ~e;
  }
  if (q == 0) B.n = __popc(have);
}

// level-Lq value (Lq = L or L - 1) at block-local point (i, j, k) through the
// region tables, or through the owner map beyond the neighbouring regions; NaN where
// no leaf holds the point (BND: and T.miss set)
template <bool BND, typename TI>
__device__ __noinline__ TI prep_fetch(const Tree &t, PrepTab &T, const TI *phi, int b, int L, int Lq, int i, int j,
                                      int k, int *err) {
  const int nb = t.nb, hb = nb / 2, sc = Lq == L ? 1 : 2;
  const size_t nb3 = (size_t)nb * nb * nb;
  const int f[3] = {i * sc, j * sc, k * sc};
  bool in = true;
  int r = 0, rl[3], h = 0;
  for (int d = 2; d >= 0; --d) {
    in &= f[d] >= -nb && f[d] < 2 * nb;
    const int c = f[d] < 0 ? 0 : f[d] >= nb ? 2 : 1;
    r = 3 * r + c, rl[d] = f[d] - (c - 1) * nb;
    h |= (rl[d] >= hb) << d;
  }
  if (in) {
    if (T.rlev[r] == L) return ld(phi + T.rslot[r] * nb3 + rl[0] + nb * (rl[1] + nb * rl[2]));
    if (T.rlev[r] == L + 1 && T.rsub[r][h] >= 0)
      return ld(phi + T.rsub[r][h] * nb3 + (2 * rl[0] - (h & 1) * nb) +
                nb * ((2 * rl[1] - ((h >> 1) & 1) * nb) + nb * (2 * rl[2] - (h >> 2) * nb)));
  }
  int g[3];
  for (int d = 0; d < 3; ++d) g[d] = (Lq == L ? T.ranc[13][d] * nb : T.ranc[13][d] * nb / 2) + (d == 0 ? i : d == 1 ? j : k);
  const int o = owner(t, Lq, g[0], g[1], g[2], b);
  if (__ldg(t.lev + o) < Lq) {
    if (BND) T.miss = 1;
    return TI(__int_as_float(0x7fc00000));
  }
  return leaf_value(t, phi, o, Lq, g[0], g[1], g[2], err);
}

// ---------------------------------------------------------------------------
// The gather part of a leaf's padded block Pb (Alg. SM1): interior, the values
// of same-level neighbours (copy) and the coincident values of finer neighbours
// (their fine-to-coarse values are merged afterwards) -- everything but the
// regions of coarser leaves.
// One thread per (x, y) column of the padded block: along z the column crosses
// at most three regions (a finer one in two halves), each of which is a run
// of values a fixed stride apart in one leaf, so a point costs a load, a
// store and two additions (a source index per point cost 113 instructions: 327
// against 133 us for the 1 696 leaves next to coarser ones of a 3 424-leaf grid
// of 24^3 blocks, shell 6).
// LEAN (passes whose blocks are read in their interior and next to coarser
// leaves alone): beside the interior only the points within reach of a coarser
// neighbour, the layers that the substitution and the push read -- a third of the
// ghosts is left out where one face borders on a coarser leaf (the pre-pass of
// the grid above 390 -> 376 us, of 42 400 leaves of 24^3 2.56 -> 2.42 ms).
// ---------------------------------------------------------------------------
template <bool LEAN, typename TI, typename TP>
__device__ __forceinline__ void gather_block(const Tree &t, const PrepTab &T, const TI *__restrict__ phi, TP *Pb, int b,
                                             int L, int Gi, int reach, int *err) {
  const int nb = t.nb, Wd = nb + 2 * Gi, hb = nb / 2, W2 = Wd * Wd, nb2 = nb * nb;
  const size_t nb3 = (size_t)nb * nb2;
  const DivM dW = divm(Wd);
  // n values st apart from src to padded planes from d on, four in flight
  auto run = [&](TP *d, const TI *src, int st, int n) {
    for (; n >= 4; n -= 4, d += 4 * W2, src += 4 * st) {
      const TI v0 = ld(src), v1 = ld(src + st), v2 = ld(src + 2 * st), v3 = ld(src + 3 * st);
      d[0] = Cvt<TP>::f(v0), d[W2] = Cvt<TP>::f(v1), d[2 * W2] = Cvt<TP>::f(v2), d[3 * W2] = Cvt<TP>::f(v3);
    }
    for (; n > 0; --n, d += W2, src += st) *d = Cvt<TP>::f(ld(src));
  };
  // bit m of all / some: a column near the outward sides m (bit 0: x, 1: y) lies
  // within reach of a coarser neighbour everywhere / near the outward side of z
  unsigned all = 0, some = 0;
  for (int m = 0; m < 4 && LEAN; ++m)
    for (int e = 1; e < 8; ++e)
      if (((T.ce >> e) & 1) && !(e & 3 & ~m)) (e & 4 ? some : all) |= 1u << m;
  auto near = [&](int x, int d) { return T.s[d] > 0 ? x >= nb - reach : x < reach; };
  for (int c = threadIdx.x; c < W2; c += blockDim.x) {
    const int row = divq(c, dW), i = c - row * Wd - Gi, j = row - Gi;
    int za = -Gi, zb = nb + Gi;  // planes wanted of this column
    if (LEAN) {
      const int m = (near(i, 0) ? 1 : 0) | (near(j, 1) ? 2 : 0);
      const bool in = i >= 0 && i < nb && j >= 0 && j < nb;
      if (!((all >> m) & 1)) {
        const bool zn = (some >> m) & 1;
        if (!zn && !in) continue;
        za = !zn ? 0 : T.s[2] < 0 ? -Gi : in ? min(0, nb - reach) : nb - reach;
        zb = !zn ? nb : T.s[2] > 0 ? nb + Gi : in ? max(nb, reach) : reach;
      }
    }
    const int rx = i < 0 ? 0 : i >= nb ? 2 : 1, ry = j < 0 ? 0 : j >= nb ? 2 : 1;
    const int ri = i - (rx - 1) * nb, rj = j - (ry - 1) * nb;  // region-local
    TP *col = Pb + c + (size_t)W2 * Gi;                        // (i, j, 0)
    for (int rz = 0; rz < 3; ++rz) {
      const int r = rx + 3 * ry + 9 * rz, Lo = T.rlev[r];
      if (Lo < L) continue;  // a coarser leaf's region: refined below
      const int z0 = (rz - 1) * nb;  // region-local planes
      int k0 = rz == 0 ? nb - Gi : 0, k1 = rz == 2 ? Gi : nb;
      if (LEAN) {
        k0 = max(k0, za - z0), k1 = min(k1, zb - z0);
        if (k0 >= k1) continue;
      }
      if (Lo == L) {
        run(col + (ptrdiff_t)W2 * (z0 + k0), phi + (size_t)T.rslot[r] * nb3 + ri + nb * rj + nb2 * k0, nb2, k1 - k0);
        continue;
      }
      const int hx = ri >= hb, hy = rj >= hb;
      for (int hz = 0; hz < 2; ++hz) {
        const int ka = hz ? max(k0, hb) : k0, kb = hz ? k1 : min(k1, hb);
        if (ka >= kb) continue;
        const int o2 = T.rsub[r][hx + 2 * hy + 4 * hz];
        if (o2 >= 0) {
          run(col + (ptrdiff_t)W2 * (z0 + ka),
              phi + (size_t)o2 * nb3 + (2 * ri - hx * nb) + nb * (2 * rj - hy * nb) + nb2 * (2 * ka - hz * nb),
              2 * nb2, kb - ka);
        } else {  // two levels down (shells wider than half a block)
          for (int k = ka; k < kb; ++k) {
            const int gx = T.ranc[13][0] * nb + i, gy = T.ranc[13][1] * nb + j, gz = T.ranc[13][2] * nb + z0 + k;
            const int ow = owner(t, L, gx, gy, gz, b);
            col[(ptrdiff_t)W2 * (z0 + k)] = Cvt<TP>::f(leaf_value(t, phi, ow, L, gx, gy, gz, err));
          }
        }
      }
    }
  }
}

// One box of a coarser leaf's region: expanded along the thin axis a, then b,
// then c (b = x where it can, so that neighbouring threads are neighbours in
// memory; the box is cut along c so that its sums fit in shared memory).
struct RefBox {
  int a, b, c;                 // axes
  int la, lb, lc, na, nb, nc;  // fine range per axis of the walk: [l, l + n)
  int cb, cc, mb, mc;          // coarse range of the sums along b, c
  int mbp, nbp, S;             // pitches (odd: no bank conflicts)
  int off;                     // U1 at off, U2 at off + na * mbp * mc
  unsigned dmb, dna, dnb;      // reciprocals of mb, na, nb
  unsigned dl2, dl3;           // and of the lines of pass 2 (na mc) and pass 3 (na nb)
};

// next start of the thread rotation after n items
__device__ __forceinline__ int turn(int rot, int n, int bd) {
  rot += n;
  while (rot >= bd) rot -= bd;
  return rot;
}

constexpr int SUB_RUN = 4;  // points of one item of the substitution

// Flat axes are used where arithmetic counts: FP64 blocks (ghost fills of 1 408
// leaves of 24^3 with 6.2, shell 6: 637 -> 563 us, of 2 080 with shell 11 1 770 ->
// 1 672 us); with FP32 blocks the listed coordinates cost more than the sums they
// save (42 400 leaves 2.42 -> 2.56 ms).
template <typename TP>
constexpr bool sub_flat = sizeof(TP) == 8;

// Points of a band box along a flat axis (sub_coord): even ones below lo from e0
// on, odd ones of [lo, hi) from o0 on, even ones above from e1 on
struct SubAxes {
  short lo[3], hi[3], e0[3], o0[3], e1[3], nlo[3], nod[3];
};

// One parity class (odd dimensions om) of degree deg over one band box: summed
// one odd dimension at a time (o[0] first), as walked by subst_sep.
struct SubJob {
  int om, deg, o[3];
  short st[3][3], cn[3][3];  // per pass: first point, count per axis
  int sp1[3];              // per pass: axes walked with step 1 (others 2)
  short fl[3], flat, box;  // per pass: axes walked by sub_coord; flat axes of the box; the box
  unsigned d0[3], d1[3];   // reciprocals of the item counts along axes 0, 1
  int n[3], it[3];         // points per pass; items (runs of SUB_RUN points along o[pass])
  int off, next;           // sums in shared memory; end of the batch this job opens
};

// ---------------------------------------------------------------------------
// Separable substitution.  A band point p of a class with odd dimensions o_1..
// o_deg becomes -S(p), S(p) = sum over t != 0 (t along the odd dimensions) of
// prod_d G^a(t_d) P(p + t).  S is summed one odd dimension at a time, thinnest
// box side first, with the partial sums of each (box, class) job in shared
// memory: pass 1 reads the padded block at every point the later passes need, the
// last pass writes -S into the block.  Odd dimensions not yet summed span the box
// plus the G^a half-width; along a flat axis (the band goes on to both ends of the
// box) only the box's odd points and the even ones beyond it: a band point has no
// detail along the odd dimensions it shares with the class, so the terms at even
// points inside add up to zero over the other dimensions and are left out, and
// away from the ends S is the sum of the pass before (half the points of a face
// box).  (A NaN or infinity at such a point therefore reaches the degree-1 points
// around it, but not every point of higher degree that has it among its taps.)
// Pass 1 drops its t = 0 term where every
// other odd coordinate is odd -- exactly at the class points, which no other
// term of any pass reads -- so the product over all t leaves out t = 0.
// Points of one degree read lower degrees only, so all jobs of a degree run
// together, batched so that their sums fit; a job that does not fit alone
// runs point by point.  An item is a run of SUB_RUN points along the summed
// dimension: their taps share a window of even points, loaded together (13
// loads in flight for four points instead of 28 in four dependent rounds).
// ---------------------------------------------------------------------------
// coordinate of index q along flat axis d
__device__ __forceinline__ int sub_coord(const SubAxes &J, int d, int q) {
  const int a = J.nlo[d], b = a + J.nod[d];
  return 2 * q + (q < a ? J.e0[d] : q < b ? J.o0[d] - 2 * a : J.e1[d] - 2 * b);
}

__device__ __forceinline__ void sub_job_build(SubJob &J, SubAxes *ax, int box, const int *lo, const int *hi, int om,
                                              int hG, int flat) {
  J.om = om, J.deg = __popc(om), J.flat = (short)flat, J.box = (short)box;
  int nall[3];
  for (int d = 0; d < 3; ++d) {
    const int nlo = par_count(lo[d] - hG, lo[d], 0), nod = par_count(lo[d], hi[d], 1);
    nall[d] = nlo + nod + par_count(hi[d], hi[d] + hG, 0);
    if (flat && om == 7) {  // (one job per box)
      SubAxes &A = ax[box];
      A.lo[d] = (short)lo[d], A.hi[d] = (short)hi[d], A.nlo[d] = (short)nlo, A.nod[d] = (short)nod;
      A.e0[d] = (short)par_first(lo[d] - hG, 0), A.o0[d] = (short)par_first(lo[d], 1), A.e1[d] = (short)par_first(hi[d], 0);
    }
  }
  int o[3], n = 0;
  for (int d = 0; d < 3; ++d)
    if ((om >> d) & 1) o[n++] = d;
  for (int x = 1; x < n; ++x)
    for (int y = x; y > 0 && hi[o[y]] - lo[o[y]] < hi[o[y - 1]] - lo[o[y - 1]]; --y) {
      const int w = o[y];
      o[y] = o[y - 1], o[y - 1] = w;
    }
  int summed = 0;
  for (int s = 0; s < 3; ++s) {
    J.o[s] = s < n ? o[s] : 0;
    J.n[s] = J.it[s] = 0;
    if (s >= n) continue;
    summed |= 1 << o[s];
    J.sp1[s] = om & ~summed & ~flat, J.fl[s] = (short)(om & ~summed & flat);
    for (int d = 0; d < 3; ++d) {
      const int odd = (om >> d) & 1;
      if ((J.fl[s] >> d) & 1) J.st[s][d] = 0, J.cn[s][d] = (short)nall[d];
      else if ((J.sp1[s] >> d) & 1) J.st[s][d] = (short)(lo[d] - hG), J.cn[s][d] = (short)(hi[d] - lo[d] + 2 * hG);
      else J.st[s][d] = (short)par_first(lo[d], odd), J.cn[s][d] = (short)par_count(lo[d], hi[d], odd);
    }
    J.n[s] = J.cn[s][0] * J.cn[s][1] * J.cn[s][2];
    int m[3];
    for (int d = 0; d < 3; ++d) m[d] = d == o[s] ? (J.cn[s][d] + SUB_RUN - 1) / SUB_RUN : J.cn[s][d];
    J.it[s] = m[0] * m[1] * m[2];
    J.d0[s] = divm(max(m[0], 1)).m, J.d1[s] = divm(max(m[1], 1)).m;
  }
}

// sums of the run: sum_t G^a(t) src[(2 m + t) st] for m = 0 .. n - 1 (t = 0
// only with centre); put(m, sum)
template <int N, int NT, typename TP, typename F>
__device__ __forceinline__ void subst_run(const TP *src, int st, int n, bool centre, F put) {
  using W = Wav<N, NT>;
  constexpr int hG = W::hwG;
  TP e[N - 1 + SUB_RUN], c[SUB_RUN];
#pragma unroll
  for (int x = 0; x < N - 1 + SUB_RUN; ++x) e[x] = x < N - 1 + n ? src[(2 * x - hG) * st] : TP(0);
#pragma unroll
  for (int m = 0; m < SUB_RUN; ++m) c[m] = centre && m < n ? src[2 * m * st] : TP(0);
#pragma unroll
  for (int m = 0; m < SUB_RUN; ++m) {
    if (m >= n) break;
    // (the centre in its place among the taps: the partial sums stay small)
    TP acc = TP(0);
#pragma unroll
    for (int x = 0; x < N; ++x) {
      if (x == N / 2) acc = radd(acc, c[m]);
      acc = racc(acc, TP(W::G(2 * x - hG)), e[m + x]);
    }
    put(m, acc);
  }
}

// the same along flat axis d, for its odd points i .. i + n - 1: the line src holds
// the sums at the coordinates of sub_coord, the even points inside count as 0
template <int N, int NT, typename TP, typename F>
__device__ __forceinline__ void subst_ends(const TP *src, int st, const SubAxes &J, int d, int i, int n, F put) {
  using W = Wav<N, NT>;
  constexpr int hG = W::hwG;
  const int lo = J.lo[d], hi = J.hi[d], y = J.o0[d] + 2 * i, a = J.nlo[d], b = a + J.nod[d], e0 = J.e0[d],
            e1 = J.e1[d] - 2 * b;
  const TP *c = src + (a + i) * st;
  if (y - hG >= lo && y + 2 * (n - 1) + hG < hi) {
#pragma unroll
    for (int m = 0; m < SUB_RUN; ++m)
      if (m < n) put(m, c[m * st]);
    return;
  }
  TP e[N - 1 + SUB_RUN];
#pragma unroll
  for (int x = 0; x < N - 1 + SUB_RUN; ++x) {
    const int v = y + 2 * x - hG;
    e[x] = x < N - 1 + n && (v < lo || v >= hi) ? src[((v - (v < lo ? e0 : e1)) >> 1) * st] : TP(0);
  }
#pragma unroll
  for (int m = 0; m < SUB_RUN; ++m) {
    if (m >= n) break;
    TP acc = TP(0);
#pragma unroll
    for (int x = 0; x < N; ++x) {
      if (x == N / 2) acc = radd(acc, c[m * st]);
      acc = racc(acc, TP(W::G(2 * x - hG)), e[m + x]);
    }
    put(m, acc);
  }
}

template <int N, int NT, typename TP>
__device__ __forceinline__ void subst_jobs(TP *Pb, int Wd, int Gi, const SubJob *jobs, const SubAxes *axes, int j0,
                                           int jend, TP *buf, int cap) {
  constexpr bool FLAT = sub_flat<TP>;
  const int W2 = Wd * Wd, bd = blockDim.x;
  while (j0 < jend) {
    const int j1 = jobs[j0].next, deg = jobs[j0].deg;
    const bool pointwise = jobs[j0].n[0] * (deg > 1) + jobs[j0].n[1] * (deg > 2) > cap;
    for (int s = pointwise ? deg - 1 : 0; s < deg; ++s) {
      int rot = 0;  // the items of a job continue the thread rotation of the previous one
      for (int j = j0; j < j1; ++j) {
        const SubJob &J = jobs[j];
        const SubAxes &A = axes[J.box];
        const int n = J.it[s];
        int idx = (int)threadIdx.x - rot;
        if (idx < 0) idx += bd;
        rot = turn(rot, n, bd);
        if (idx >= n) continue;
        const int st0 = J.st[s][0], st1 = J.st[s][1], st2 = J.st[s][2], sp1 = J.sp1[s], fl = J.fl[s];
        const int h0 = !(sp1 & 1), h1 = !(sp1 & 2), h2 = !(sp1 & 4);  // log2 of the steps
        const int d = J.o[s], cd = J.cn[s][d];
        const int c0 = J.cn[s][0], c1 = J.cn[s][1];
        const int m0 = d == 0 ? (c0 + SUB_RUN - 1) / SUB_RUN : c0, m1 = d == 1 ? (c1 + SUB_RUN - 1) / SUB_RUN : c1;
        const DivM dc0{J.d0[s], m0}, dc1{J.d1[s], m1};
        const int str = d == 0 ? 1 : d == 1 ? Wd : W2, ds = d == 0 ? 1 : d == 1 ? c0 : c0 * c1;
        TP *dst = buf + J.off + (s == 1 ? J.n[0] : 0);
        const bool last = s == deg - 1;
        for (; idx < n; idx += bd) {
          const int r = divq(idx, dc0), q2 = divq(r, dc1), q0 = idx - r * m0, q1 = r - q2 * m1;
          const int i0 = d == 0 ? q0 * SUB_RUN : q0, i1 = d == 1 ? q1 * SUB_RUN : q1, i2 = d == 2 ? q2 * SUB_RUN : q2;
          const int nr = min(SUB_RUN, cd - (d == 0 ? i0 : d == 1 ? i1 : i2));  // points of this run
          const int p0 = FLAT && fl & 1 ? sub_coord(A, 0, i0) : st0 + (i0 << h0),
                    p1 = FLAT && fl & 2 ? sub_coord(A, 1, i1) : st1 + (i1 << h1),
                    p2 = FLAT && fl & 4 ? sub_coord(A, 2, i2) : st2 + (i2 << h2);
          TP *pt = Pb + (p0 + Gi) + Wd * (p1 + Gi) + W2 * (p2 + Gi);
          TP *out = dst + i0 + c0 * (i1 + c1 * i2);
          auto put = [&](int m, TP acc) {
            if (last) pt[2 * m * str] = -acc;
            else out[m * ds] = acc;
          };
          if (pointwise) {
            for (int m = 0; m < nr; ++m) {
              TP *c = pt + 2 * m * str;
              *c = subst_dispatch<N, NT, TP>(J.om & 1, J.om & 2, J.om & 4,
                                             [&](int tx, int ty, int tz) -> TP { return c[tx + Wd * ty + W2 * tz]; });
            }
          } else {
            // pass 1 reads the block; a later one the previous pass's sums, which
            // run with step 1 from st[s-1] along this dimension and hold this
            // pass's points along the others
            const int oth = J.om & ~(1 << d);
            const bool centre = s > 0 || (oth & ~((p0 & 1) | ((p1 & 1) << 1) | ((p2 & 1) << 2))) != 0;
            const TP *src = pt;
            int ss = str;
            if (s > 0) {
              const int k0 = J.cn[s - 1][0], k1 = k0 * J.cn[s - 1][1];
              ss = d == 0 ? 1 : d == 1 ? k0 : k1;
              if (FLAT && ((J.flat >> d) & 1)) {
                subst_ends<N, NT>(buf + J.off + (s == 2 ? J.n[0] : 0) + (d == 0 ? 0 : i0) + k0 * (d == 1 ? 0 : i1) +
                                      k1 * (d == 2 ? 0 : i2),
                                  ss, A, d, d == 0 ? i0 : d == 1 ? i1 : i2, nr, put);
                continue;
              }
              src = buf + J.off + (s == 2 ? J.n[0] : 0) + (J.st[s][d] - J.st[s - 1][d]) * ss +
                    (d == 0 ? 2 * i0 : i0) + k0 * (d == 1 ? 2 * i1 : i1) + k1 * (d == 2 ? 2 * i2 : i2);
            }
            subst_run<N, NT>(src, ss, nr, centre, put);
          }
        }
      }
      __syncthreads();
    }
    j0 = j1;
  }
}

constexpr int PUSH_LAYERS = 4;

// One box of coarse points to push: coarsened along the thinnest axis a, then b,
// then c, layers layers of a at a time.
struct PushBox {
  int a, b, c;                 // axes
  int na, nb, nc, fb, fc;      // coarse points per axis; fine extents along b, c
  int la, layers, base;        // first layer; fine block index of (la, lo_b - h, lo_c - h); linear index of lo
  int off, next;               // sums in shared memory; end of the batch this box opens
  unsigned dfb, dfc, drb, dnb, dnc;  // reciprocals of fb, fc, ceil(nb / 4), nb, nc
};

// boxes, jobs and tables of the three phases (one set per CTA)
struct PrepPlan {
  Boxes band, push;
  RefBox ref[28];
  int nref, refnext[28];  // refinement boxes; end of the batch a box opens
  SubJob job[49];
  SubAxes axes[7];
  int job0[4];            // first job of each degree (job0[3]: end)
  PushBox pbox[7];
  int npb;
  // coarser neighbours: direction, and the address in the side buffer of the
  // leaf's coarse point (0, 0, 0) (every coordinate shifts by a constant)
  int nq, qdir[7];
  long long qbase[7];
};

// The boundary polynomial on the sums U1 of one box (beyond the domain along b
// and c; the refinement along a acts on another index, so it may go first).
template <int N, typename TP>
__device__ __noinline__ void bc_sums(const Tree &t, int Lc, const RefBox &B, int ax, int ay, int az, TP *U1) {
  __shared__ double wt[MR_MAX_SHELL + 4][N];
  __shared__ int nd[N], nn;
  for (int w = 0; w < 4; ++w) {
    const int d = w < 2 ? B.b : B.c, side = w & 1, anc = d == 0 ? ax : d == 1 ? ay : az;
    const int lo = w < 2 ? B.cb : B.cc, hi = lo + (w < 2 ? B.mb : B.mc);
    const int org = side ? bc_end(t, Lc, anc, d) : bc_first(t, anc, d);
    const int l0 = side ? max(org, lo) : lo, l1 = side ? hi : min(org, hi), n = l1 - l0;
    if (n <= 0) continue;
    __syncthreads();
    if ((int)threadIdx.x < n) {
      double wv[N];
      int node[N];
      const int c = bc_weights<N>(t.bc, l0 + (int)threadIdx.x - org, !side, node, wv);
      for (int j = 0; j < c; ++j) wt[threadIdx.x][j] = wv[j];
      if (threadIdx.x == 0) {
        nn = c;
        for (int j = 0; j < c; ++j) nd[j] = node[j] + org - lo;
      }
    }
    __syncthreads();
    // strides: along the axis; the two others of the box
    const int pa = B.mbp, pc = B.mbp * B.na, str = w < 2 ? 1 : pc, so = w < 2 ? pc : 1, no = w < 2 ? B.mc : B.mb;
    for (int p = threadIdx.x; p < n * B.na * no; p += blockDim.x) {
      const int l = p % n, r = p / n;
      TP *c = U1 + pa * (r % B.na) + so * (r / B.na), v = TP(0);
      for (int j = 0; j < nn; ++j) v += TP(wt[l][j]) * c[str * nd[j]];
      c[str * (l0 + l - lo)] = v;
    }
  }
  __syncthreads();
}

// planes of the sums along c: a chunk of eight fine points (so that no leaf
// has more than 28 boxes), and on grids with physical boundaries the nodes of
// the polynomial
constexpr int prep_min_planes(int N, bool bounded) { return (N - 1) + 2 + 4 + (bounded ? N : 0); }

// Blocks so narrow that coarse columns of the refinement leave the neighbouring
// regions, where values are looked up through the owner map: 8^3 with 6.0, 8^3 and
// 10^3 with 6.2.  Their kernel (NARROW) looks every value of such a column up once
// (fills of 576 leaves of 8^3 with 6.2, shell 3: FP32 384 -> 206 us, FP64 426 -> 265;
// of 55 leaves, FP64: 212 -> 149).  In the other blocks only columns that meet a finer
// leaf are looked up; there the tap-by-tap form stays, since the window costs every
// column registers (fill and crop of 2 080 leaves of 24^3 with 6.2, FP32: 488 us so, 492
// with it).
__host__ __device__ constexpr bool prep_narrow(int N, int nb, int Gi) { return (Gi + N) / 2 * 2 > nb; }

// only_coarse: 0 every (needed) leaf, 1 the leaves next to coarser ones, 2 those
// without the push
template <typename TI, typename TP, int N, int NT, bool BND, bool NARROW>
__global__ void __launch_bounds__(sizeof(TP) == 4 ? 512 : 384, 2) k_prep(Tree t, const TI *__restrict__ phi,
                                                                     TP *__restrict__ P, TP *__restrict__ Q, int Gi,
                                                                     int Gpush, int only_coarse, int *cmask_out,
                                                                     int *err, const int *__restrict__ need,
                                                                     int *__restrict__ pneed, int sum_bytes) {
  using W = Wav<N, NT>;
  using RS = RefSum<TI, TP>;
  using U = typename RS::U;
  constexpr int ko = N - 1;  // widest odd K^s tap
  const int b = blockIdx.x;
  if (need && !need[b]) {
    if (threadIdx.x == 0) pneed[b] = 0;
    return;
  }
  const int nb = t.nb, Wd = nb + 2 * Gi, W2 = Wd * Wd, hb = nb / 2, tid = threadIdx.x, bd = blockDim.x;
  const size_t np = (size_t)Wd * W2, nb3 = (size_t)nb * nb * nb;
  const int L = __ldg(t.lev + b);
  const int ax = __ldg(t.anc + 3 * b) * nb, ay = __ldg(t.anc + 3 * b + 1) * nb, az = __ldg(t.anc + 3 * b + 2) * nb;
  __shared__ PrepTab T;
  __shared__ PrepPlan plan;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int capU = sum_bytes / (int)sizeof(U), capP = sum_bytes / (int)sizeof(TP);
  if (tid == 0) T.cmask = 0, T.ce = 0;
  if (BND && tid == 0) T.miss = 0;
  __syncthreads();
  // owners of the 27 block-sized regions around b (same or coarser leaves own
  // a whole region); regions beyond a physical boundary count as the block
  if (tid < 27) {
    const int r = tid;
    const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1}, an[3] = {ax / nb, ay / nb, az / nb};
    int g[3], e = 0;
    bool parent = true;  // the direction of a parent-level neighbour
    for (int d = 0; d < 3; ++d) {
      g[d] = an[d] * nb + (dd[d] < 0 ? -1 : dd[d] > 0 ? nb : 0);
      const int s = (an[d] & 1) ? 1 : -1;
      if (dd[d] == s) e |= 1 << d;
      else parent &= dd[d] == 0;
    }
    const int o = BND && beyond3(t, L, g) ? b : owner(t, L, g[0], g[1], g[2], b);
    const int Lo = __ldg(t.lev + o);
    T.rslot[r] = o, T.rlev[r] = Lo;
    long long base = 0;
    int mul = 0;
    if (Lo == L || Lo == L - 1) {
      mul = Lo == L ? 2 : 1;
      int st = 1;
      base = (long long)o * (long long)nb3;
      for (int d = 0; d < 3; ++d, st *= nb) {
        const bool out = (e >> d) & 1;
        const int od = an[d] & 1;
        // same level: 2 q relative to the region; coarser: q relative to the
        // neighbour of the parent (or, along this axis, the parent's own range)
        base += (long long)st * (Lo == L ? -dd[d] * nb : out ? (od ? -hb : nb) : od * hb);
      }
    }
    T.rbase[r] = base, T.rmul[r] = mul;
    if (r != 13) {
      if (Lo < L - 1 || Lo > L + 1) atomicOr(err, 4);
      if (Lo < L) atomicOr(&T.cmask, 1 << r);
      if (Lo < L && parent && e) atomicOr(&T.ce, 1 << e);
    }
    for (int d = 0; d < 3; ++d) T.ranc[r][d] = __ldg(t.anc + 3 * o + d);
    if (r < 3) T.s[r] = (an[r] & 1) ? 1 : -1, T.odd[r] = an[r] & 1;
  }
  __syncthreads();
  const int mask = T.cmask, ce = T.ce;
  if (tid == 0) cmask_out[b] = mask, pneed[b] = mask ? 1 : 0;
  if (only_coarse && !mask) return;
  // one warp per phase builds its boxes (a lane per direction); the sub-blocks
  // of finer regions (-1: refined further) are looked up meanwhile
  if (!mask) {
  } else if (tid < 32) {
    const int e = tid;
    const bool on = e < 8 && ((ce >> e) & 1);
    RefBox B;
    int nch = 0, step = 2, lc0 = 0, lenc = 0, plane = 0;
    if (on) {
      int l[3], m[3];
      for (int d = 0; d < 3; ++d) {
        const bool od = (e >> d) & 1;
        l[d] = od ? (T.s[d] > 0 ? nb : -Gi) : (T.s[d] > 0 ? -Gi : 0);
        m[d] = od ? Gi : nb + Gi;
      }
      B.a = (e & 1) ? 0 : (e & 2) ? 1 : 2;
      B.b = B.a == 0 ? 1 : 0, B.c = 3 - B.a - B.b;
      B.la = l[B.a], B.na = m[B.a], B.lb = l[B.b], B.nb = m[B.b];
      B.cb = (B.lb - ko) >> 1, B.mb = ((B.lb + B.nb - 1 + ko) >> 1) - B.cb + 1;
      B.mbp = B.mb | 1, B.nbp = B.nb | 1;
      B.S = (B.a == 0 ? B.na * B.nb : B.na * B.nbp) | 1;
      B.dmb = divm(B.mb).m, B.dna = divm(B.na).m, B.dnb = divm(B.nb).m, B.dl3 = divm(B.na * B.nb).m;
      // cut along c: mc planes of both sums
      plane = B.na * B.mbp + B.S;
      step = max(2 * (capU / plane - ko - 2 - (BND ? N : 0)), 2);
      lc0 = l[B.c], lenc = m[B.c], nch = (lenc + step - 1) / step;
    }
    int pos = nch;  // first box of this direction
    for (int w = 1; w < 8; w <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, pos, w);
      if (tid >= w) pos += v;
    }
    const int total = __shfl_sync(0xffffffffu, pos, 7);
    pos -= nch;
    for (int c0 = 0; c0 < lenc; c0 += step) {
      B.lc = lc0 + c0, B.nc = min(step, lenc - c0);
      B.cc = (B.lc - ko) >> 1;
      int ce1 = ((B.lc + B.nc - 1 + ko) >> 1) + 1;
      if (BND) {  // the polynomial's nodes, where the chunk reaches beyond the domain
        const int anc = (B.c == 0 ? ax : B.c == 1 ? ay : az) / 2;
        const int first = bc_first(t, anc, B.c), end = bc_end(t, L - 1, anc, B.c);
        if (B.cc < first) ce1 = max(ce1, first + N);
        if (ce1 > end) B.cc = min(B.cc, end - N);
      }
      B.mc = ce1 - B.cc;
      B.dl2 = divm(B.na * B.mc).m;
      B.off = plane * B.mc;  // (its size, until the batches are laid out)
      plan.ref[pos++] = B;
    }
    __syncwarp();
    if (tid == 0) {
      int used = 0, open = 0;
      for (int n = 0; n < total; ++n) {
        const int sz = plan.ref[n].off;
        if (n > open && used + sz > capU) {
          for (int q = open; q < n; ++q) plan.refnext[q] = n;
          open = n, used = 0;
        }
        plan.ref[n].off = used, used += sz;
      }
      for (int q = open; q < total; ++q) plan.refnext[q] = total;
      plan.nref = total;
    }
  } else if (tid < 64) {
    outward_boxes(plan.band, ce, T.s, nb, W::ext_b, W::ext_f);
  } else if (tid < 96) {
    const int gp = min(Gpush, hb), q = tid - 64;
    outward_boxes(plan.push, ce, T.s, hb, gp, gp);
    __syncwarp();
    if constexpr (NT != 0) {
      constexpr int hH = W::hwH;
      if (q < plan.push.n) {
        const int *lo = plan.push.lo[q], *hi = plan.push.hi[q];
        const int e0 = hi[0] - lo[0], e1 = hi[1] - lo[1], e2 = hi[2] - lo[2];
        PushBox B;
        B.a = e0 <= e1 && e0 <= e2 ? 0 : e1 <= e2 ? 1 : 2, B.b = B.a == 0 ? 1 : 0, B.c = 3 - B.a - B.b;
        B.na = hi[B.a] - lo[B.a], B.nb = hi[B.b] - lo[B.b], B.nc = hi[B.c] - lo[B.c], B.la = lo[B.a];
        B.fb = 2 * B.nb - 1 + 2 * hH, B.fc = 2 * B.nc - 1 + 2 * hH;
        B.layers = max(1, min(min(B.na, PUSH_LAYERS), capP / (B.fc * (B.fb + B.nb))));
        const int sA = B.a == 0 ? 1 : B.a == 1 ? Wd : W2, sB = B.b == 0 ? 1 : Wd, sC = B.c == 1 ? Wd : W2;
        B.base = (2 * B.la + Gi) * sA + (2 * lo[B.b] - hH + Gi) * sB + (2 * lo[B.c] - hH + Gi) * sC;
        B.dfb = divm(B.fb).m, B.dfc = divm(B.fc).m, B.drb = divm((B.nb + 3) >> 2).m, B.dnb = divm(B.nb).m;
        B.dnc = divm(B.nc).m;
        B.off = B.layers * B.fc * (B.fb + B.nb);  // (its size, until the batches are laid out)
        plan.pbox[q] = B;
      }
      // the neighbour in direction f holds point p at p - hb or p + nb along the
      // axes of f, in the leaf's half along the others
      if (q >= 8 && q < 16) {
        const int f = q - 8;
        const bool on = f && ((ce >> f) & 1);
        const unsigned have = __ballot_sync(0x0000ff00u, on);
        if (on) {
          int r2 = 13, st = 1;
          long long x = 0;
          for (int d = 0; d < 3; ++d, st *= Wd) {
            const bool od = (f >> d) & 1;
            if (od) r2 += T.s[d] * (d == 0 ? 1 : d == 1 ? 3 : 9);
            x += (long long)st * ((od ? (T.s[d] > 0 ? -hb : nb) : T.odd[d] * hb) + Gi);
          }
          const int at = __popc(have & ((1u << q) - 1u));
          plan.qdir[at] = f, plan.qbase[at] = (long long)T.rslot[r2] * (long long)np + x;
        }
        if (q == 15) plan.nq = __popc(have);
      }
      __syncwarp();
      if (q == 0) {
        const int n = plan.push.n;
        int used = 0, open = 0;
        for (int e = 0; e < n; ++e) {
          const int sz = plan.pbox[e].off;
          if (e > open && used + sz > capP) plan.pbox[open].next = e, open = e, used = 0;
          plan.pbox[e].off = used, used += sz;
        }
        if (n) plan.pbox[open].next = n;
        plan.npb = n;
      }
    }
  }
  for (int q = tid; q < 216; q += bd) {
    const int r = q >> 3, h = q & 7;
    int o2 = -1;
    if (T.rlev[r] == L + 1 && L < t.M) {
      const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
      int g[3];
      for (int d = 0; d < 3; ++d) g[d] = 2 * (T.ranc[13][d] + dd[d]) * nb + ((h >> d) & 1) * nb;
      o2 = owner(t, L + 1, g[0], g[1], g[2], b);
      if (o2 < 0 || o2 >= t.nleaf || __ldg(t.lev + o2) != L + 1) o2 = -1;
    }
    T.rsub[r][h] = o2;
  }
  __syncthreads();
  TP *Pb = P + (size_t)b * np;
  // The band is ext_b or ext_f layers deep and reads hwG further; the push starts
  // 2 Gpush layers from the side and reads hwH further.  In blocks less than twice
  // as wide the tests cost more than they leave out (11 019 leaves of 16^3 with
  // 4.2, reach 10: 738 -> 766 us).
  const int reach = max(max(W::ext_b, W::ext_f) + W::hwG, only_coarse == 1 && NT ? 2 * min(Gpush, hb) + W::hwH : 0);
  if (!BND && sizeof(TP) == 4 && only_coarse && 2 * reach <= nb) gather_block<true>(t, T, phi, Pb, b, L, Gi, reach, err);
  else gather_block<false>(t, T, phi, Pb, b, L, Gi, 0, err);
  if (!mask) return;
  // substitution jobs: one thread each (degree 1: classes x, y, z; 2: xy, xz,
  // yz; 3: xyz), then one thread lays out their sums
  {
    const int nbx = plan.band.n, cls[7] = {1, 2, 4, 3, 5, 6, 7};
    if (tid < 7 * nbx) {
      const int k = tid < 3 * nbx ? tid % 3 : tid < 6 * nbx ? 3 + (tid - 3 * nbx) % 3 : 6;
      const int e = tid < 3 * nbx ? tid / 3 : tid < 6 * nbx ? (tid - 3 * nbx) / 3 : tid - 6 * nbx;
      sub_job_build(plan.job[tid], plan.axes, e, plan.band.lo[e], plan.band.hi[e], cls[k], W::hwG, sub_flat<TP> ? plan.band.flat[e] : 0);
    }
  }
  // layout of the substitution sums: batches within a degree (by one thread,
  // while the others refine)
  auto sub_layout = [&]() {
    const int nbx = plan.band.n;
    int j = 0;
    for (int deg = 1; deg <= 3; ++deg) {
      const int end = j + (deg < 3 ? 3 : 1) * nbx;
      plan.job0[deg - 1] = j;
      int used = 0, open = j;
      for (; j < end; ++j) {
        SubJob &J = plan.job[j];
        const int sz = deg == 1 ? 0 : J.n[0] + (deg == 3 ? J.n[1] : 0);
        if (j > open && used + sz > capP) {
          plan.job[open].next = j;
          open = j, used = 0;
        }
        J.off = used, used += sz;
      }
      if (open < end) plan.job[open].next = end;
    }
    plan.job0[3] = j;
  };
  const long long lin1 = nb, lin2 = (long long)nb * nb;
  // coarse values beyond a physical boundary (the leaf's own parent range or
  // its lateral ghosts): the polynomial is applied to the sums along b and c;
  // float pairs (FP64 blocks of an FP32 field) go point by point instead
  const bool cbc = BND && bc_touches(t, L, ax, ay, az, -Gi - ko - 1, nb + Gi + ko + 1);
  bool bad = false;  // a refined value is NaN: one flag per CTA, set below
  if (BND && cbc && sizeof(TI) != sizeof(TP)) {
    __syncthreads();
    if (tid == bd - 1) sub_layout();
    for (int e = 0; e < plan.nref; ++e) {
      const RefBox &B = plan.ref[e];
      const DivM dna = divm(B.na), dnb = divm(B.nb);
      for (int idx = tid; idx < B.na * B.nb * B.nc; idx += bd) {
        const int r = divq(idx, dna), kc = divq(r, dnb);
        int p[3];
        p[B.a] = B.la + idx - r * B.na, p[B.b] = B.lb + r - kc * B.nb, p[B.c] = B.lc + kc;
        const TP v = refine_point<TI, TP, N, NT>(t, phi, L, ax + p[0], ay + p[1], az + p[2], err, b);
        bad |= nan_bits(v);
        Pb[(p[0] + Gi) + Wd * (p[1] + Gi) + W2 * (p[2] + Gi)] = v;
      }
    }
  } else {
    for (int e0 = 0; e0 < plan.nref;) {
      const int e1 = plan.refnext[e0];
      U *UB = reinterpret_cast<U *>(smraw);
      // pass 1: one thread per coarse column along a.  The column's values come
      // from two runs (the coarser region, and the block's side of the face);
      // its fine points go to U1.
      int rot = 0;
      for (int e = e0; e < e1; ++e) {
        const RefBox &B = plan.ref[e];
        const int a = B.a, ncol = B.mb * B.mc, na = B.na, par = B.la & 1;
        const int ca = (B.la - ko) >> 1, cna = ((B.la + na - 1 + ko) >> 1) - ca + 1;
        const int sta = a == 0 ? 1 : a == 1 ? nb : nb * nb;
        const int pitch = B.mbp;
        int idx = tid - rot;
        if (idx < 0) idx += bd;
        rot = turn(rot, ncol, bd);
        for (; idx < ncol; idx += bd) {
          const int kc = divq(idx, DivM{B.dmb, B.mb}), jb = idx - kc * B.mb;
          int q[3];
          q[B.b] = B.cb + jb, q[B.c] = B.cc + kc, q[a] = ca;
          // regions along b and c; the run along a changes region at the face
          int rr = 0, ra = a == 0 ? 1 : a == 1 ? 3 : 9;
          bool ok = 2 * ca >= -nb && 2 * (ca + cna - 1) < 2 * nb;
          for (int d = 0; d < 3; ++d) {
            if (d == a) continue;
            const int f = 2 * q[d];
            ok &= f >= -nb && f < 2 * nb;
            rr += (f < 0 ? 0 : f >= nb ? 2 : 1) * (d == 0 ? 1 : d == 1 ? 3 : 9);
          }
          const int cut = B.la < 0 ? 0 : hb;  // first coarse point of the upper run
          const int r0 = rr + (B.la < 0 ? 0 : 1) * ra, r1 = r0 + ra;
          if (ok) ok = T.rmul[r0] && T.rmul[r1];
          U *d = UB + B.off + jb + pitch * na * kc;
          if (!ok && NARROW) {  // a finer leaf or a region beyond the neighbours
            auto at = [&](int qa) {
              q[a] = qa;
              return RS::from(prep_fetch<BND, TI>(t, T, phi, b, L, L - 1, q[0], q[1], q[2], err));
            };
            refine_run<N, NT, RS>(at, B.la, na, [&](int ia, U v) { d[pitch * ia] = RS::norm(v); });
            continue;
          }
          if (!ok) {
            for (int ia = 0; ia < na; ++ia) {
              U s = RS::zero();
              const int f = B.la + ia;
              for (int o = (f & 1) ? -ko : 0; o <= ((f & 1) ? ko : 0); o += 2) {
                q[a] = (f + o) >> 1;
                s = RS::acc(s, (f & 1) ? W::K(o) : 1.0,
                            RS::from(prep_fetch<BND, TI>(t, T, phi, b, L, L - 1, q[0], q[1], q[2], err)));
              }
              d[pitch * ia] = RS::norm(s);
            }
            continue;
          }
          TI v[MR_MAX_SHELL];
          {
            const long long lin = q[0] + lin1 * q[1] + lin2 * q[2];
            const TI *p0 = phi + (T.rbase[r0] + T.rmul[r0] * lin), *p1 = phi + (T.rbase[r1] + T.rmul[r1] * lin);
            const int s0 = T.rmul[r0] * sta, s1 = T.rmul[r1] * sta, n0 = cut - ca;
#pragma unroll
            for (int u = 0; u < MR_MAX_SHELL; ++u) v[u] = u < cna ? ld(u < n0 ? p0 + u * s0 : p1 + u * s1) : TI(0);
          }
          auto column = [&](auto parity) {
            constexpr int PAR = decltype(parity)::x, base = (PAR - ko) >> 1;
#pragma unroll
            for (int ia = 0; ia < MR_MAX_SHELL; ++ia) {
              if (ia >= na) break;
              U s;
              if ((PAR + ia) & 1) {
                s = RS::zero();
#pragma unroll
                for (int o = -ko; o <= ko; o += 2) {
                  const int x = ((PAR + ia + o) >> 1) - base;
                  if (x < MR_MAX_SHELL) s = RS::acc(s, W::K(o), RS::from(v[x]));
                }
                s = RS::norm(s);
              } else {
                const int x = ((PAR + ia) >> 1) - base;
                s = RS::from(x < MR_MAX_SHELL ? v[x] : TI(0));
              }
              d[pitch * ia] = s;
            }
          };
          if (par) column(Cls<1, 0, 0>());
          else column(Cls<0, 0, 0>());
        }
      }
      __syncthreads();
      if (e0 == 0 && tid == bd - 1) sub_layout();
      if constexpr (BND && sizeof(TI) == sizeof(TP))
        if (cbc)
          for (int e = e0; e < e1; ++e)
            bc_sums<N>(t, L - 1, plan.ref[e], ax / 2, ay / 2, az / 2, UB + plan.ref[e].off);
      // pass 2: along b, U1 -> U2; segments of 8 coarse points, a register
      // window of N coarse values, two fine points per step
      rot = 0;
      for (int e = e0; e < e1; ++e) {
        const RefBox &B = plan.ref[e];
        const int na = B.na, lines = na * B.mc, nseg = (B.nb + 15) >> 4, n = lines * nseg;
        const DivM dl{B.dl2, lines}, dna{B.dna, na};
        const int sb = B.a == 0 ? na : 1, sa = B.a == 0 ? 1 : B.nbp;
        const U *U1 = UB + B.off;
        U *U2 = UB + B.off + na * B.mbp * B.mc;
        int idx = tid - rot;
        if (idx < 0) idx += bd;
        rot = turn(rot, n, bd);
        for (; idx < n; idx += bd) {
          const int sg = divq(idx, dl), ln = idx - sg * lines, kc = divq(ln, dna), ia = ln - kc * na;
          const int f0 = B.lb + 16 * sg, n1 = min(16, B.nb - 16 * sg);
          const U *src = U1 + B.mbp * ln - B.cb;  // (line kc, ia: U1 pitch mbp)
          U *dst = U2 + B.S * kc + sa * ia + sb * (16 * sg);
          refine_run<N, NT, RS>(src, 1, f0, n1, [&](int m, U v) { dst[sb * m] = RS::norm(v); });
        }
      }
      __syncthreads();
      // pass 3: along c, U2 -> padded block
      rot = 0;
      for (int e = e0; e < e1; ++e) {
        const RefBox &B = plan.ref[e];
        const int na = B.na, lines = na * B.nb, nseg = (B.nc + 15) >> 4, n = lines * nseg;
        const int n1d = B.a == 0 ? na : B.nb;  // dimension that varies fastest over threads
        const DivM dl{B.dl3, lines}, df{B.a == 0 ? B.dna : B.dnb, n1d};
        const int sb = B.a == 0 ? na : 1, sa = B.a == 0 ? 1 : B.nbp;
        const int psa = B.a == 0 ? 1 : B.a == 1 ? Wd : W2, psb = B.b == 0 ? 1 : B.b == 1 ? Wd : W2,
                  psc = B.c == 0 ? 1 : B.c == 1 ? Wd : W2;
        const U *U2 = UB + B.off + na * B.mbp * B.mc;
        int idx = tid - rot;
        if (idx < 0) idx += bd;
        rot = turn(rot, n, bd);
        for (; idx < n; idx += bd) {
          const int sg = divq(idx, dl), ln = idx - sg * lines, hi = divq(ln, df), lo = ln - hi * n1d;
          const int ia = B.a == 0 ? lo : hi, ib = B.a == 0 ? hi : lo;
          const int f0 = B.lc + 16 * sg, n1 = min(16, B.nc - 16 * sg);
          TP *dst = Pb + (B.la + ia + Gi) * psa + (B.lb + ib + Gi) * psb + (f0 + Gi) * psc;
          refine_run<N, NT, RS>(U2 + sa * ia + sb * ib - B.S * B.cc, B.S, f0, n1, [&](int m, U v) {
            const TP d = RS::value(v);
            bad |= nan_bits(d);
            dst[psc * m] = d;
          });
        }
      }
      __syncthreads();
      e0 = e1;
    }
  }
  // (a NaN of the field itself is no error on grids with physical boundaries)
  if (__syncthreads_or(bad) && (!BND || T.miss) && tid == 0) atomicOr(err, 2);
  if (BND && bc_touches(t, L, ax, ay, az, -Gi, nb + Gi))
    bc_box<N>(t, L, ax, ay, az, Pb + Gi * (1 + Wd + W2), Wd, W2, -Gi, -Gi, -Gi, Wd, Wd, Wd);
  // substitution, degree by degree (a point of degree d reads lower degrees
  // only, so the classes of one degree are independent)
  for (int deg = 1; deg <= 3; ++deg)
    subst_jobs<N, NT, TP>(Pb, Wd, Gi, plan.job, plan.axes, plan.job0[deg - 1], plan.job0[deg], reinterpret_cast<TP *>(smraw), capP);
  // (N.0: H^a is the identity and even points are never substituted, so the
  // coincident values the gather took are already the coarsened ones)
  if (only_coarse == 2 || NT == 0) return;
  // Part 2: H^a coarsening of the padded block at the coarse points of the push
  // boxes: one thread loads a fine column along a and sums every layer from it;
  // along b a thread sums four points from one window; along c one point, which
  // goes to the side buffer of every coarser neighbour in whose shell it lies.
  if constexpr (NT != 0) {
    constexpr int hH = W::hwH;
    const int gp = min(Gpush, hb), npb = plan.npb, nq = plan.nq;
    TP *buf = reinterpret_cast<TP *>(smraw);
    for (int e0 = 0; e0 < npb;) {
      const int e1 = plan.pbox[e0].next;
      bool more = true;
      for (int it = 0; more; ++it) {
        more = false;
        int rot = 0;
        for (int e = e0; e < e1; ++e) {
          const PushBox &B = plan.pbox[e];
          const int l0 = it * B.layers, nl = min(B.layers, B.na - l0), n = B.fc * B.fb;
          more |= l0 + B.layers < B.na;
          if (nl <= 0) continue;
          int idx = tid - rot;
          if (idx < 0) idx += bd;
          rot = turn(rot, n, bd);
          const int sA = B.a == 0 ? 1 : B.a == 1 ? Wd : W2, sB = B.b == 0 ? 1 : Wd, sC = B.c == 1 ? Wd : W2;
          TP *A = buf + B.off;  // [l][fc][fb]
          for (; idx < n; idx += bd) {
            const int ic = divq(idx, DivM{B.dfb, B.fb}), ib = idx - ic * B.fb;
            coarsen_run<N, NT, PUSH_LAYERS>(Pb + B.base + 2 * l0 * sA + ib * sB + ic * sC, sA, nl,
                                            [&](int l, TP v) { A[l * n + idx] = v; });
          }
        }
        __syncthreads();
        rot = 0;
        for (int e = e0; e < e1; ++e) {
          const PushBox &B = plan.pbox[e];
          const int nl = min(B.layers, B.na - it * B.layers), rb = (B.nb + 3) >> 2, n = nl * B.fc * rb;
          if (nl <= 0) continue;
          int idx = tid - rot;
          if (idx < 0) idx += bd;
          rot = turn(rot, n, bd);
          const TP *A = buf + B.off + hH;
          TP *D = buf + B.off + B.layers * B.fc * B.fb;  // [l][fc][nb]
          for (; idx < n; idx += bd) {
            const int r = divq(idx, DivM{B.drb, rb}), ib = 4 * (idx - r * rb);
            TP *d = D + r * B.nb + ib;
            coarsen_run<N, NT, 4>(A + r * B.fb + 2 * ib, 1, min(4, B.nb - ib), [&](int m, TP v) { d[m] = v; });
          }
        }
        __syncthreads();
        rot = 0;
        for (int e = e0; e < e1; ++e) {
          const PushBox &B = plan.pbox[e];
          const int l0 = it * B.layers, nl = min(B.layers, B.na - l0), n = nl * B.nc * B.nb;
          if (nl <= 0) continue;
          int idx = tid - rot;
          if (idx < 0) idx += bd;
          rot = turn(rot, n, bd);
          const TP *D = buf + B.off + B.layers * B.fc * B.fb;
          const int lob = plan.push.lo[e][B.b], loc = plan.push.lo[e][B.c];
          for (; idx < n; idx += bd) {
            const int r = divq(idx, DivM{B.dnb, B.nb}), l = divq(r, DivM{B.dnc, B.nc}), ib = idx - r * B.nb,
                      ic = r - l * B.nc;
            const TP sv = tap_sum<N, NT, FK_H>(D + (l * B.fc + 2 * ic + hH) * B.nb + ib, B.nb);
            const int va = B.la + l0 + l, vb = lob + ib, vc = loc + ic;
            const int px = B.a == 0 ? va : vb, py = B.a == 0 ? vb : B.a == 1 ? va : vc, pz = B.a == 2 ? va : vc;
            const int inb = (T.s[0] > 0 ? px >= hb - gp : px < gp) | (T.s[1] > 0 ? py >= hb - gp : py < gp) << 1 |
                            (T.s[2] > 0 ? pz >= hb - gp : pz < gp) << 2;
            const int lin = px + Wd * py + W2 * pz;
            for (int f = 0; f < nq; ++f)
              if (!(plan.qdir[f] & ~inb)) Q[plan.qbase[f] + lin] = sv;
          }
        }
        __syncthreads();
      }
      e0 = e1;
    }
  }
}

// Shared memory of the pre-pass's sums, or what a chunk of the largest box
// takes.  Four CTAs of 256 threads per SM with FP32 blocks, three with FP64
// ones; the sums stay small enough that the L1 cache keeps a share of the SM's
// memory, since the block is read back through it: without the gather the kernel took
// 312 us at 3 424 leaves of 24^3 with 6.2 with 27 or 34 KB, 417 with 42 KB (L1 almost
// gone) and 323 with 54 KB (three CTAs).
static size_t prep_sum_bytes(int N, int nb, int Gi, size_t es, bool bounded) {
  const int ko = N - 1, m = nb + Gi, mb = ((m - 1 + 2 * ko) >> 1) + 2;
  const size_t plane = (size_t)Gi * (mb | 1) + ((size_t)Gi * (m | 1) | 1);
  return std::max<size_t>(es == 4 ? 34 * 1024 : 48 * 1024, (plane * prep_min_planes(N, bounded) * es + 15) & ~(size_t)15);
}

// Merge the part-2 values into P (only the neighbour regions owned by finer
// leaves hold them) and write the substituted interior back to the field of
// leaves that have a coarser neighbour.
template <typename TO, typename TP, int N, int NT, bool BND>
__global__ void __launch_bounds__(512) k_merge(Tree t, TP *__restrict__ P, const TP *__restrict__ Q,
                                               int Gi, int G, const int *__restrict__ cmask,
                                               TO *__restrict__ phi_out, const int *__restrict__ need) {
  const int b = blockIdx.x;
  if (need && !need[b]) return;
  const int nb = t.nb, Wd = nb + 2 * Gi;
  const size_t np = (size_t)Wd * Wd * Wd;
  const int L = __ldg(t.lev + b);
  __shared__ int rfin[27];
  if (threadIdx.x < 27) {
    const int r = threadIdx.x;
    const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
    int g[3];
    for (int d = 0; d < 3; ++d) g[d] = __ldg(t.anc + 3 * b + d) * nb + (dd[d] < 0 ? -1 : dd[d] > 0 ? nb : 0);
    rfin[r] = r != 13 && !(BND && beyond3(t, L, g)) && __ldg(t.lev + owner(t, L, g[0], g[1], g[2], b)) > L;
  }
  __syncthreads();
  // (N.0 pushes nothing: the gather's coincident values stand)
  for (int r = 0; r < 27; ++r) {
    if (NT == 0 || !rfin[r]) continue;
    const int dd[3] = {r % 3 - 1, (r / 3) % 3 - 1, r / 9 - 1};
    int lo[3], ext[3];
    for (int d = 0; d < 3; ++d) {
      lo[d] = dd[d] < 0 ? -G : dd[d] > 0 ? nb : 0;
      ext[d] = dd[d] ? G : nb;
    }
    const int cnt = ext[0] * ext[1] * ext[2];
    const DivM de0 = divm(ext[0]), de1 = divm(ext[1]);
    for (int p = threadIdx.x; p < cnt; p += blockDim.x) {
      const int r = divq(p, de0), z = divq(r, de1);
      const int i = lo[0] + p - r * ext[0], j = lo[1] + r - z * ext[1], k = lo[2] + z;
      const size_t q = (size_t)b * np + (i + Gi) + Wd * ((j + Gi) + (size_t)Wd * (k + Gi));
      P[q] = Q[q];
    }
  }
  if constexpr (BND) {
    const int ax = __ldg(t.anc + 3 * b) * nb, ay = __ldg(t.anc + 3 * b + 1) * nb, az = __ldg(t.anc + 3 * b + 2) * nb;
    if (bc_touches(t, L, ax, ay, az, -G, nb + G))
      bc_box<N>(t, L, ax, ay, az, P + b * np + Gi * (1 + Wd + Wd * Wd), Wd, Wd * Wd, -G, -G, -G, nb + 2 * G,
                nb + 2 * G, nb + 2 * G);
  }
  if (phi_out && cmask[b]) {
    const DivM dnb = divm(nb);
    for (int p = threadIdx.x; p < nb * nb * nb; p += blockDim.x) {
      const int r = divq(p, dnb), k = divq(r, dnb), i = p - r * nb, j = r - k * nb;
      if (!((i | j | k) & 1)) continue;  // 0-degree points are never substituted
      phi_out[(size_t)b * nb * nb * nb + p] =
          TO(P[(size_t)b * np + (i + Gi) + Wd * ((j + Gi) + (size_t)Wd * (k + Gi))]);
    }
  }
}

// The requested shell G of the padded blocks (internal shell Gi).  One thread
// per (x, y) column, so a point costs a load, a store and two additions; bound
// by the copy.
template <typename TO, typename TP>
__global__ void __launch_bounds__(256) k_crop(const TP *__restrict__ P, int Gi, TO *__restrict__ out, int G, int nb) {
  const int b = blockIdx.x;
  const int Wd = nb + 2 * Gi, Wg = nb + 2 * G, W2 = Wd * Wd, Wg2 = Wg * Wg, o = Gi - G;
  const TP *src = P + (size_t)b * Wd * W2 + o * (1 + Wd + (size_t)W2);
  TO *dst = out + (size_t)b * Wg * Wg2;
  const DivM dg = divm(Wg);
  for (int c = threadIdx.x; c < Wg2; c += blockDim.x) {
    const int j = divq(c, dg);
    const TP *s = src + c - j * Wg + Wd * j;
    TO *d = dst + c;
#pragma unroll 6
    for (int k = 0; k < Wg; ++k) d[(size_t)k * Wg2] = TO(__ldg(s + (size_t)k * W2));
  }
}

// internal shell: the requested one, the substitution reach, and what the
// part-2 coarsening of a finer neighbour reads
static int internal_shell(int N, int Nt, int G, int nb) {
  const int hwH = Nt ? N : 0, hwG = N - 1;
  int gi = G;
  if (hwH > gi) gi = hwH;
  if (hwG > gi) gi = hwG;
  if (2 * G + hwH - nb > gi) gi = 2 * G + hwH - nb;
  return gi;
}

template <typename TI, typename TP, int N, int NT>
int ghost_impl(mr_grid *g, const TI *phi_in, TI *phi_out, int G, TP *P, TP *Q, int Gi, int only_coarse,
                      const int *need) {
  Tree t = tree_view(g);
  const int n = g->nleaf, nb = g->desc.nb;
  int *err = g->counter + 1;
  // (bounded grids have their own instantiations: their out-of-line calls would
  // cost the others registers)
  auto prep = t.bnd ? k_prep<TI, TP, N, NT, true, false> : k_prep<TI, TP, N, NT, false, false>;
  if constexpr (N == 6)  // (shorter filters never reach that far)
    if (!t.bnd && prep_narrow(N, nb, Gi)) prep = k_prep<TI, TP, N, NT, false, true>;
  const auto merge = t.bnd ? k_merge<TI, TP, N, NT, true> : k_merge<TI, TP, N, NT, false>;
  const size_t sm = prep_sum_bytes(N, nb, Gi, sizeof(TP), t.bnd != 0);
  constexpr size_t most = 200 * 1024;  // leaves room for the kernel's static tables
  if (sm > most) return MR_ERR_UNSUPPORTED;
  if (smem_limit(prep, most, "k_prep smem")) return MR_ERR_CUDA;
  const int tp = sizeof(TP) == 4 ? 4 : sizeof(TI) == 4 ? 5 : 8;
  // 256 threads per leaf; more where the grid does not fill the chip (a leaf's
  // phases are latency-bound: 120 leaves of 16^3 with 4.2)
  const int big = sizeof(TP) == 4 ? 512 : 384, many = n > 2 * 152, cp[2] = {many ? 256 : big, many ? 128 : 256};
  const int bnd = t.bnd != 0;
  const int thp = tune_threads(g, TuneKey{1, N, NT, nb, tp, Gi, only_coarse + 4 * many + 8 * bnd}, cp, 2, [&](int th) {
    prep<<<n, th, sm, g->stream>>>(t, phi_in, P, Q, Gi, G, only_coarse, g->cmask, err, need, g->pneed, (int)sm);
  });
  MR_LAUNCH(g, MRK_PART1, prep<<<n, thp, sm, g->stream>>>(t, phi_in, P, Q, Gi, G, only_coarse, g->cmask, err, need,
                                                          g->pneed, (int)sm));
  if (check_cuda(cudaGetLastError(), "k_prep")) return MR_ERR_CUDA;
  if (only_coarse != 2) {  // the substitution-only pass fills no shell
    const double wd = nb + 2.0 * G;  // the requested shell (not the internal one)
    const double bytes = (wd * wd * wd - (double)nb * nb * nb) * (double)(sizeof(TI) + sizeof(TP));
    count_units(g, MRK_PART1, g->pneed, n, bytes);
    if (!only_coarse) count_units(g, MRK_PART2, need, n, bytes, g->pneed);  // leaves that only gather
  }
  if (only_coarse) return MR_OK;
  static const int cm[3] = {256, 128, 512};
  const int thm = tune_threads(g, TuneKey{5, N, NT, nb, tp, Gi, 8 * bnd}, cm, 3, [&](int th) {
    merge<<<n, th, 0, g->stream>>>(t, P, Q, Gi, G, g->cmask, phi_out, need);
  });
  MR_LAUNCH(g, MRK_MERGE, merge<<<n, thm, 0, g->stream>>>(t, P, Q, Gi, G, g->cmask, phi_out, need));
  if (check_cuda(cudaGetLastError(), "k_merge")) return MR_ERR_CUDA;
  return MR_OK;
}

}  // namespace mr
