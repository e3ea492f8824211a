// stage.cu -- the FP32 stage kernels: ghost faces + advection right-hand side
// + RK3 stage in one launch.  Two kernels compute the same values with the
// same arithmetic.  k_fused runs unless mr_set_stage_kernel or the autotuner, which
// times both, says otherwise; k_march took twice its time wherever both were timed
// (3 424 leaves of 24^3 with velocity fields 1 070 against 526 us, 42 400 with a
// constant velocity 8.5 against 3.99 ms, 11 019 of 16^3 1 047 against 477 us):
//   k_fused  one CTA per slab of a leaf: the slab with its ghosts in shared
//            memory, one thread per pair of grid lines;
//   k_march  one CTA per leaf marching through the block's z-planes: the six
//            face slabs in shared memory, one thread per (x, y) column with a
//            register window along z, x/y fluxes of one plane at a time.
#include <algorithm>

#include "stage_kernels.cuh"

namespace mr {

// ---------------------------------------------------------------------------
// Where the three ghost layers behind each face f = 2*axis + (0: -side, 1:
// +side) of leaf b come from:
//   same-level face  the neighbour's field;
//   coarser face     b's padded block: the pre-pass (k_prep) of every leaf next
//                    to a coarser one has refined the coarse values there;
//   finer face       the Part-2 coarsening pushed by the finer leaves into Q
//                    (lifted wavelets), or the coincident values of the finer
//                    leaves (N.0): one sub-block per face quadrant.
// ---------------------------------------------------------------------------
struct FaceSrc {
  int kind;              // 0: block stride, 1: padded stride, 2: finer leaves
  const float *base[4];  // address of the (virtual) block point (0, 0, 0)
};

__device__ __forceinline__ void face_sources(const Tree &t, int b, int L, const int *a, const float *phi,
                                             const float *P, const float *Q, int Gi, int lifted, FaceSrc *fs) {
  if (threadIdx.x >= 6) return;
  const int f = threadIdx.x, ax = f >> 1, sg = f & 1, nb = t.nb, Wd = nb + 2 * Gi;
  const long long nb3 = (long long)nb * nb * nb, np = (long long)Wd * Wd * Wd, org = Gi * (1 + Wd + (long long)Wd * Wd);
  const int st[3] = {1, nb, nb * nb};
  int g[3] = {a[0], a[1], a[2]};
  g[ax] += sg ? nb : -1;
  const int o = owner(t, L, g[0], g[1], g[2], b), Lo = __ldg(t.lev + o);
  FaceSrc s;
  s.base[1] = s.base[2] = s.base[3] = nullptr;
  if (Lo == L) {
    s.kind = 0, s.base[0] = phi + o * nb3 + (sg ? -nb : nb) * st[ax];
  } else if (Lo < L || lifted) {
    s.kind = 1, s.base[0] = (Lo < L ? P : Q) + b * np + org;
  } else {
    s.kind = 2;
    const int e1 = ax == 0 ? 1 : 0, e2 = ax == 2 ? 1 : 2;
    for (int q = 0; q < 4; ++q) {
      int h[3], gf[3];
      h[ax] = sg ? 0 : 1, h[e1] = q & 1, h[e2] = q >> 1;
      long long off = 0;
      for (int d = 0; d < 3; ++d) {
        const int dd = d == ax ? (sg ? 1 : -1) : 0;
        gf[d] = 2 * (a[d] + dd * nb) + h[d] * nb;
        off -= (long long)st[d] * (2 * dd + h[d]) * nb;
      }
      s.base[q] = phi + owner(t, L + 1, gf[0], gf[1], gf[2], b) * nb3 + off;
    }
  }
  fs[f] = s;
}

// ghost value behind face f at block-local point (i, j, k)
__device__ __forceinline__ const float *face_ptr(const FaceSrc &s, int ax, int i, int j, int k, int nb, int Wd) {
  if (s.kind == 0) return s.base[0] + i + nb * (j + nb * k);
  if (s.kind == 1) return s.base[0] + i + Wd * (j + Wd * k);
  const int hb = nb / 2, p = ax == 0 ? j : i, q = ax == 2 ? j : k;
  return s.base[(p >= hb) + 2 * (q >= hb)] + 2 * (i + nb * (j + nb * k));
}

// step from one z-plane to the next behind a face
__device__ __forceinline__ int face_step(const FaceSrc &s, int nb, int Wd) {
  return s.kind == 1 ? Wd * Wd : (nb * nb) << (s.kind == 2);
}

// one float from global to shared memory, asynchronously
__device__ __forceinline__ void copy_async(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
// two floats (both addresses multiples of 8)
__device__ __forceinline__ void copy_async2(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// n floats from global memory into the L2 cache (16-byte multiples)
__device__ __forceinline__ void prefetch_l2(const float *p, int n) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(4 * n) : "memory");
}

struct StageArgs {
  const float *phi, *P, *Q;
  int Gi, lifted;
  const int *cmask;
  const float *u;   // u^n (stages 1, 2), may alias out
  float *out;
  int stage, rhs_only;
  float dt, ux, uy, uz;
  const float *vpad;  // ghost-filled velocity components (shell 3) or null
  float nu, vscale;
  int diff;
  DivM dws;     // nb + 6
  float cu, cv;  // the stage: cu u^n + cv (phi + dt r)
};

// RK3-TVD stage (or the bare rhs r) of one cell with value c (uo: 0 in stage 0)
__device__ __forceinline__ float stage_value(const StageArgs &s, float c, float r, float uo) {
  return s.rhs_only ? r : fmaf(s.cv, fmaf(s.dt, r, c), s.cu * uo);
}

// ---------------------------------------------------------------------------
// k_fused: one CTA per slab of at most nz z-planes (the block is cut evenly, at
// least three planes to a slab).  Shared memory (floats):
//   T  [nz][nb+6][RS]    the slab's planes with their x and y ghosts
//   X  [nz][nb][XS]      half velocity u_x on the x rows (velocity fields);
//                        each row's walk leaves its flux differences there
//   Y  [nz][nb+6][nb]    likewise u_y on the y columns
// The x and y lines of the slab are walked first, a pair of lines per thread
// with the same code, then the z lines (pairs of neighbours in x), whose thread
// finishes its cells.  What one thread alone reads (the three values beyond each
// end of a z line, u_z, u^n) goes straight to its registers.  Bound by issued
// instructions (243 per point with velocity fields; 323 with one line per thread)
// and by the latency of the copies, which alone take 40 to 57 % of the time,
// overlapped with the walks of the other CTAs.  Slabs of a quarter block (half of a
// block of at most 16) keep three CTAs on an SM with velocity fields (more would
// spill), four without; the z walks' extra interface per slab costs 5 %.  Per launch
// (WENO-Z5): 3 424 leaves of 24^3 with velocity fields and 6.2 526 us (the block in
// shared memory as a whole, one line per thread: 1 660); 42 400 leaves with a constant
// velocity 3.99 ms (15.35); 11 019 leaves of 16^3 with velocity fields and 4.2 477 us
// (1 333); 1 272 leaves of 20^3 with diffusion and 2.2 74 us (104 in slabs of one line
// per thread).  Separate code for x and y walks, or unrolled z walks, is slower by a
// tenth (instruction cache).
// ---------------------------------------------------------------------------
// row pitch for n floats per row: twice an odd number (two-way bank conflicts at
// worst where neighbouring threads walk neighbouring rows)
__host__ __device__ constexpr int fused_pitch(int n) { return n + (n % 4 == 0 ? 2 : 0); }
__host__ __device__ constexpr int fused_smem_floats(int nb, int nz, bool vel) {
  return nz * (nb + 6) * fused_pitch(nb + 6) + 2 + nz * nb * fused_pitch(vel ? nb + 6 : nb) +
         nz * (vel ? nb + 6 : nb) * nb;
}

// largest block accepted (the slabs of 28^3 to 32^3 would fit an SM, too: 84 to 121 KB
// with velocity fields), and its slabs: a quarter of a large and half of a small one
constexpr int FUSED_MAX_NB = 26;
__host__ __device__ constexpr int fused_height(int nb) { return nb > 16 ? (nb + 3) / 4 : nb / 2; }

template <int SCHEME, bool VEL, bool LAP>
__global__ void __launch_bounds__(160, VEL ? 3 : 4) k_fused(Tree t, StageArgs s, int nz, int nslab) {
  const int b = blockIdx.x / nslab, sl = blockIdx.x - b * nslab;
  const int nb = t.nb, nb2 = nb * nb, Ws = nb + 6, W2 = Ws * Ws, RS = fused_pitch(nb + 6),
            XS = VEL ? RS : fused_pitch(nb), Wd = nb + 2 * s.Gi;
  const int k0 = sl * nb / nslab, nzs = (sl + 1) * nb / nslab - k0;
  const int tid = threadIdx.x, bd = blockDim.x, tst = Ws * RS;
  const int L = __ldg(t.lev + b);
  const int a[3] = {__ldg(t.anc + 3 * b) * nb, __ldg(t.anc + 3 * b + 1) * nb, __ldg(t.anc + 3 * b + 2) * nb};
  extern __shared__ __align__(16) float sm[];
  // (x = -3 is column 1 of a row, x = nb + 2 the first float of the next one)
  float *T = sm, *X = T + nz * tst + 2, *Y = X + nz * nb * XS;
  __shared__ FaceSrc fs[6];
  face_sources(t, b, L, a, s.phi, s.P, s.Q, s.Gi, s.lifted, fs);
  const DivM dnb = t.dnb;
  __shared__ float sh_h;
  if (tid == bd - 1) sh_h = (float)(t.tree_len / ((double)nb * (double)(1 << L)));
  // Values go to shared memory by asynchronous copies (all in flight at once;
  // nothing waits for memory before the barrier), two floats each where the
  // source allows it.  Each thread keeps its (x, y) and steps through the planes.
  // Interior of the leaf: the field, or the substituted block that the pre-pass wrote.
  const bool pad = s.cmask[b] != 0;
  const int sy = pad ? Wd : nb, sz = sy * sy;
  const float *src = (pad ? s.P + (size_t)b * Wd * sz + s.Gi * (1 + Wd + sz) : s.phi + (size_t)b * nb2 * nb) + k0 * sz;
  if (!pad || !(s.Gi & 1)) {  // rows at even addresses
    for (int c = tid; c < nb2 / 2; c += bd) {
      const int j = divq(2 * c, dnb), i = 2 * c - j * nb;
      const float *p = src + i + sy * j;
      float *tp = T + (j + 3) * RS + i + 4;
#pragma unroll 2
      for (int k = 0; k < nzs; ++k, p += sz, tp += tst) copy_async2(tp, p);
    }
  } else {
    for (int c = tid; c < nb2; c += bd) {
      const int j = divq(c, dnb), i = c - j * nb;
      const float *p = src + i + sy * j;
      float *tp = T + (j + 3) * RS + i + 4;
      for (int k = 0; k < nzs; ++k, p += sz, tp += tst) copy_async(tp, p);
    }
  }
  const float hscale = 0.5f * s.vscale;
  const size_t vblk = (size_t)W2 * Ws;
  const float *vb = VEL ? s.vpad + (size_t)b * vblk + k0 * W2 : nullptr;
  const size_t vcomp = (size_t)t.nleaf * vblk;
  // u_z and u^n are read one plane ahead of the z walks: less than memory's
  // latency, more than that of the L2 cache
  const bool rk_u = !s.rhs_only && s.stage > 0;
  if (tid == bd - 1) {
    if (VEL) prefetch_l2(vb + 2 * vcomp, (nzs + 6) * W2);
    if (rk_u) prefetch_l2(s.u + (size_t)b * nb2 * nb + k0 * nb2, nzs * nb2);
  }
  if (VEL) {
    const float *vx = vb + 3 * W2 + 3 * Ws, *vy = vb + vcomp + 3 * W2 + 3;
    for (int c = tid; c < nb * Ws / 2; c += bd) {
      const int j = divq(2 * c, s.dws), x = 2 * c - j * Ws;
      float *xp = X + j * XS + x;
      const float *px = vx + 2 * c;
#pragma unroll 2
      for (int k = 0; k < nzs; ++k, xp += nb * XS, px += W2) copy_async2(xp, px);
    }
    for (int c = tid; c < nb * Ws; c += bd) {
      const int j = divq(c, dnb), i = c - j * nb;
      float *yp = Y + c;
      const float *py = vy + i + Ws * j;
#pragma unroll 2
      for (int k = 0; k < nzs; ++k, yp += Ws * nb, py += W2) copy_async(yp, py);
    }
  }
  __syncthreads();  // fs
  // x and y ghosts of the slab's planes
  for (int c = tid; c < 12 * nb; c += bd) {
    const bool yd = c >= 6 * nb;
    const int cc = yd ? c - 6 * nb : c, q = yd ? divq(cc, dnb) : cc / 6, r = cc - q * (yd ? nb : 6);
    const int m = yd ? q : r, o = m < 3 ? m - 3 : nb + m - 3;  // ghost layer
    const int i = yd ? r : o, j = yd ? o : q;
    const FaceSrc &f = fs[2 * yd + (m >= 3)];
    float *tp = T + (j + 3) * RS + i + 4;
    const float *p = face_ptr(f, yd, i, j, k0, nb, Wd);
    const int st = face_step(f, nb, Wd);
    const bool two = f.kind == 2;
    for (int k = 0; k < nzs; ++k, p += st, tp += tst) {
      if (two && k0 + k == nb / 2) p = face_ptr(f, yd, i, j, k0 + k, nb, Wd);  // the next finer leaf
      copy_async(tp, p);
    }
  }
  copy_wait();
  __syncthreads();
  const float invh = 1.0f / sh_h;
  const float lk = LAP ? 0.5f * s.nu * invh : 0.f;  // rhs = -2/h (dF - lk lap)
  // (axes walked for the Laplacian alone add no flux: 0 times an infinity or NaN
  // would reach the whole stencil)
  const bool xon = VEL || LAP || s.ux != 0.f, yon = VEL || LAP || s.uy != 0.f, zon = VEL || LAP || s.uz != 0.f;
  // Pairs of x lines, then of y lines: line q and line q + np, which lie os and
  // ov floats apart in T and in X / Y (y lines: neighbours, np = 1).  A constant
  // velocity u < 0 is walked in the other direction with |u|: the right-biased
  // flux of u phi is minus the left-biased one of |u| phi on the mirrored line,
  // and the order of the difference reverses with it.  So neither sign selects
  // an upwind side.
  const int np = nb * nzs / 2;
  for (int idx = tid; idx < 2 * np; idx += bd) {
    const bool yd = idx >= np;
    if (yd ? !yon : !xon) continue;
    const int q = yd ? 2 * (idx - np) : idx, k = divq(q, dnb), l = q - k * nb;
    const int q2 = yd ? q + 1 : q + np, k2 = divq(q2, dnb), l2 = q2 - k2 * nb;
    const float *p = T + (yd ? (k * Ws + 3) * RS + l + 4 : (k * Ws + l + 3) * RS + 4);
    const int st = yd ? RS : 1, os = yd ? 1 : ((k2 - k) * Ws + l2 - l) * RS, ov = yd ? 1 : np * XS;
    // (the differences of an x row go one float further than its velocities: to
    // even addresses, and never ahead of the velocities still to be read)
    float *v = yd ? Y + (VEL ? (k * Ws + 3) * nb : k * nb2) + l : X + q * XS + (VEL ? 3 : -1);
    const int sv = yd ? nb : 1, oe = yd ? 0 : 1;
    const float uu = VEL ? 0.f : yd ? s.uy : s.ux, hu = 0.5f * fabsf(uu);
    const bool rev = !VEL && uu < 0.f;
    const int dst = rev ? -st : st, dsv = rev ? -sv : sv;
    p += rev ? (nb - 1) * st : 0;
    float *w = v + oe + (rev ? (nb - 1) * sv : 0);
    auto phi = [&](int m) { return make_float2(p[m * dst], p[m * dst + os]); };
    auto hv = [&](int m) {
      return VEL ? pmul(both(hscale), make_float2(v[m * sv], v[m * sv + ov])) : both(hu);
    };
    Walk2<SCHEME, LAP, !VEL> wk;
    wk.start(phi, hv);
#pragma unroll 4
    for (int m = 0; m < nb; ++m) {
      const float2 vn = hv(m + 3), an = phi(m + 3);
      wk.step(s.diff, an, vn, [&](float2 dF, float2, float2 lap) {
        if (LAP) dF = pfma(-lk, lap, VEL || uu != 0.f ? dF : both(0.f));
        w[m * dsv] = dF.x, w[m * dsv + ov] = dF.y;
      });
    }
  }
  // z lines, pairs of neighbours in x.  The three values beyond either end of the
  // slab: the leaf's own planes or the ghosts behind its z faces, loaded for the
  // thread's first pair before the barrier.
  const bool down = !VEL && s.uz < 0.f;  // walk direction
  const int e = down ? nzs - 1 : 0, d = down ? -1 : 1;
  float2 lo[3], hi[3];  // in walk order
  auto ends = [&](int c) {
    const int j = divq(2 * c, dnb), i = 2 * c - j * nb;
    auto line = [&](bool top, float2 *v) {
      const int z = top ? nzs : -3;
      const FaceSrc &f = fs[4 + top];
      const bool own = top ? k0 + nzs < nb : k0 > 0;
      const float *p = own ? src + i + sy * j + z * sz : face_ptr(f, 2, i, j, k0 + z, nb, Wd);
      const int st = own ? sz : face_step(f, nb, Wd);
      // (the two points of a pair lie in the same quadrant of a face: nb / 2 odd
      // is the exception)
      const float *p2 = own || f.kind != 2 ? p + 1 : face_ptr(f, 2, i + 1, j, k0 + z, nb, Wd);
      const float2 v0 = make_float2(__ldg(p), __ldg(p2)), v1 = make_float2(__ldg(p + st), __ldg(p2 + st)),
                   v2 = make_float2(__ldg(p + 2 * st), __ldg(p2 + 2 * st));
      v[0] = down ? v2 : v0, v[1] = v1, v[2] = down ? v0 : v2;
    };
    line(down, lo), line(!down, hi);
  };
  const int nc = nb2 / 2;
  if (tid < nc) ends(tid);
  __syncthreads();
  const float k2 = -2.f * invh;
  const int xst = nb * XS * d, yst = (VEL ? Ws * nb : nb2) * d, pst = d * tst;
  const ptrdiff_t gst = d * nb2;
  auto ld2 = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
  for (int c = tid; c < nc; c += bd) {
    const int j = divq(2 * c, dnb), i = 2 * c - j * nb;
    const float *tp = T + (j + 3) * RS + i + 4 + e * tst;
    const float *xp = X + j * XS + i + (VEL ? 4 : 0) + e * d * xst;
    const float *yp = (VEL ? Y + (j + 3) * nb + i : Y + 2 * c) + e * d * yst;
    const size_t q0 = (size_t)b * nb2 * nb + (k0 + e) * nb2 + 2 * c;
    const float *up = s.u + q0;
    float *op = s.out + q0;
    float2 uo = rk_u ? ld2(up) : both(0.f);  // u^n of the current cell
    auto finish = [&](float2 dF, float2 ph, float2 lap, float2 un) {
      if (LAP && !VEL && s.uz == 0.f) dF = both(0.f);
      const float2 acc = padd(padd(xon ? ld2(xp) : both(0.f), yon ? ld2(yp) : both(0.f)), LAP ? pfma(-lk, lap, dF) : dF);
      float2 r = pmul(acc, both(k2));
      if (!s.rhs_only) r = pfma(s.cv, pfma(s.dt, r, ph), pmul(both(s.cu), un));
      *reinterpret_cast<float2 *>(op) = r;
      xp += xst, yp += yst, op += gst;
    };
    if (zon) {
      const float *vp = vb + 2 * vcomp + Ws * (j + 3) + i + 3;  // plane k0 - 3
      float2 vz[7];
#pragma unroll
      for (int x = 0; x < 7; ++x, vp += W2) vz[x] = VEL ? make_float2(__ldg(vp), __ldg(vp + 1)) : both(0.f);
      const float hu = 0.5f * fabsf(s.uz);
      auto half = [&](float2 v) { return VEL ? pmul(both(hscale), v) : both(hu); };
      Walk2<SCHEME, LAP, !VEL> w;
      w.start([&](int m) { return m < 0 ? lo[m + 3] : ld2(tp + m * pst); }, [&](int m) { return half(vz[m + 3]); });
      float2 vn = vz[6];  // one plane ahead
      tp += 3 * pst;
      auto cell = [&](float2 an, bool more) {
        const float2 v = half(vn), un = uo;
        if (more) {  // the next cell's velocity and u^n
          if (VEL) vn = make_float2(__ldg(vp), __ldg(vp + 1)), vp += W2;
          up += gst;
          if (rk_u) uo = ld2(up);
        }
        w.step(s.diff, an, v, [&](float2 dF, float2 ph, float2 lap) { finish(dF, ph, lap, un); });
      };
      // (unrolled, the kernel falls out of the instruction cache)
#pragma unroll 1
      for (int m = 3; m < nzs; ++m, tp += pst) cell(ld2(tp), true);
      cell(hi[0], true);
      cell(hi[1], true);
      cell(hi[2], false);
    } else {
      for (int m = 0; m < nzs; ++m, tp += pst, up += gst) {
        if (rk_u) uo = ld2(up);
        finish(both(0.f), ld2(tp), both(0.f), uo);
      }
    }
    if (c + bd < nc) ends(c + bd);
  }
}

// ---------------------------------------------------------------------------
// k_march: blockDim = nb*nb threads (12 <= nb, nb*nb <= 576); thread (ti, tj)
// owns the grid column (ti, tj, 0..nb-1).  Shared memory: the six face slabs
// (face f at F + f*3nb^2), then plane buffers laid out like one z-plane of a
// block with a 3-point shell, (y+3)*Ws + x+3 (the layout of a velocity plane):
//   XP[2]  u_x phi / 2 on the x rows of a plane, x ghosts included
//   YP[2]  u_y phi / 2 on the y columns, y ghosts included
//   PH[3]  phi of the plane with its x/y ghosts (diffusion only)
//   UX[2], UY[2]  u_x / 2 on the x rows, u_y / 2 on the y columns (velocity
//          fields: the interface velocity that picks the upwind side)
//   FX[2][nb][nb+1], FY[2][nb+1][nb]  halved x and y interface fluxes.
// The column's phi and u_z at planes k-2..k+3 stay in registers, so the z fluxes need no
// shared memory.  Interval t of the march (one barrier each) evaluates the
// x/y fluxes of plane t, completes plane t-1 (z flux, rhs, RK stage,
// coalesced store) and assembles plane t+1: XP/YP/FX/FY are double-buffered,
// PH triple-buffered (plane t-1 is read while plane t+1 is written).  Every
// flux is computed with the operations of k_fused (the point fluxes u*phi are
// rounded products in both, never contracted; where the compiler fuses another
// multiply-add differently the two may differ in the last bit).
// ---------------------------------------------------------------------------
constexpr int MARCH_MAX_NB = 24;
// faces, XP..FY, PH[3], and (velocity fields) UX[2], UY[2]
__host__ __device__ constexpr int march_smem_floats(int nb, bool vel) {
  return 18 * nb * nb + 4 * nb * (nb + 1) + (vel ? 11 : 7) * (nb + 6) * (nb + 6);
}

template <int SCHEME, bool VEL>
__global__ void __launch_bounds__(576, 2) k_march(Tree t, StageArgs s) {
  constexpr int GS = 3;
  const int b = blockIdx.x, nb = t.nb, Ws = nb + 2 * GS, W2 = Ws * Ws, nb1 = nb + 1, nth = nb * nb;
  const int fs = 3 * nb * nb, Gi = s.Gi, diff = s.diff;
  const float ux = 0.5f * s.ux, uy = 0.5f * s.uy, uz = 0.5f * s.uz, vscale = 0.5f * s.vscale;  // halved point fluxes
  const float *const phi = s.phi;
  const int tid = threadIdx.x, tj = tid / nb, ti = tid - tj * nb;
  const int L = __ldg(t.lev + b);
  const size_t nb3 = (size_t)nb * nb * nb;
  extern __shared__ float sm[];
  float *F = sm;
  float *XP = F + 6 * fs;
  float *YP = XP + 2 * W2;
  float *FX = YP + 2 * W2;
  float *FY = FX + 2 * nb * nb1;
  float *PH = FY + 2 * nb * nb1;
  float *UX = PH + 3 * W2, *UY = UX + 2 * W2;  // velocity fields only
  // prologue: the face slabs
  {
    const int a[3] = {__ldg(t.anc + 3 * b) * nb, __ldg(t.anc + 3 * b + 1) * nb, __ldg(t.anc + 3 * b + 2) * nb};
    __shared__ FaceSrc src[6];
    face_sources(t, b, L, a, phi, s.P, s.Q, Gi, s.lifted, src);
    __syncthreads();
    const int Wd = nb + 2 * Gi;
    for (int f = 0; f < 6; ++f)
      for (int p = tid; p < fs; p += nth) {
        // F index: the face's axis runs over 3 layers, the others over nb
        const int n0 = f < 2 ? 3 : nb, n1 = f == 2 || f == 3 ? 3 : nb, r = p / n0, c2 = r / n1;
        int c[3] = {p - r * n0, r - c2 * n1, c2};
        c[f >> 1] += (f & 1) ? nb : -GS;
        F[f * fs + p] = __ldg(face_ptr(src[f], f >> 1, c[0], c[1], c[2], nb, Wd));
      }
  }
  // the column: interior from the field, or from the substituted padded block
  // that k_prep wrote for leaves next to a coarser leaf
  const float *col;
  int cst;
  if (s.cmask[b]) {
    const int Wd = nb + 2 * Gi;
    col = s.P + (size_t)b * Wd * Wd * Wd + (ti + Gi) + (size_t)Wd * ((tj + Gi) + (size_t)Wd * Gi);
    cst = Wd * Wd;
  } else {
    col = phi + (size_t)b * nb3 + ti + nb * tj;
    cst = nb * nb;
  }
  // velocity components: ghost-filled blocks with shell GS; the plane-buffer
  // offset o of a point of plane z is o + W2*(z+GS) in them
  const size_t vblk = (size_t)Ws * W2;
  const float *vbx = VEL ? s.vpad + (size_t)b * vblk : nullptr;
  const float *vby = VEL ? vbx + (size_t)t.nleaf * vblk : nullptr;
  const float *vbz = VEL ? vby + (size_t)t.nleaf * vblk : nullptr;
  const int cidx = (tj + GS) * Ws + ti + GS;  // the column's plane offset
  // a velocity component at plane offset o of plane z
  auto vat = [&](const float *vb, int o, int z) -> float { return vscale * __ldg(vb + o + W2 * (z + GS)); };
  const bool xon = VEL || ux != 0.f, yon = VEL || uy != 0.f, zon = VEL || uz != 0.f;
  // ghost columns/rows of a plane: thread tid < 12 nb fetches one of them
  // (face index hsrc at plane 0, plane offset hdst; hy: a y ghost)
  int hsrc = -1, hdst = 0, hy = 0;
  if (tid < 6 * nb) {
    const int j = tid / 6, m = tid - 6 * j, x = m < 3 ? m - GS : nb + m - GS;
    hsrc = (m < 3 ? 0 : fs) + (m < 3 ? m : m - 3) + 3 * j;
    hdst = (j + GS) * Ws + x + GS;
  } else if (tid < 12 * nb) {
    const int h = tid - 6 * nb, m = h / nb, i = h - m * nb, y = m < 3 ? m - GS : nb + m - GS;
    hsrc = (m < 3 ? 2 * fs : 3 * fs) + i + nb * (m < 3 ? m : m - 3);
    hdst = (y + GS) * Ws + i + GS;
    hy = 1;
  }
  // x interfaces of a plane: flattened index tid, and tid + nth for tid < nb;
  // interface i of row r is F_{i-1/2}, stored at FX[r*(nb+1) + i] = FX[index]
  int xo0, xo1;
  {
    const int r0 = tid / nb1, r1 = (tid + nth) / nb1;
    xo0 = (r0 + GS) * Ws + tid - r0 * nb1;  // plane offset of x = i-3 on row r
    xo1 = (r1 + GS) * Ws + tid + nth - r1 * nb1;
  }
  auto xflux = [&](int buf, int z, int o, int fi) {
    const float *p = XP + buf * W2 + o;
    const float f6[6] = {p[0], p[1], p[2], p[3], p[4], p[5]};
    const float *v = UX + buf * W2 + o;
    const bool left = VEL ? (v[2] + v[3] >= 0.f) : ux >= 0.f;
    FX[buf * nb * nb1 + fi] = half_flux6<float, SCHEME>(f6, left);
  };
  // y interfaces: F_{r-1/2} of column ti for r = tj, and r = nb for the last
  // row of threads, stored at FY[r*nb + ti]
  auto yflux = [&](int buf, int z, int r) {
    const int o = r * Ws + ti + GS;  // plane offset of y = r-3
    const float *p = YP + buf * W2 + o;
    const float f6[6] = {p[0], p[Ws], p[2 * Ws], p[3 * Ws], p[4 * Ws], p[5 * Ws]};
    const float *v = UY + buf * W2 + o;
    const bool left = VEL ? (v[2 * Ws] + v[3 * Ws] >= 0.f) : uy >= 0.f;
    FY[buf * nb1 * nb + r * nb + ti] = half_flux6<float, SCHEME>(f6, left);
  };
  // plane z into the buffers (z & 1) and z % 3; ph = phi at (ti, tj, z)
  auto assemble = [&](int z, float ph, float vxv, float vyv) {
    const int xb = (z & 1) * W2;
    XP[xb + cidx] = __fmul_rn(vxv, ph);
    YP[xb + cidx] = __fmul_rn(vyv, ph);
    if (VEL) UX[xb + cidx] = vxv, UY[xb + cidx] = vyv;
    if (diff) PH[(z % 3) * W2 + cidx] = ph;
    if (hsrc >= 0) {
      const float fv = F[hsrc + 3 * nb * z];
      const float hu = VEL ? vat(hy ? vby : vbx, hdst, z) : (hy ? uy : ux);
      (hy ? YP : XP)[xb + hdst] = __fmul_rn(hu, fv);
      if (VEL) (hy ? UY : UX)[xb + hdst] = hu;
      if (diff) PH[(z % 3) * W2 + hdst] = fv;
    }
  };
  __syncthreads();
  auto phi_at = [&](int m) -> float {
    if (m < 0) return F[4 * fs + ti + nb * (tj + nb * (m + GS))];
    if (m >= nb) return F[5 * fs + ti + nb * (tj + nb * (m - nb))];
    return __ldg(col + (size_t)m * cst);
  };
  auto velz = [&](int z) -> float { return VEL ? vat(vbz, cidx, z) : uz; };
  // register windows: phi and u_z at planes k-2..k+3 (k: the plane the next
  // completion finishes); F_{k-1/2} along z
  float pw[6], uw[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    pw[m] = phi_at(m - 2);
    uw[m] = velz(m - 2);
  }
  float Fzm = 0.f;
  if (zon) {
    const float u3 = velz(-3);
    const float f6[6] = {__fmul_rn(u3, phi_at(-3)), __fmul_rn(uw[0], pw[0]), __fmul_rn(uw[1], pw[1]),
                         __fmul_rn(uw[2], pw[2]),     __fmul_rn(uw[3], pw[3]), __fmul_rn(uw[4], pw[4])};
    Fzm = half_flux6<float, SCHEME>(f6, VEL ? (uw[1] + uw[2] >= 0.f) : uz >= 0.f);
  }
  assemble(0, pw[2], VEL ? vat(vbx, cidx, 0) : ux, VEL ? vat(vby, cidx, 0) : uy);
  __syncthreads();
  const float h = (float)(t.tree_len / ((double)nb * (double)(1 << L)));
  const float invh = 1.0f / h;
  const bool rk_u = !s.rhs_only && s.stage > 0;
  for (int tt = 0; tt <= nb; ++tt) {
    // loads of this interval: the column's next window entries, the velocity
    // of plane tt+1 and u^n of plane tt-1
    const bool shift = tt >= 1 && tt < nb, asmb = tt + 1 < nb;
    float pn = 0.f, uzn = 0.f, vxn = ux, vyn = uy, uo = 0.f;
    if (shift) {
      pn = phi_at(tt + 3);
      uzn = velz(tt + 3);
    }
    if (VEL && asmb) {
      vxn = vat(vbx, cidx, tt + 1);
      vyn = vat(vby, cidx, tt + 1);
    }
    const size_t q = (size_t)b * nb3 + ti + nb * (tj + (size_t)nb * (tt - 1));
    if (tt >= 1 && rk_u) uo = s.u[q];
    // fluxes of plane tt
    if (tt < nb) {
      const int buf = tt & 1;
      if (xon) {
        xflux(buf, tt, xo0, tid);
        if (tid < nb) xflux(buf, tt, xo1, tid + nth);
      }
      if (yon) {
        yflux(buf, tt, tj);
        if (tj == nb - 1) yflux(buf, tt, nb);
      }
    }
    // completion of plane k = tt-1
    if (tt >= 1) {
      const int k = tt - 1, fb = k & 1;
      float acc = 0.f;
      if (xon) acc = FX[fb * nb * nb1 + tj * nb1 + ti + 1] - FX[fb * nb * nb1 + tj * nb1 + ti];
      if (yon) acc += FY[fb * nb1 * nb + (tj + 1) * nb + ti] - FY[fb * nb1 * nb + tj * nb + ti];
      if (zon) {
        const float f6[6] = {__fmul_rn(uw[0], pw[0]), __fmul_rn(uw[1], pw[1]), __fmul_rn(uw[2], pw[2]),
                             __fmul_rn(uw[3], pw[3]), __fmul_rn(uw[4], pw[4]), __fmul_rn(uw[5], pw[5])};
        const float Fzp = half_flux6<float, SCHEME>(f6, VEL ? (uw[2] + uw[3] >= 0.f) : uz >= 0.f);
        acc += Fzp - Fzm;
        Fzm = Fzp;
      }
      float r = -2.f * (acc * invh);
      if (diff) {
        const float *pc = PH + (k % 3) * W2 + cidx;
        float lp = 0.f;
        lp += lap_term<float>(pc[-2], pc[-1], pc[0], pc[1], pc[2], diff);
        lp += lap_term<float>(pc[-2 * Ws], pc[-Ws], pc[0], pc[Ws], pc[2 * Ws], diff);
        lp += lap_term<float>(pw[0], pw[1], pw[2], pw[3], pw[4], diff);
        r += s.nu * invh * invh * lp;
      }
      s.out[q] = stage_value(s, pw[2], r, uo);
      if (shift) {
#pragma unroll
        for (int m = 0; m < 5; ++m) pw[m] = pw[m + 1], uw[m] = uw[m + 1];
        pw[5] = pn;
        uw[5] = uzn;
      }
    }
    // plane tt+1 (the window now holds planes tt-2..tt+3)
    if (asmb) assemble(tt + 1, pw[3], vxn, vyn);
    __syncthreads();
  }
}

// Host side: the variant (mr_set_stage_kernel: 0 tuned, 1 k_fused, 2
// k_march) and, for k_fused, the slab height, tuned on launches that do not
// overwrite their input (the bare right-hand side, stage 0).
int launch_fused(mr_grid *g, const void *phi, const void *P, const void *Q, int Gi, const void *u, void *out,
                 int stage, double dt, const double *uc, int scheme, bool rhs_only, const void *vpad) {
  static const double zero3[3] = {0.0, 0.0, 0.0};
  if (!uc) uc = zero3;
  Tree t = tree_view(g);
  const bool vel = vpad != nullptr;
  const int nb = g->desc.nb, N = g->desc.wav_N, NT = g->desc.wav_Nt;
  StageArgs s{(const float *)phi, (const float *)P, (const float *)Q, Gi, NT != 0, g->cmask, (const float *)u,
              (float *)out, stage, rhs_only ? 1 : 0, (float)dt, (float)uc[0], (float)uc[1], (float)uc[2],
              (const float *)vpad, (float)g->diff_nu, (float)g->vel_scale, g->diff_order, divm(nb + 6),
              stage == 0 ? 0.f : stage == 1 ? 0.75f : 1.0f / 3, stage == 0 ? 1.f : stage == 1 ? 0.25f : 2.0f / 3};
  const bool march_ok = nb >= 12 && nb <= MARCH_MAX_NB;
  const size_t smm = sizeof(float) * (size_t)march_smem_floats(nb, vel);
  // slab heights: fused_height, or four planes
  // (four instead of eight at 16^3: 613 against 500 us for 11 019 leaves; instead
  // of six at 24^3: 4.88 against 4.44 ms for 42 400)
  const int hq = fused_height(nb), ht = 4;
  auto threads_of = [&](int nz) { return std::min(160, (nb * nz + 31) / 32 * 32); };
  const int cand[2] = {threads_of(hq), threads_of(ht)};
  const int ncand = cand[0] != cand[1] ? 2 : 1;
  const int vcand[2] = {1, 2};
  const bool can_tune = rhs_only || stage == 0;
  auto run = [&](auto kf, auto km) -> int {
    if (nb > FUSED_MAX_NB) {
      set_error("FP32 stage: blocks of more than 26 points per edge");
      return MR_ERR_CUDA;
    }
    if (smem_limit(kf, sizeof(float) * fused_smem_floats(FUSED_MAX_NB, fused_height(FUSED_MAX_NB), vel), "fused smem"))
      return MR_ERR_CUDA;
    if (march_ok && smem_limit(km, sizeof(float) * march_smem_floats(MARCH_MAX_NB, vel), "march smem"))
      return MR_ERR_CUDA;
    const int mode = 2 * scheme + (vel ? 1 : 0) + (g->diff_order ? 8 : 0);
    auto fused = [&](int th) {
      const int ns = (nb + (th == cand[0] ? hq : ht) - 1) / (th == cand[0] ? hq : ht), nz = (nb + ns - 1) / ns;
      kf<<<g->nleaf * ns, th, sizeof(float) * fused_smem_floats(nb, nz, vel), g->stream>>>(t, s, nz, ns);
    };
    auto march = [&]() { km<<<g->nleaf, nb * nb, smm, g->stream>>>(t, s); };
    const int threads = tune_threads(g, TuneKey{3, N, NT, nb, 4, Gi, mode}, cand, can_tune ? ncand : 1, fused);
    int variant = march_ok ? g->stage_kernel : 1;
    if (variant == 0)
      variant = tune_threads(g, TuneKey{6, N, NT, nb, 4, Gi, mode}, vcand, can_tune ? 2 : 1,
                             [&](int v) { v == 2 ? march() : fused(threads); });
    if (variant == 2) MR_LAUNCH(g, MRK_RHS, march());
    else MR_LAUNCH(g, MRK_RHS, fused(threads));
    return check_cuda(cudaGetLastError(), variant == 2 ? "k_march" : "k_fused") ? MR_ERR_CUDA : MR_OK;
  };
#define MR_FV(S)                                                                                         \
  do {                                                                                                   \
    if (g->diff_order)                                                                                   \
      return vel ? run(k_fused<S, true, true>, k_march<S, true>) : run(k_fused<S, false, true>, k_march<S, false>); \
    return vel ? run(k_fused<S, true, false>, k_march<S, true>) : run(k_fused<S, false, false>, k_march<S, false>); \
  } while (0)
  if (scheme == MR_CONS3) MR_FV(MR_CONS3);
  if (scheme == MR_CONS5) MR_FV(MR_CONS5);
  if (scheme == MR_WENOZ5) MR_FV(MR_WENOZ5);
#undef MR_FV
  return MR_ERR_INVALID;
}

}  // namespace mr
