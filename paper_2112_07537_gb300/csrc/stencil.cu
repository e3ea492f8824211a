// stencil.cu -- advection right-hand side fused with the RK3-TVD stage,
// analytic field initialisation and the FP64 mass reduction.
#include <cmath>

#include "stage_kernels.cuh"

namespace mr {

// Right-hand side from the padded block P (shell Gi >= 3), then the RK stage
// combination (or the bare rhs).  u: u^n (stages 1, 2), may alias out.
// One CTA per slab of nz z-planes of a leaf.  The x and y grid lines of the
// slab, cut into segments of seg cells, are walked first (walk_line: every
// interface flux once, differences shared along the line), their flux
// differences left in shared memory; the z lines of the slab then add theirs
// and finish their cells.  FP64 is bound by the FP64 pipe: about 45 of its
// instructions per interface, so the walk (each flux once, one division
// instead of four) is what counts; slabs and segments only spread small grids
// over the chip (see rhs_dispatch) and change no value: point fluxes are
// rounded products and the sums of walk_line leave nothing to contract, so a
// flux does not depend on where its line was cut.  Measured (WENO-Z5, velocity
// fields, 1 408 leaves of 24^3 = 19.5 M points): 23.9 ms per launch with both
// fluxes of every point evaluated per thread and four divisions each, 5.88 ms
// so (the FP64 pipe's floor for 147 instructions a point is 4.6 ms; flat parts of
// a field skip some, see weno_corr); 15 leaves of 16^3: 680 us in 15 CTAs, 38 us.
template <typename T, int SCHEME>
__global__ void __launch_bounds__(256) k_rhs_stage(Tree t, const T *__restrict__ P, int Gi, const T *u, T *out,
                                                   int stage, T dt, T ux, T uy, T uz, int rhs_only,
                                                   const T *__restrict__ vpad, T nu, int diff, T vscale, int nz,
                                                   int nslab, int seg) {
  // vpad: ghost-filled velocity components (shell 3) or null for constant u
  const int b = blockIdx.x / nslab, k0 = (blockIdx.x - b * nslab) * nz;
  const int nb = t.nb, Wd = nb + 2 * Gi, Wv = nb + 6, nzs = min(nz, nb - k0), RS = nb + 1;
  const size_t np = (size_t)Wd * Wd * Wd, vblk = (size_t)Wv * Wv * Wv, vcomp = (size_t)t.nleaf * vblk;
  const T *Pb = P + (size_t)b * np + Gi + Wd * (Gi + (size_t)Wd * (Gi + k0));  // cell (0, 0, k0)
  const T *Vb = vpad ? vpad + (size_t)b * vblk + 3 + Wv * (3 + (size_t)Wv * (3 + k0)) : nullptr;
  const T hscale = T(0.5) * vscale;
  extern __shared__ double smd[];
  T *R0 = reinterpret_cast<T *>(smd), *R1 = R0 + (size_t)nz * nb * RS;  // x and y flux differences
  auto walk = [&](int d, const T *p, const T *v, int st, int sv, int n, auto emit) {
    if (vpad) {
      v += d * vcomp;
      walk_line<T, SCHEME>(
          n, [&](int m) { return p[m * st]; }, [&](int m) { return rmul(hscale, v[m * sv]); }, emit);
    } else {
      const T hu = T(0.5) * (d == 0 ? ux : d == 1 ? uy : uz);
      walk_line<T, SCHEME>(n, [&](int m) { return p[m * st]; }, [&](int) { return hu; }, emit);
    }
  };
  const bool xon = vpad || ux != T(0), yon = vpad || uy != T(0), zon = vpad || uz != T(0);
  // x segments, then y segments: nseg per line, lines (other axis, plane)
  const int nseg = (nb + seg - 1) / seg, nx = nb * nzs * nseg;
  for (int idx = threadIdx.x; idx < 2 * nx; idx += blockDim.x) {
    const bool yd = idx >= nx;
    const int q = yd ? idx - nx : idx, l = q % nb, r = q / nb, s = r % nseg, k = r / nseg;
    const int m0 = s * seg, n = min(seg, nb - m0);
    if (yd ? !yon : !xon) continue;
    const int i = yd ? l : m0, j = yd ? m0 : l;
    const size_t o = i + Wd * (j + (size_t)Wd * k), ov = i + Wv * (j + (size_t)Wv * k);
    T *rr = (yd ? R1 : R0) + i + RS * (j + nb * k);
    const int rs = yd ? RS : 1;
    walk(yd ? 1 : 0, Pb + o, Vb + (vpad ? ov : 0), yd ? Wd : 1, yd ? Wv : 1, n,
         [&](int m, T dF, T) { rr[m * rs] = dF; });
  }
  __syncthreads();
  const T h = T(t.tree_len / ((double)nb * (double)(1 << __ldg(t.lev + b)))), inv2 = T(2) / h, invh2 = T(1) / (h * h);
  const int stride[3] = {1, Wd, Wd * Wd};
  for (int c = threadIdx.x; c < nb * nb; c += blockDim.x) {
    const int j = c / nb, i = c - j * nb;
    const T *p = Pb + i + Wd * j;
    const size_t q0 = (size_t)b * nb * nb * nb + c + (size_t)nb * nb * k0;
    auto finish = [&](int m, T dz, T ph) {
      const int ro = i + RS * (j + nb * m);
      T acc = T(0);
      if (xon) acc = R0[ro];
      if (yon) acc += R1[ro];
      if (zon) acc += dz;
      T r = -acc * inv2;
      const T *pc = p + (size_t)m * Wd * Wd;
      if (diff) r += nu * lap_at<T>(pc, stride, diff) * invh2;
      const size_t q = q0 + (size_t)m * nb * nb;
      if (rhs_only) {
        out[q] = r;
      } else {
        const T v = ph + dt * r;
        T o;
        if (stage == 0) o = v;
        else if (stage == 1) o = T(0.75) * u[q] + T(0.25) * v;
        else o = T(1.0 / 3) * u[q] + T(2.0 / 3) * v;
        out[q] = o;
      }
    };
    if (zon)
      walk(2, p, Vb + (vpad ? i + Wv * j : 0), Wd * Wd, Wv * Wv, nzs, finish);
    else
      for (int m = 0; m < nzs; ++m) finish(m, T(0), p[(size_t)m * Wd * Wd]);
  }
}

template <typename T>
static int rhs_dispatch(mr_grid *g, const T *P, int Gi, const T *u, T *out, int stage, double dt,
                        const double *uc, int scheme, bool rhs_only, const T *vpad) {
  Tree t = tree_view(g);
  const int n = g->nleaf;
  static const double zero3[3] = {0.0, 0.0, 0.0};
  if (!uc) uc = zero3;
  const T ux = T(uc[0]), uy = T(uc[1]), uz = T(uc[2]);
  // Slabs of 8 planes (a z line of 8 cells evaluates 9 fluxes; its sums take
  // 77 KB of shared memory at nb = 24 in FP64, two CTAs per SM).  Grids too
  // small to give every SM two such slabs get thinner ones, down to 2 planes,
  // and x/y lines cut until the CTA's threads all have a segment.
  const int nb = g->desc.nb;
  int nslab = (nb + 7) / 8;
  while (nslab * 2 <= nb / 2 && (long)n * nslab < 2 * 152) nslab *= 2;
  const int nz = (nb + nslab - 1) / nslab;
  nslab = (nb + nz - 1) / nz;
  int seg = nb;
  if ((long)n * nslab < 4 * 152)
    while (seg > 4 && 2 * nb * nz * ((nb + seg - 1) / seg) < 256) seg = (seg + 1) / 2;
  const size_t sm = 2 * sizeof(T) * (size_t)nz * nb * (nb + 1);
  auto go = [&](auto kern) -> int {
    if (smem_limit(kern, 2 * sizeof(T) * 8 * MAX_NB * (MAX_NB + 1), "rhs smem")) return MR_ERR_CUDA;
    MR_LAUNCH(g, MRK_RHS, kern<<<n * nslab, 256, sm, g->stream>>>(t, P, Gi, u, out, stage, T(dt), ux, uy, uz, rhs_only,
                                                                  vpad, T(g->diff_nu), g->diff_order, T(g->vel_scale),
                                                                  nz, nslab, seg));
    return check_cuda(cudaGetLastError(), "k_rhs_stage") ? MR_ERR_CUDA : MR_OK;
  };
  if (scheme == MR_CONS3) return go(k_rhs_stage<T, MR_CONS3>);
  if (scheme == MR_CONS5) return go(k_rhs_stage<T, MR_CONS5>);
  if (scheme == MR_WENOZ5) return go(k_rhs_stage<T, MR_WENOZ5>);
  return MR_ERR_INVALID;
}

int launch_rhs_stage(mr_grid *g, const void *P, int Gi, const void *u, void *out, int stage,
                     double dt, const double *uc, int scheme, bool rhs_only, const void *vpad) {
  if (Gi < 3) return MR_ERR_INVALID;
  if (g->desc.precision == MR_F32)
    return rhs_dispatch<float>(g, (const float *)P, Gi, (const float *)u, (float *)out, stage, dt, uc,
                               scheme, rhs_only, (const float *)vpad);
  return rhs_dispatch<double>(g, (const double *)P, Gi, (const double *)u, (double *)out, stage, dt,
                              uc, scheme, rhs_only, (const double *)vpad);
}

template <typename T>
__global__ void k_rk_combine(size_t n, int stage, T dt, const T *u, const T *y, const T *r, T *out) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
    const T v = y[q] + dt * r[q];
    T o;
    if (stage == 0) o = v;
    else if (stage == 1) o = T(0.75) * u[q] + T(0.25) * v;
    else o = T(1.0 / 3) * u[q] + T(2.0 / 3) * v;
    out[q] = o;
  }
}


int launch_rk_combine(mr_grid *g, int stage, double dt, const void *u, const void *y, const void *r,
                      void *out) {
  const size_t n = (size_t)g->nleaf * g->nb3;
  const int blocks = 152 * 8;
  if (g->desc.precision == MR_F32)
    MR_LAUNCH(g, MRK_COMBINE, k_rk_combine<float><<<blocks, 256, 0, g->stream>>>(n, stage, (float)dt, (const float *)u,
                                                        (const float *)y, (const float *)r, (float *)out));
  else
    MR_LAUNCH(g, MRK_COMBINE, k_rk_combine<double><<<blocks, 256, 0, g->stream>>>(n, stage, dt, (const double *)u,
                                                         (const double *)y, (const double *)r,
                                                         (double *)out));
  return check_cuda(cudaGetLastError(), "k_rk_combine") ? MR_ERR_CUDA : MR_OK;
}

// ---------------------------------------------------------------- analytic
struct InitParams {
  double p[256];
};

__device__ __forceinline__ double pdelta(double x, double c, double ext) {
  double d = x - c;
  return d - ext * rint(d / ext);
}

template <typename T>
__global__ void k_field_set(Tree t, T *f, int kind, InitParams ip) {
  const int b = blockIdx.x, nb = t.nb;
  const int L = __ldg(t.lev + b);
  const double h = t.tree_len / ((double)nb * (double)(1 << L));
  // independent trees: every tree holds the field in its own coordinates
  const double ext[3] = {(t.indep ? 1 : t.nt[0]) * t.tree_len, (t.indep ? 1 : t.nt[1]) * t.tree_len,
                         (t.indep ? 1 : t.nt[2]) * t.tree_len};
  int a[3];
  for (int d = 0; d < 3; ++d) {
    a[d] = __ldg(t.anc + 3 * b + d);
    if (t.indep) a[d] &= (1 << L) - 1;  // anchor within the leaf's tree
  }
  // kinds that depend on the distance from one centre: the squared distance
  // along each axis, once per block (a point adds three of them; the divisions
  // and roundings of the nearest image took 40 % of the FP64 instructions)
  const bool radial = kind == MR_INIT_GAUSSIAN || kind == MR_INIT_TANH_SPHERE || kind == MR_INIT_COMPACT_GAUSSIAN;
  __shared__ double sq[3][32];
  if (radial) {
    for (int q = threadIdx.x; q < 3 * nb; q += blockDim.x) {
      const int d = q / nb, i = q - d * nb;
      const double dd = pdelta((a[d] * nb + i) * h, ip.p[d], ext[d]);
      sq[d][i] = dd * dd;
    }
    __syncthreads();
  }
  // the sphere's width divides every point: by its reciprocal, once per thread,
  // and one step on the residual (the quotient to rounding), three instructions
  // for about ten (92.8 M points 7.64 -> 6.81 ms); widths and distances near the
  // ends of the exponent range divide
  const double wi = kind == MR_INIT_TANH_SPHERE ? 1.0 / ip.p[4] : 0.0;
  const bool wok = fabs(ip.p[4]) > 1e-150 && fabs(ip.p[4]) < 1e150;
  for (int p = threadIdx.x; p < nb * nb * nb; p += blockDim.x) {
    const int rr = divq(p, t.dnb), k = divq(rr, t.dnb), i = p - rr * nb, j = rr - k * nb;
    const double r2 = radial ? sq[0][i] + sq[1][j] + sq[2][k] : 0.0;
    double x[3] = {0.0, 0.0, 0.0};
    if (!radial) x[0] = (a[0] * nb + i) * h, x[1] = (a[1] * nb + j) * h, x[2] = (a[2] * nb + k) * h;
    double v = 0.0;
    if (kind == MR_INIT_GAUSSIAN) {
      v = ip.p[4] * exp(-r2 / (ip.p[3] * ip.p[3]));
    } else if (kind == MR_INIT_TANH_SPHERE) {
      // (1 - tanh y) / 2 = 1 / (1 + exp 2y): one exponential and one division,
      // and no cancellation where tanh y nears 1; 0 and 1 from |y| = 19.07 on,
      // where tanh y rounds to +-1 (the FP64 pipe bounds this kernel)
      const double u = sqrt(r2) - ip.p[3];
      double y = u * wi;
      const bool fin = (__double2hiint(u) & 0x7fffffff) < 0x5f000000;  // below 1e150
      y = wok && fin ? fma(fma(-y, ip.p[4], u), wi, y) : u / ip.p[4];
      v = y > 19.07 ? 0.0 : y < -19.07 ? 1.0 : 1.0 / (1.0 + exp(2.0 * y));
    } else if (kind == MR_INIT_GAUSSIAN_SUM || kind == MR_INIT_GAUSSIAN_SUM_ADD) {
      const int ng = (int)ip.p[0];
      for (int q = 0; q < ng; ++q) {
        const double *c = ip.p + 1 + 5 * q;
        double r2 = 0.0;
        for (int d = 0; d < 3; ++d) {
          const double dd = pdelta(x[d], c[d], ext[d]);
          r2 += dd * dd;
        }
        v += c[4] * exp(-r2 / (c[3] * c[3]));
      }
    } else if (kind == MR_INIT_COMPACT_GAUSSIAN) {
      const double s2 = ip.p[3] * ip.p[3], b2 = ip.p[4] * ip.p[4];
      v = r2 < b2 ? ip.p[5] * exp(-(r2 / s2) / (1.0 - r2 / b2)) : 0.0;
    } else if (kind == MR_INIT_DEFORMATION) {
      const double pi = M_PI, s = ip.p[1];
      const int comp = (int)ip.p[0];
      const double sx = sin(pi * x[0]), sy = sin(pi * x[1]), sz = sin(pi * x[2]);
      const double s2x = sin(2 * pi * x[0]), s2y = sin(2 * pi * x[1]), s2z = sin(2 * pi * x[2]);
      if (comp == 0) v = 2.0 * s * sx * sx * s2y * s2z;
      else if (comp == 1) v = -s * s2x * sy * sy * s2z;
      else v = -s * s2x * s2y * sz * sz;
    } else if (kind == MR_INIT_TAYLOR_GREEN) {
      const double w = 2.0 * M_PI, s = ip.p[1], ph = ip.p[2];
      const int comp = (int)ip.p[0];
      if (comp == 0) v = s * sin(w * x[0] + ph) * cos(w * x[1]) * cos(w * x[2]);
      else if (comp == 1) v = -s * cos(w * x[0] + ph) * sin(w * x[1]) * cos(w * x[2]);
      else v = 0.0;
    }
    const size_t q = (size_t)b * nb * nb * nb + p;
    if (kind == MR_INIT_GAUSSIAN_SUM_ADD) v += (double)f[q];  // the field value, then the sum
    f[q] = T(v);
  }
}

int launch_field_set(mr_grid *g, void *f, int kind, const double *p, int np) {
  InitParams ip{};
  for (int i = 0; i < np && i < 256; ++i) ip.p[i] = p[i];
  Tree t = tree_view(g);
  if (g->desc.precision == MR_F32)
    MR_LAUNCH(g, MRK_FIELDSET, k_field_set<float><<<g->nleaf, 256, 0, g->stream>>>(t, (float *)f, kind, ip));
  else
    MR_LAUNCH(g, MRK_FIELDSET, k_field_set<double><<<g->nleaf, 256, 0, g->stream>>>(t, (double *)f, kind, ip));
  return check_cuda(cudaGetLastError(), "k_field_set") ? MR_ERR_CUDA : MR_OK;
}

// FP64 mass: per-leaf sums (fixed order within a CTA), then one CTA sums the
// per-leaf partials in slot order: deterministic for a given leaf count.
template <typename T>
__global__ void k_mass_leaf(Tree t, const T *f, double *part) {
  const int b = blockIdx.x, nb = t.nb;
  const double h = t.tree_len / ((double)nb * (double)(1 << __ldg(t.lev + b)));
  // one FP64 addition per value (the pipe's floor); the widening runs on the
  // integer pipe, two sums per thread hide the addition's latency
  const T *fb = f + (size_t)b * nb * nb * nb;
  const int n = nb * nb * nb, bd = blockDim.x;
  double s0 = 0.0, s1 = 0.0;
  int p = threadIdx.x;
#pragma unroll 4
  for (; p + bd < n; p += 2 * bd) s0 += Cvt<double>::f(__ldg(fb + p)), s1 += Cvt<double>::f(__ldg(fb + p + bd));
  if (p < n) s0 += Cvt<double>::f(__ldg(fb + p));
  double s = s0 + s1;
  for (int w = 16; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
  __shared__ double red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (bd >> 5); ++w) s += red[w];
    part[b] = s * h * h * h;
  }
}

__global__ void __launch_bounds__(1024) k_sum_serial(const double *part, int n, double *out) {
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  for (int w = 16; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    *out = s;
  }
}

int launch_mass(mr_grid *g, const void *f, double *host_out) {
  Tree t = tree_view(g);
  if (g->desc.precision == MR_F32)
    MR_LAUNCH(g, MRK_MASS, k_mass_leaf<float><<<g->nleaf, 256, 0, g->stream>>>(t, (const float *)f, g->maxdet));
  else
    MR_LAUNCH(g, MRK_MASS, k_mass_leaf<double><<<g->nleaf, 256, 0, g->stream>>>(t, (const double *)f, g->maxdet));
  MR_LAUNCH(g, MRK_MASS, k_sum_serial<<<1, 1024, 0, g->stream>>>(g->maxdet, g->nleaf, g->dscratch));
  if (check_cuda(cudaGetLastError(), "k_mass")) return MR_ERR_CUDA;
  if (check_cuda(cudaMemcpyAsync(host_out, g->dscratch, sizeof(double), cudaMemcpyDeviceToHost, g->stream),
                 "mass copy"))
    return MR_ERR_CUDA;
  return check_cuda(cudaStreamSynchronize(g->stream), "mass sync") ? MR_ERR_CUDA : MR_OK;
}

// Time step (reading of Sec. 5.1): dt = CFL h_min / max_x sum_d |u_d|.  Per
// leaf: max over its points of |u_0| + |u_1| + |u_2| (FP64 sums of the stored
// values, x, then y, then z) and its level; one CTA then takes the maxima --
// max is exact, so the result does not depend on the order.
template <typename T>
__global__ void __launch_bounds__(256) k_umax_leaf(int nb, const T *__restrict__ u0, const T *__restrict__ u1,
                                                   const T *__restrict__ u2, double *part) {
  const int b = blockIdx.x;
  const size_t nb3 = (size_t)nb * nb * nb, o = (size_t)b * nb3;
  unsigned long long m = 0;
  auto exact = [&](size_t p) {
    const double s = fabs((double)u0[o + p]) + fabs((double)u1[o + p]) + fabs((double)u2[o + p]);
    m = max(m, abs_key(s));
  };
  if constexpr (sizeof(T) == 4) {
    // FP32 sums rounded down and up enclose the FP64 sum (rounding is monotone
    // and every FP32 number is an FP64 one), so only points whose upper bound
    // reaches the block's largest lower bound need it: the two FP64 additions
    // and three conversions of every point were what bound this kernel.
    float lo = 0.f;
#pragma unroll 4
    for (size_t p = threadIdx.x; p < nb3; p += blockDim.x)
      lo = fmaxf(lo, __fadd_rd(__fadd_rd(fabsf(u0[o + p]), fabsf(u1[o + p])), fabsf(u2[o + p])));
    __shared__ unsigned best;
    if (threadIdx.x == 0) best = 0;
    __syncthreads();
    for (int w = 16; w > 0; w >>= 1) lo = fmaxf(lo, __shfl_xor_sync(0xffffffffu, lo, w));
    if ((threadIdx.x & 31) == 0) atomicMax(&best, __float_as_uint(lo));  // lo >= 0: ordered as integers
    __syncthreads();
    const float top = __uint_as_float(best);
#pragma unroll 4
    for (size_t p = threadIdx.x; p < nb3; p += blockDim.x) {
      const float hi = __fadd_ru(__fadd_ru(fabsf(u0[o + p]), fabsf(u1[o + p])), fabsf(u2[o + p]));
      if (!(hi < top)) exact(p);  // (NaN included)
    }
  } else {
    for (size_t p = threadIdx.x; p < nb3; p += blockDim.x) exact(p);
  }
  for (int w = 16; w > 0; w >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, w));
  __shared__ unsigned long long red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
    part[b] = __longlong_as_double((long long)max(m, red[0]));
  }
}

__global__ void __launch_bounds__(256) k_dt_reduce(const double *__restrict__ part, const int *__restrict__ lev, int n,
                                                   double usum_const, double cfl, double tree_len, int nb,
                                                   double *out) {
  unsigned long long m = 0;
  int lm = 0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) {
    if (part) m = max(m, abs_key(part[b]));
    lm = max(lm, lev[b]);
  }
  for (int w = 16; w > 0; w >>= 1) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, w));
    lm = max(lm, __shfl_xor_sync(0xffffffffu, lm, w));
  }
  __shared__ unsigned long long rm[8];
  __shared__ int rl[8];
  if ((threadIdx.x & 31) == 0) rm[threadIdx.x >> 5] = m, rl[threadIdx.x >> 5] = lm;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, rm[w]), lm = max(lm, rl[w]);
    const double us = part ? __longlong_as_double((long long)m) : usum_const;
    const double h = tree_len / ((double)nb * (double)(1LL << lm));
    out[0] = us > 0.0 ? cfl * h / us : __longlong_as_double(0x7ff0000000000000LL);
  }
}

int launch_dt(mr_grid *g, double cfl, const double *uc, const void *const *vel, double *host_out) {
  Tree t = tree_view(g);
  const int n = g->nleaf, nb = g->desc.nb;
  double *part = nullptr;
  if (vel) {
    part = g->maxdet;
    if (g->desc.precision == MR_F32)
      MR_LAUNCH(g, MRK_MISC, k_umax_leaf<float><<<n, 256, 0, g->stream>>>(
                                 nb, (const float *)vel[0], (const float *)vel[1], (const float *)vel[2], part));
    else
      MR_LAUNCH(g, MRK_MISC, k_umax_leaf<double><<<n, 256, 0, g->stream>>>(
                                 nb, (const double *)vel[0], (const double *)vel[1], (const double *)vel[2], part));
  }
  const double us = uc ? fabs(uc[0]) + fabs(uc[1]) + fabs(uc[2]) : 0.0;
  MR_LAUNCH(g, MRK_MISC, k_dt_reduce<<<1, 256, 0, g->stream>>>(part, t.lev, n, us, cfl, t.tree_len, nb,
                                                              g->dscratch + 1));
  if (check_cuda(cudaGetLastError(), "k_dt")) return MR_ERR_CUDA;
  if (check_cuda(cudaMemcpyAsync(host_out, g->dscratch + 1, sizeof(double), cudaMemcpyDeviceToHost, g->stream),
                 "dt copy"))
    return MR_ERR_CUDA;
  return check_cuda(cudaStreamSynchronize(g->stream), "dt sync") ? MR_ERR_CUDA : MR_OK;
}

}  // namespace mr
