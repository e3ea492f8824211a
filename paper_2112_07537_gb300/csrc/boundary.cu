// boundary.cu -- block criterion on forests with physical boundaries
// (Sec. 2.4).  The ghost reconstruction of such grids runs in the kernels of
// all grids (ghost_kernels.cuh: bc_box fills the points beyond the domain).
#include "mr_internal.cuh"

namespace mr {

// Block criterion (Sec. 2.2.5) on a bounded grid: max |gamma| over the part
// of [-ext_f, nb-1+ext_b]^3 inside the domain, gamma at points with an odd
// coordinate by the 1D filters applied x, then y, then z (G^a along odd,
// H^a along even coordinates), from the FP64 padded blocks of the
// adaptation-shell ghost fill.
template <int N, int NT>
__global__ void __launch_bounds__(256) k_bcriterion(Tree t, const double *__restrict__ P, int Gi, double *maxdet) {
  using W = Wav<N, NT>;
  const int b = blockIdx.x, nb = t.nb, Wd = nb + 2 * Gi;
  const int L = __ldg(t.lev + b);
  const int a[3] = {__ldg(t.anc + 3 * b) * nb, __ldg(t.anc + 3 * b + 1) * nb, __ldg(t.anc + 3 * b + 2) * nb};
  const double *Pb = P + (size_t)b * Wd * Wd * Wd;
  const int lo = -W::ext_f, E = nb + W::ext_f + W::ext_b;
  unsigned long long best = 0;
  for (int p = threadIdx.x; p < E * E * E; p += blockDim.x) {
    const int c[3] = {lo + p % E, lo + (p / E) % E, lo + p / (E * E)};
    if (!((c[0] | c[1] | c[2]) & 1)) continue;
    const int g[3] = {a[0] + c[0], a[1] + c[1], a[2] + c[2]};
    if (beyond3(t, L, g)) continue;
    const int hx = (c[0] & 1) ? W::hwG : W::hwH, hy = (c[1] & 1) ? W::hwG : W::hwH, hz = (c[2] & 1) ? W::hwG : W::hwH;
    double bz = 0.0;
    for (int tz = -hz; tz <= hz; ++tz) {
      const double wz = (c[2] & 1) ? W::G(tz) : W::H(tz);
      if (wz == 0.0) continue;
      double by = 0.0;
      for (int ty = -hy; ty <= hy; ++ty) {
        const double wy = (c[1] & 1) ? W::G(ty) : W::H(ty);
        if (wy == 0.0) continue;
        double bx = 0.0;
        for (int tx = -hx; tx <= hx; ++tx) {
          const double wx = (c[0] & 1) ? W::G(tx) : W::H(tx);
          if (wx == 0.0) continue;
          bx += wx * Pb[(c[0] + tx + Gi) + Wd * ((c[1] + ty + Gi) + (size_t)Wd * (c[2] + tz + Gi))];
        }
        by += wy * bx;
      }
      bz += wz * by;
    }
    const unsigned long long key = abs_key(bz);
    if (key > best) best = key;
  }
  __shared__ unsigned long long red;
  if (threadIdx.x == 0) red = 0;
  __syncthreads();
  atomicMax(&red, best);
  __syncthreads();
  if (threadIdx.x == 0) maxdet[b] = __longlong_as_double((long long)red);
}

int launch_criterion_bounded(mr_grid *g, const double *P, int Gi, double *maxdet) {
  Tree t = tree_view(g);
  const int N = g->desc.wav_N, Nt = g->desc.wav_Nt, n = g->nleaf;
#define MR_KCASE(n_, nt_)                                                                                     \
  if (N == n_ && Nt == nt_) {                                                                                 \
    MR_LAUNCH(g, MRK_CRITERION, k_bcriterion<n_, nt_><<<n, 256, 0, g->stream>>>(t, P, Gi, maxdet));           \
    return check_cuda(cudaGetLastError(), "k_bcriterion") ? MR_ERR_CUDA : MR_OK;                              \
  }
  MR_KCASE(2, 0) MR_KCASE(2, 2) MR_KCASE(4, 0) MR_KCASE(4, 2) MR_KCASE(6, 0) MR_KCASE(6, 2)
#undef MR_KCASE
  return MR_ERR_UNSUPPORTED;
}

}  // namespace mr
