// Constraint monitors (Eqs. hamilton_constraints and momentum_constraints)
// with a deterministic two-stage reduction, and the standalone algebraic
// enforcement kernel.
//
// The Ricci tensor of the monitor is the modified Ricci tensor of Eq.
// NR_foccz4_modified_ricci with Z = 0: Gamma-hat replaced by the contracted
// Christoffel symbol G~^k of the metric, whose derivative is taken through
// the closing relations (d_k g~^ij = -2 D_k^ij and the derivative of the
// Christoffel symbols), i.e. from first and second derivatives of g~. Only
// its trace enters H, and the trace needs no tensor: with G~_kij, G~^k_ij the
// Christoffel symbols of g~ and G~_k = g~^ij G~_kij, the terms of the
// contracted derivative cancel against the quadratic ones to
//   g~^ij R~_ij = g~^kn g~^ml (d_k d_m g~_ln - d_k d_l g~_mn)
//                 + g~^ij g~^ml G~^k_im G~_kjl - G~^k G~_k,
// and with the conformal factor
//   phi^2 g~^ij R_ij = phi^2 g~^ij R~_ij + 4 phi (g~^ij d_i d_j phi - G~^k d_k phi)
//                      - 6 g~^ij d_i phi d_j phi.
#include "ccz4_algebra.cuh"
#include "der_view.cuh"

namespace ccz4 {
namespace {

constexpr int RED_THREADS = 256;

// NB: the point's derivatives (DerView), or its neighbourhood in halo'd tiles (Nbhd).
template <class NB>
__device__ __forceinline__ void constraints_point(const NB &N, const StencilCoef<double> &C, double &H, double M[3]) {
  double g[6], ig[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) g[c] = N.at(GXX + c, 0);
  sym_inverse<double>(g, ig);
  const double igw[6] = {ig[0], ig[1] + ig[1], ig[2] + ig[2], ig[3], ig[4] + ig[4], ig[5]};
  double Gd[3][6], Gu[3][6], Gc[3], Gl[3];
  {
    double dg[3][6];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int c = 0; c < 6; ++c) dg[k][c] = fd1<double>(N, GXX + c, N.st[k], 0.5 * C.c1);  // (1/2) d_k g~_ij
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) Gd[k][S6(i, j)] = dg[i][S6(j, k)] + dg[j][S6(i, k)] - dg[k][S6(i, j)];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int c = 0; c < 6; ++c)
      Gu[k][c] = fma(ig[S6(k, 0)], Gd[0][c], fma(ig[S6(k, 1)], Gd[1][c], ig[S6(k, 2)] * Gd[2][c]));
    double s = igw[0] * Gu[k][0], t = igw[0] * Gd[k][0];
#pragma unroll
    for (int c = 1; c < 6; ++c) {
      s = fma(igw[c], Gu[k][c], s);
      t = fma(igw[c], Gd[k][c], t);
    }
    Gc[k] = s;  // G~^k
    Gl[k] = t;  // G~_k
  }
  // the second derivatives, one component g~_ln at a time
  double R = 0.0;
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int n = l; n < 3; ++n) {
      const int c = S6(l, n);
      double dd[6];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int m = k; m < 3; ++m) dd[S6(k, m)] = fdkl<double>(N, GXX + c, k, m, C);
      double s = 0.0, lap = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        s = fma(ig[S6(k, n)], fma(ig[S6(0, l)], dd[S6(k, 0)], fma(ig[S6(1, l)], dd[S6(k, 1)], ig[S6(2, l)] * dd[S6(k, 2)])), s);
#pragma unroll
      for (int q = 0; q < 6; ++q) lap = fma(igw[q], dd[q], lap);
      // both orders of (l, n) give the same first sum
      R = fma(-igw[c], lap, l == n ? R + s : fma(2.0, s, R));
    }
  // the quadratic terms
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double E[3][3];  // G~_ki^m
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int m = 0; m < 3; ++m)
        E[i][m] = fma(ig[S6(0, m)], Gd[k][S6(i, 0)], fma(ig[S6(1, m)], Gd[k][S6(i, 1)], ig[S6(2, m)] * Gd[k][S6(i, 2)]));
    double y = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int m = i; m < 3; ++m) {
        const double u = fma(ig[S6(i, 0)], E[0][m], fma(ig[S6(i, 1)], E[1][m], ig[S6(i, 2)] * E[2][m]));
        y = fma(i == m ? u : u + u, Gu[k][S6(i, m)], y);
      }
    R += fma(-Gc[k], Gl[k], y);
  }
  const double ph = N.at(PHI, 0), Kt = N.at(KTR, 0);
  double dP[3], Pu[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) dP[k] = fd1<double>(N, PHI, N.st[k], C.c1);
#pragma unroll
  for (int k = 0; k < 3; ++k) Pu[k] = fma(ig[S6(k, 0)], dP[0], fma(ig[S6(k, 1)], dP[1], ig[S6(k, 2)] * dP[2]));
  const double PP = fma(Pu[0], dP[0], fma(Pu[1], dP[1], Pu[2] * dP[2]));
  double tr = fma(-Gc[0], dP[0], fma(-Gc[1], dP[1], -Gc[2] * dP[2]));
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int l = k; l < 3; ++l) tr = fma(igw[S6(k, l)], fdkl<double>(N, PHI, k, l, C), tr);
  double A[6], Am[3][3];
#pragma unroll
  for (int c = 0; c < 6; ++c) A[c] = N.at(AXX + c, 0);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int m = 0; m < 3; ++m)
      Am[i][m] = fma(A[S6(i, 0)], ig[S6(0, m)], fma(A[S6(i, 1)], ig[S6(1, m)], A[S6(i, 2)] * ig[S6(2, m)]));
  double AA = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int m = 0; m < 3; ++m) AA = fma(Am[i][m], Am[m][i], AA);
  H = fma(ph, fma(ph, R, 4.0 * tr), fma(-6.0, PP, fma((2.0 / 3.0) * Kt, Kt, -AA)));
  const double iph3 = -3.0 / ph;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    M[i] = fd1<double>(N, KTR, N.st[i], (-2.0 / 3.0) * C.c1);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
#pragma unroll
      for (int l = 0; l < 3; ++l) M[i] = fma(-Gu[m][S6(l, i)], Am[m][l], M[i]);
      M[i] = fma(fma(iph3, Pu[m], -Gc[m]), A[S6(i, m)], M[i]);
    }
  }
  // g~^kl d_k A~_li, one derivative at a time
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int i = l; i < 3; ++i) {
        const double d = fd1<double>(N, AXX + S6(l, i), N.st[k], C.c1);
        M[i] = fma(ig[S6(k, l)], d, M[i]);
        if (i != l) M[l] = fma(ig[S6(k, i)], d, M[l]);
      }
}

struct ConsCoef {
  StencilCoef<double> C[MAX_LEVELS];
};

// What the monitors read: the derivative pass (DER), or halo'd tiles alone
// (the caller's own, which have no derivatives beside them).
struct ConsSrc {
  const double *tile;
  const double *der, *mix, *in;
};

// (From tiles: one block per SM, so that its stack stays within the context's
// default and the first launch needs no larger local-memory pool.)
template <bool DER>
__global__ void __launch_bounds__(RED_THREADS, DER ? 2 : 1) constraints_kernel(GridView g, ConsCoef LC, ConsSrc src, double *H,
                                                                     double *M, double *partial) {
  __shared__ double sh[5][RED_THREADS];
  const int p = g.p, T = g.T;
  const int p3 = p * p * p;  // 32-bit division: every state index is below 2^31
  const long long q0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, i = (long long)g.w0 * p3 + q0;
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (q0 < (long long)g.wn * p3) {
    const int n = (int)i / p3;
    const int r = (int)i - n * p3;
    double h, m[3];
    if constexpr (DER) {
      constraints_point(der_view<false>(g, src.der, src.mix, src.in, i, q0), LC.C[patch_level(g, n)], h, m);
    } else {
      const int z = r / (p * p), y = (r / p) % p, x = r % p;
      Nbhd N;
      N.c = src.tile + n * g.T3 + ((long long)(z + HALO) * T + (y + HALO)) * T + (x + HALO);
      N.fs = (long long)g.n_patches * g.T3;
      N.st[0] = 1;
      N.st[1] = T;
      N.st[2] = T * T;
      N.mix = nullptr;
      N.ms = 0;
      N.mixf = nullptr;
      N.msf = 0;
      constraints_point(N, LC.C[patch_level(g, n)], h, m);
    }
    if (H) H[i] = h;
    if (M) {
      M[i] = m[0];
      M[g.n_points + i] = m[1];
      M[2 * g.n_points + i] = m[2];
    }
    const double m2 = m[0] * m[0] + m[1] * m[1] + m[2] * m[2];
    // the norms count leaf patches only (a covered point is not counted twice)
    const bool counted = !g.leaf || __ldg(g.leaf + n);
    if (counted && isfinite(h) && isfinite(m2)) {
      v[0] = h * h;
      v[1] = m2;
      v[2] = fabs(h);
      v[3] = sqrt(m2);
    } else if (counted) {
      v[4] = 1.0;
    }
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
      sh[2][threadIdx.x] = fmax(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
      sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
      sh[4][threadIdx.x] += sh[4][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x < 5) partial[blockIdx.x * 5 + threadIdx.x] = sh[threadIdx.x][0];
}

// One block folds the per-block partials in a fixed order.
__global__ void __launch_bounds__(RED_THREADS) reduce_partials(const double *partial, int blocks,
                                                               double n_points, double *out) {
  __shared__ double sh[5][RED_THREADS];
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < blocks; b += RED_THREADS) {
    v[0] += partial[b * 5 + 0];
    v[1] += partial[b * 5 + 1];
    v[2] = fmax(v[2], partial[b * 5 + 2]);
    v[3] = fmax(v[3], partial[b * 5 + 3]);
    v[4] += partial[b * 5 + 4];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
      sh[2][threadIdx.x] = fmax(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
      sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
      sh[4][threadIdx.x] += sh[4][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = sqrt(sh[0][0] / n_points);
    out[1] = sqrt(sh[1][0] / n_points);
    out[2] = sh[2][0];
    out[3] = sh[3][0];
    out[4] = sh[4][0];
  }
}

// Centres and radius of the regions left out of the constraint norms.
struct Excl {
  int n;
  double c[CCZ4_MAX_EXCLUDED][3];
  double r2;
};

// Per-block partial sums of H^2 and |M|^2, maxima of |H| and |M| and the
// count over the interior points of leaf patches outside every ball.
__global__ void __launch_bounds__(RED_THREADS) excluded_kernel(GridView g, Excl E, const double *__restrict__ H,
                                                               const double *__restrict__ M, double *partial) {
  __shared__ double sh[5][RED_THREADS];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (i < g.n_points) {
    const int p = g.p;
    const int p3 = p * p * p;
    const int n = (int)i / p3;
    const int r = (int)i - n * p3;
    const int z = r / (p * p), y = (r / p) % p, x = r % p;
    const double h = g.ldx[patch_level(g, n)];
    const double pos[3] = {g.origin[0] + (__ldg(g.ijk + 3 * n) * p + x + 0.5) * h,
                           g.origin[1] + (__ldg(g.ijk + 3 * n + 1) * p + y + 0.5) * h,
                           g.origin[2] + (__ldg(g.ijk + 3 * n + 2) * p + z + 0.5) * h};
    bool near = false;
    for (int c = 0; c < E.n; ++c) {
      const double d0 = pos[0] - E.c[c][0], d1 = pos[1] - E.c[c][1], d2 = pos[2] - E.c[c][2];
      near = near || d0 * d0 + d1 * d1 + d2 * d2 < E.r2;
    }
    const bool counted = (!g.leaf || __ldg(g.leaf + n)) && !near;
    const double hv = H[i];
    const double m2 = M[i] * M[i] + M[g.n_points + i] * M[g.n_points + i] + M[2 * g.n_points + i] * M[2 * g.n_points + i];
    if (counted && isfinite(hv) && isfinite(m2)) {
      v[0] = hv * hv;
      v[1] = m2;
      v[2] = fabs(hv);
      v[3] = sqrt(m2);
      v[4] = 1.0;
    }
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
      sh[2][threadIdx.x] = fmax(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
      sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
      sh[4][threadIdx.x] += sh[4][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x < 5) partial[blockIdx.x * 5 + threadIdx.x] = sh[threadIdx.x][0];
}

// Folds the partials in a fixed order; the norms divide by the point count.
__global__ void __launch_bounds__(RED_THREADS) reduce_excluded(const double *partial, int blocks, double *out) {
  __shared__ double sh[5][RED_THREADS];
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int b = threadIdx.x; b < blocks; b += RED_THREADS) {
    v[0] += partial[b * 5 + 0];
    v[1] += partial[b * 5 + 1];
    v[2] = fmax(v[2], partial[b * 5 + 2]);
    v[3] = fmax(v[3], partial[b * 5 + 3]);
    v[4] += partial[b * 5 + 4];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = RED_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + w];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + w];
      sh[2][threadIdx.x] = fmax(sh[2][threadIdx.x], sh[2][threadIdx.x + w]);
      sh[3][threadIdx.x] = fmax(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
      sh[4][threadIdx.x] += sh[4][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double cnt = sh[4][0];
    out[0] = cnt > 0.0 ? sqrt(sh[0][0] / cnt) : 0.0;
    out[1] = cnt > 0.0 ? sqrt(sh[1][0] / cnt) : 0.0;
    out[2] = sh[2][0];
    out[3] = sh[3][0];
    out[4] = cnt;
  }
}

__global__ void __launch_bounds__(256) enforce_kernel(GridView g, double *U) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.n_points) return;
  double gm[6], A[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    gm[c] = U[(GXX + c) * g.S + i];
    A[c] = U[(AXX + c) * g.S + i];
  }
  enforce_point<double>(gm, A);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    U[(GXX + c) * g.S + i] = gm[c];
    U[(AXX + c) * g.S + i] = A[c];
  }
}

}  // namespace

int constraint_blocks(long long n_points) { return (int)((n_points + RED_THREADS - 1) / RED_THREADS); }

// The block sums of the points of g's window, at their places among all blocks' (a window starts at a
// multiple of RED_THREADS points).
static cudaError_t launch_constraints_from(const GridView &g, const ConsSrc &src, double *H, double *M, double *partial,
                                           cudaStream_t s) {
  ConsCoef LC;
  for (int l = 0; l < MAX_LEVELS; ++l) {
    const double dx = g.ldx[l];
    LC.C[l].c1 = 1.0 / (12.0 * dx);
    LC.C[l].c2 = 1.0 / (12.0 * dx * dx);
    LC.C[l].c3 = 1.0 / (144.0 * dx * dx);
    LC.C[l].cko = 0.0;
  }
  const long long p3 = (long long)g.p * g.p * g.p;
  const int blocks = constraint_blocks(g.wn * p3);
  if (blocks == 0) return cudaSuccess;
  partial += 5 * (g.w0 * p3 / RED_THREADS);
  if (src.der) constraints_kernel<true><<<blocks, RED_THREADS, 0, s>>>(g, LC, src, H, M, partial);
  else constraints_kernel<false><<<blocks, RED_THREADS, 0, s>>>(g, LC, src, H, M, partial);
  return cudaGetLastError();
}

cudaError_t launch_constraints_norms(const GridView &g, const double *partial, int blocks, double *out5, cudaStream_t s) {
  reduce_partials<<<1, RED_THREADS, 0, s>>>(partial, blocks, (double)g.n_leaf_points, out5);
  return cudaGetLastError();
}

cudaError_t launch_constraints(const GridView &g, const double *tile, double *H, double *M, double *partial,
                               int blocks, double *out5, cudaStream_t s) {
  const cudaError_t e = launch_constraints_from(g, ConsSrc{tile, nullptr, nullptr, nullptr}, H, M, partial, s);
  return e == cudaSuccess ? launch_constraints_norms(g, partial, blocks, out5, s) : e;
}

// Loads the kernels of the monitors that take tiles alone (a kernel's first
// launch may take device memory for its code, and their caller may have none
// to give); once per grid.
cudaError_t prepare_constraints() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, constraints_kernel<false>);
  return e == cudaSuccess ? cudaFuncGetAttributes(&a, reduce_partials) : e;
}

cudaError_t launch_constraints_der(const GridView &g, const double *der, const double *mix, const double *in, double *H,
                                   double *M, double *partial, cudaStream_t s) {
  return launch_constraints_from(g, ConsSrc{nullptr, der, mix, in}, H, M, partial, s);
}

cudaError_t launch_constraints_excluded(const GridView &g, const double *H, const double *M, int n_centres,
                                        const double *centres, double radius, double *partial, int blocks,
                                        double *out5, cudaStream_t s) {
  Excl E;
  E.n = n_centres;
  for (int c = 0; c < n_centres; ++c)
    for (int d = 0; d < 3; ++d) E.c[c][d] = centres[3 * c + d];
  E.r2 = radius * radius;
  if (blocks > 0) {
    excluded_kernel<<<blocks, RED_THREADS, 0, s>>>(g, E, H, M, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  reduce_excluded<<<1, RED_THREADS, 0, s>>>(partial, blocks, out5);
  return cudaGetLastError();
}

cudaError_t launch_enforce(const GridView &g, double *U, cudaStream_t s) {
  if (g.n_points == 0) return cudaSuccess;
  enforce_kernel<<<(unsigned)((g.n_points + 255) / 256), 256, 0, s>>>(g, U);
  return cudaGetLastError();
}

}  // namespace ccz4
