// psi_4 at every interior point (appendix "psi_4 in ExaGRyPE"): the
// electric and magnetic parts of the Weyl tensor in their Z4 form
// (Eqs. eq_NR_psi4_E_ij, eq_NR_psi4_B_ij, vacuum), contracted with mbar of
// the Gram-Schmidt tetrad (Eqs. eq_NR_psi4_m_conj,
// eq_NR_psi_code_implementation). A monitor, evaluated in FP64 from the
// derivative pass; Re and Im
// go to fields 0 and 1 of a state-shaped buffer, where the particle tracers
// can sample them (the paper attaches psi_4 to the solution vector and
// interpolates it onto tracers arranged on a sphere).
//
// The physical Ricci tensor is taken through the conformal decomposition,
// R_ij = R~_ij + R^phi_ij, with R~_ij of the conformal metric alone (its
// contracted Christoffel symbol G~^k from the metric's derivatives) and
// R^phi_ij = (nabla~_i nabla~_j phi + g~_ij nabla~^l nabla~_l phi) / phi
//            - 2 g~_ij g~^kl d_k phi d_l phi / phi^2;
// Z_i = 1/2 g~_ij (Gamma-hat^j - G~^j) enters through D_(i Z_j).
//
// What bounds it is the FP64 pipe, so the contraction is arranged for few
// operations: mbar is null and built of two unit vectors w, v orthogonal to
// each other, so every part of E_ij and B_ij proportional to g~_ij drops out
// (the trace parts, g~_ij nabla~^2 phi, g~_ij (d phi)^2, the g~_ij K parts and
// the trace-free projection) and is not formed. B is taken as the curl of the
// lowered K_ij, eps^kmn D_m K_nj, in which the symmetric part of the
// Christoffel symbols cancels:
//   D_m K_nj - D_n K_mj = phi^-2 (T_mnj - T_nmj),
//   T_mnj = d_m A~_nj - G~^q_mj A~_nq - (d_m phi A~_nj + g~_mj A~_nq d~^q phi) / phi + g~_nj d_m K / 3,
// and contracted with w and v at once. (1350 FP64 operations a point instead
// of 4500; with the derivative pass 13.24 -> 6.03 ms on the two-level mesh of
// 1.63 M points.)
#include "ccz4_algebra.cuh"
#include "der_view.cuh"

namespace ccz4 {
namespace {

struct Psi4Coef {
  StencilCoef<double> C[MAX_LEVELS];
};

// a^i b^j T_ij of a symmetric T stored as six components
__device__ __forceinline__ double quad(const double T[6], const double a[3], const double b[3]) {
  const double t0 = fma(T[0], b[0], fma(T[1], b[1], T[2] * b[2])), t1 = fma(T[1], b[0], fma(T[3], b[1], T[4] * b[2])),
               t2 = fma(T[2], b[0], fma(T[4], b[1], T[5] * b[2]));
  return fma(a[0], t0, fma(a[1], t1, a[2] * t2));
}

__device__ __forceinline__ void psi4_point(const DerView<false> &N, const StencilCoef<double> &C, const double X[3],
                                           double out[2]) {
  double g[6], ig[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) g[c] = N.at(GXX + c, 0);
  const double det = sym_inverse<double>(g, ig);
  const double igw[6] = {ig[0], ig[1] + ig[1], ig[2] + ig[2], ig[3], ig[4] + ig[4], ig[5]};
  const double ph = N.at(PHI, 0), iph = 1.0 / ph;
  // conformal Christoffel symbols, G~^k and G~_k; dIg[l][c] = g~^ma g~^nb d_l g~_ab
  double Gd[3][6], Gu[3][6], Gt[3], Gl[3], dIg[3][6], dg[3][6];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int c = 0; c < 6; ++c) dg[k][c] = fd1<double>(N, GXX + c, N.st[k], C.c1);
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j)
        Gd[k][S6(i, j)] = 0.5 * (dg[i][S6(j, k)] + dg[j][S6(i, k)] - dg[k][S6(i, j)]);
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
    Gt[k] = s;
    Gl[k] = t;
    double E[3][3];
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        E[m][b] = fma(ig[S6(m, 0)], dg[k][S6(0, b)], fma(ig[S6(m, 1)], dg[k][S6(1, b)], ig[S6(m, 2)] * dg[k][S6(2, b)]));
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int l = m; l < 3; ++l)
        dIg[k][S6(m, l)] = fma(E[m][0], ig[S6(0, l)], fma(E[m][1], ig[S6(1, l)], E[m][2] * ig[S6(2, l)]));
  }
  // d_j G~_n = -dIg[j]:G~_n + g~^ml (d_j d_m g~_ln - 1/2 d_j d_n g~_ml) and the Laplacians of g~,
  // one component's second derivatives at a time; Ric collects the Ricci tensor
  double dGl[3][3], Ric[6];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      double s = 0.0;
#pragma unroll
      for (int c = 0; c < 6; ++c) s = fma((c == 1 || c == 2 || c == 4) ? -2.0 * dIg[j][c] : -dIg[j][c], Gd[n][c], s);
      dGl[j][n] = s;
    }
  {
    double Q[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
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
        double lap = 0.0;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          lap = fma(igw[q], dd[q], lap);
          Q[q] = fma(igw[c], dd[q], Q[q]);
        }
        Ric[c] = -0.5 * lap;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            dGl[j][n] = fma(ig[S6(m, l)], dd[S6(j, m)], dGl[j][n]);
            if (l != n) dGl[j][l] = fma(ig[S6(m, n)], dd[S6(j, m)], dGl[j][l]);
          }
        }
      }
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int n = 0; n < 3; ++n) dGl[j][n] = fma(-0.5, Q[S6(j, n)], dGl[j][n]);
  }
  double dGt[3][3];  // dGt[j][k] = d_j G~^k
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      double s = 0.0;
#pragma unroll
      for (int n = 0; n < 3; ++n) s = fma(-dIg[j][S6(k, n)], Gl[n], fma(ig[S6(k, n)], dGl[j][n], s));
      dGt[j][k] = s;
    }
  // R~_ij = -1/2 g~^lm d_l d_m g~_ij + g~_k(i d_j) G~^k + 1/2 G~^k d_k g~_ij
  //         + g~^lm (G~^k_li G~_jkm + G~^k_lj G~_ikm + G~^k_im G~_klj)
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      double t = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        t = fma(g[S6(k, i)], dGt[j][k], fma(g[S6(k, j)], dGt[i][k], fma(Gt[k], dg[k][S6(i, j)], t)));
      Ric[S6(i, j)] = fma(0.5, t, Ric[S6(i, j)]);
    }
  {
    double Cm[3][3][3], Xq[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int m = 0; m < 3; ++m)
          Cm[k][i][m] = fma(ig[S6(0, m)], Gu[k][S6(0, i)], fma(ig[S6(1, m)], Gu[k][S6(1, i)], ig[S6(2, m)] * Gu[k][S6(2, i)]));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 9; ++q) s = fma(Cm[q / 3][i][q % 3], Gd[j][S6(q / 3, q % 3)], s);
        Xq[i][j] = s;
      }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        double s = Xq[i][j] + Xq[j][i];
#pragma unroll
        for (int q = 0; q < 9; ++q) s = fma(Cm[q / 3][i][q % 3], Gd[q / 3][S6(q % 3, j)], s);
        Ric[S6(i, j)] += s;
      }
  }
  // E_ij = R_ij - K_im K^m_j + K_ij (K - Theta) + D_(i Z_j) without its parts proportional to g~_ij:
  // nabla~_i nabla~_j phi / phi, (A~_ij (K - Theta) - A~_im A~^m_j - (2/3) K A~_ij) / phi^2,
  // d_(i Z_j) - G~^m_ij Z_m + (Z_i d_j phi + Z_j d_i phi) / phi
  double dP[3], Pu[3], A[6], E[6], AP[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) dP[k] = fd1<double>(N, PHI, N.st[k], C.c1);
#pragma unroll
  for (int k = 0; k < 3; ++k) Pu[k] = fma(ig[S6(k, 0)], dP[0], fma(ig[S6(k, 1)], dP[1], ig[S6(k, 2)] * dP[2]));
#pragma unroll
  for (int c = 0; c < 6; ++c) A[c] = N.at(AXX + c, 0);
  {
    const double Kt = N.at(KTR, 0), iph2 = iph * iph, ck = fma(1.0 / 3.0, Kt, -N.at(THETA, 0));  // K - Theta - 2 K / 3
    double dG[3], Z[3], dZ[3][3], Am[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) dG[i] = N.at(GHX + i, 0) - Gt[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) Z[i] = 0.5 * fma(g[S6(i, 0)], dG[0], fma(g[S6(i, 1)], dG[1], g[S6(i, 2)] * dG[2]));
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) dGt[k][j] = fd1<double>(N, GHX + j, N.st[k], C.c1) - dGt[k][j];  // d_k (Gamma-hat^j - G~^j)
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) s = fma(dg[k][S6(i, j)], dG[j], fma(g[S6(i, j)], dGt[k][j], s));
        dZ[k][i] = s;  // 2 d_k Z_i
      }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int m = 0; m < 3; ++m)
        Am[i][m] = fma(A[S6(i, 0)], ig[S6(0, m)], fma(A[S6(i, 1)], ig[S6(1, m)], A[S6(i, 2)] * ig[S6(2, m)]));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int c = S6(i, j);
        double s = fma(0.25, dZ[i][j] + dZ[j][i], Ric[c]), q = fdkl<double>(N, PHI, i, j, C);
        double a = ck * A[c];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          s = fma(-Gu[m][c], Z[m], s);
          q = fma(-Gu[m][c], dP[m], q);
          a = fma(-Am[i][m], A[S6(m, j)], a);
        }
        q = fma(Z[i], dP[j], fma(Z[j], dP[i], q));
        E[c] = fma(iph2, a, fma(iph, q, s));
      }
#pragma unroll
    for (int i = 0; i < 3; ++i) AP[i] = fma(A[S6(i, 0)], Pu[0], fma(A[S6(i, 1)], Pu[1], A[S6(i, 2)] * Pu[2]));
  }
  // curl[k][j] = T_mnj - T_nmj, (m, n, k) cyclic: sqrt(det g~) / phi times eps^kmn D_m K_nj
  double curl[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int m = (k + 1) % 3, n = (k + 2) % 3;
      double s = fd1<double>(N, AXX + S6(n, j), N.st[m], C.c1) - fd1<double>(N, AXX + S6(m, j), N.st[n], C.c1);
#pragma unroll
      for (int q = 0; q < 3; ++q) s = fma(Gu[q][S6(n, j)], A[S6(m, q)], fma(-Gu[q][S6(m, j)], A[S6(n, q)], s));
      double t = fma(dP[n], A[S6(m, j)], -dP[m] * A[S6(n, j)]);
      t = fma(g[S6(n, j)], AP[m], fma(-g[S6(m, j)], AP[n], t));
      curl[k][j] = fma(iph, t, s);
    }
  {
    double dK[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) dK[k] = fd1<double>(N, KTR, N.st[k], (1.0 / 3.0) * C.c1);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int m = (k + 1) % 3, n = (k + 2) % 3;
        curl[k][j] = fma(g[S6(n, j)], dK[m], fma(-g[S6(m, j)], dK[n], curl[k][j]));
      }
  }
  // the tetrad: Gram-Schmidt of v = (-y, x, 0), u = (x, y, z), w = gamma^-1 eps(v, u) with gamma = g~ / phi^2
  const double i2 = iph * iph;
  auto dot = [&](const double a[3], const double b[3]) { return quad(g, a, b) * i2; };
  const double sdet = sqrt(det) * iph * iph * iph;  // sqrt(det gamma)
  double v[3] = {-X[1], X[0], 0.0}, u[3] = {X[0], X[1], X[2]}, w[3];
  double nrm = rsqrt(dot(v, v));
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] *= nrm;
  const double vu = dot(v, u);
#pragma unroll
  for (int i = 0; i < 3; ++i) u[i] -= vu * v[i];
  nrm = rsqrt(dot(u, u));
#pragma unroll
  for (int i = 0; i < 3; ++i) u[i] *= nrm;
  const double c[3] = {sdet * (v[1] * u[2] - v[2] * u[1]), sdet * (v[2] * u[0] - v[0] * u[2]),
                       sdet * (v[0] * u[1] - v[1] * u[0])};  // eps_jkl v^k u^l
#pragma unroll
  for (int i = 0; i < 3; ++i)
    w[i] = ph * ph * fma(ig[S6(i, 0)], c[0], fma(ig[S6(i, 1)], c[1], ig[S6(i, 2)] * c[2]));
  const double vw = dot(v, w), uw = dot(u, w);
#pragma unroll
  for (int i = 0; i < 3; ++i) w[i] -= vw * v[i] + uw * u[i];
  nrm = rsqrt(dot(w, w));
#pragma unroll
  for (int i = 0; i < 3; ++i) w[i] *= nrm;
  // B_ij a^i b^j = gamma_ik a^i (eps^kmn D_m K_nj) b^j, symmetrised: eps^kmn D_m K_nj = phi^3 / sqrt(det g~) phi^-2 curl
  double wl[3], vl[3], cw[3], cv[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    wl[i] = fma(g[S6(i, 0)], w[0], fma(g[S6(i, 1)], w[1], g[S6(i, 2)] * w[2]));
    vl[i] = fma(g[S6(i, 0)], v[0], fma(g[S6(i, 1)], v[1], g[S6(i, 2)] * v[2]));
    cw[i] = fma(curl[i][0], w[0], fma(curl[i][1], w[1], curl[i][2] * w[2]));
    cv[i] = fma(curl[i][0], v[0], fma(curl[i][1], v[1], curl[i][2] * v[2]));
  }
  const double sb = iph * rsqrt(det);  // phi^-2 (lowering) phi^3 phi^-2 / sqrt(det g~)
  const double Bww = fma(wl[0], cw[0], fma(wl[1], cw[1], wl[2] * cw[2])) * sb;
  const double Bvv = fma(vl[0], cv[0], fma(vl[1], cv[1], vl[2] * cv[2])) * sb;
  const double Bwv = 0.5 * sb * (fma(wl[0], cv[0], fma(wl[1], cv[1], wl[2] * cv[2])) +
                                 fma(vl[0], cw[0], fma(vl[1], cw[1], vl[2] * cw[2])));
  // (E - i B)_ij mbar^i mbar^j, mbar = (w - i v) / sqrt 2
  out[0] = 0.5 * (quad(E, w, w) - quad(E, v, v)) - Bwv;
  out[1] = -quad(E, w, v) - 0.5 * (Bww - Bvv);
}

__global__ void __launch_bounds__(128, 3) psi4_kernel(GridView g, Psi4Coef PC, const double *__restrict__ der,
                                                      const double *__restrict__ mix, const double *__restrict__ in,
                                                      double cx, double cy, double cz, double *__restrict__ out) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int p = g.p, p3 = p * p * p;
  if (q >= (long long)g.wn * p3) return;
  const long long i = (long long)g.w0 * p3 + q;
  const int n = (int)i / p3;
  const int r = (int)i - n * p3;
  const int z = r / (p * p), y = (r / p) % p, x = r % p;
  const int lev = patch_level(g, n);
  const double h = g.ldx[lev];
  const double X[3] = {g.origin[0] + (__ldg(g.ijk + 3 * n) * p + x + 0.5) * h - cx,
                       g.origin[1] + (__ldg(g.ijk + 3 * n + 1) * p + y + 0.5) * h - cy,
                       g.origin[2] + (__ldg(g.ijk + 3 * n + 2) * p + z + 0.5) * h - cz};
  double v[2];
  psi4_point(der_view<false>(g, der, mix, in, i, q), PC.C[lev], X, v);
  out[i] = v[0];
  out[g.S + i] = v[1];
}

}  // namespace

cudaError_t launch_psi4(const GridView &g, const double *der, const double *mix, const double *in,
                        const double centre[3], double *out, cudaStream_t s) {
  const long long points = (long long)g.wn * g.p * g.p * g.p;
  if (points == 0) return cudaSuccess;
  Psi4Coef PC;
  for (int l = 0; l < MAX_LEVELS; ++l) {
    const double dx = g.ldx[l];
    PC.C[l].c1 = 1.0 / (12.0 * dx);
    PC.C[l].c2 = 1.0 / (12.0 * dx * dx);
    PC.C[l].c3 = 1.0 / (144.0 * dx * dx);
    PC.C[l].cko = 0.0;
  }
  psi4_kernel<<<(unsigned)((points + 127) / 128), 128, 0, s>>>(g, PC, der, mix, in, centre[0], centre[1], centre[2],
                                                                    out);
  return cudaGetLastError();
}

}  // namespace ccz4
