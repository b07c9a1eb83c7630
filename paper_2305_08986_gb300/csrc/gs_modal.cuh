// Cell operators of the Q2-Q1 system in the Legendre basis of the cell.
//
// On one axis of a cell, with local nodes 0, 1/2, 1, write the interpolant of nodal values (x0, x1, x2)
// as a0 / 6 L0 + a1 / 2 L1 + a2 / 3 L2 (L_k the Legendre polynomials on [0, 1]):
//   a0 = x0 + 4 x1 + x2,   a1 = x2 - x0,   a2 = x0 - 2 x1 + x2.
// The Legendre polynomials and, up to degree 2, their derivatives (L1' = 2 L0, L2' = 6 L1) are
// orthogonal, so the 1D mass and stiffness matrices are diagonal in (a0, a1, a2),
//   M = diag(1/36, 1/12, 1/45),   K = diag(0, 1, 4/3),
// and the mixed matrix (test derivative, trial value) has the two entries E[1][0] = 1/6, E[2][1] = 1/3.
// A cell application is then: 4 operations per node line into the modes of each axis, one product per
// mode for the whole diagonal block alpha M + eta (grad, grad) + ..., two FMAs per coupled pair of
// modes of two components for the off-diagonal blocks, and 4 operations per line back.  2D: about 150
// operations per cell instead of about 400 in 3 x 3 sweeps; 3D: about 800 instead of about 2,550.
// The way back, y = T^T r, takes one FMA per node because r2 is kept doubled (weights w = 1, 1, 2 on the
// outputs, folded into the coefficients):  t = r0 + r2 / 2,  y0 = t - r1,  y2 = t + r1,  y1 = 4 r0 - r2.
// Differences of nodal values come first, so a rigid translation gives exact zeros in every derivative
// mode.
#pragma once
#include "gs_kernels.h"

namespace gs {

// Coefficients of one level (see make_modal).  Mode index q = i + 3 j (+ 9 k), x fastest.
template <typename T>
struct ModalCoef {
  T dm[10];      // alpha prod h prod_a M_a w_a, by the numbers of 1s and 2s among the mode's indices
  T dk[3][27];   // component a: prod h sum_b (1 + [a = b]) K_b / h_b^2 prod_{c != b} M_c, times the w's
  T dc[3][3];    // coupling of the two components other than p: h_p M_k w_k / 36 (2D: dc[2][0] = 1/36)
  T g2[3], g3[3], g23[3];  // divergence: g_a / 2, g_a / 3, 2 g_a / 3 with g_a = prod_{b != a} h_b / 12
};

// position of a mode in dm: (number of indices equal to 1, number equal to 2)
__host__ __device__ constexpr int modal_class(int i, int j, int k) {
  const int n1 = (i == 1) + (j == 1) + (k == 1), n2 = (i == 2) + (j == 2) + (k == 2);
  return n2 == 0 ? n1 : (n2 == 1 ? 4 + n1 : (n2 == 2 ? 7 + n1 : 9));
}

template <typename T>
inline ModalCoef<T> make_modal(const Geom& g, const OpCoef<T>& c) {
  const int dim = g.dim;
  const double M[3] = {1.0 / 36.0, 1.0 / 12.0, 1.0 / 45.0}, K[3] = {0.0, 1.0, 4.0 / 3.0}, w[3] = {1.0, 1.0, 2.0};
  ModalCoef<T> m{};
  double vol = 1.0;
  for (int a = 0; a < dim; ++a) vol *= g.h[a];
  const double av = (double)c.mm * (dim == 2 ? 900.0 : 27000.0);  // alpha prod h
  for (int k = 0; k < (dim == 3 ? 3 : 1); ++k)
    for (int j = 0; j < 3; ++j)
      for (int i = 0; i < 3; ++i) {
        const int ix[3] = {i, j, k};
        double ww = 1.0, mm = 1.0;
        for (int a = 0; a < dim; ++a) {
          ww *= w[ix[a]];
          mm *= M[ix[a]];
        }
        m.dm[modal_class(i, j, dim == 3 ? k : 0)] = (T)(av * mm * ww);
        for (int comp = 0; comp < dim; ++comp) {
          double s = 0.0;
          for (int b = 0; b < dim; ++b) {
            double t = (b == comp ? 2.0 : 1.0) * K[ix[b]] / (g.h[b] * g.h[b]);
            for (int e = 0; e < dim; ++e)
              if (e != b) t *= M[ix[e]];
            s += t;
          }
          m.dk[comp][i + 3 * j + 9 * k] = (T)(vol * s * ww);
        }
      }
  for (int p = 0; p < 3; ++p)
    for (int k = 0; k < 3; ++k) m.dc[p][k] = (T)(dim == 3 ? g.h[p] * M[k] * w[k] / 36.0 : (k == 0 ? 1.0 / 36.0 : 0.0));
  for (int a = 0; a < dim; ++a) {
    double ga = 1.0;
    for (int b = 0; b < dim; ++b)
      if (b != a) ga *= g.h[b] / 12.0;
    m.g2[a] = (T)(ga / 2.0);
    m.g3[a] = (T)(ga / 3.0);
    m.g23[a] = (T)(2.0 * ga / 3.0);
  }
  return m;
}

template <typename T>
__device__ __forceinline__ void to_modes(T x0, T x1, T x2, T& a0, T& a1, T& a2) {
  const T s = x0 + x2;
  a1 = x2 - x0;
  a0 = fma(T(4), x1, s);
  a2 = fma(T(-2), x1, s);
}
template <typename T>
__device__ __forceinline__ void from_modes(T r0, T r1, T r2, T& y0, T& y1, T& y2) {
  const T t = fma(T(0.5), r2, r0);
  y0 = t - r1;
  y2 = t + r1;
  y1 = fma(T(4), r0, -r2);
}

// modes / nodes of the two trailing axes of a 3 x 3 plane (x fastest), in place
template <typename T>
__device__ __forceinline__ void plane_to_modes(T (&v)[9]) {
#pragma unroll
  for (int j = 0; j < 3; ++j) to_modes(v[3 * j], v[3 * j + 1], v[3 * j + 2], v[3 * j], v[3 * j + 1], v[3 * j + 2]);
#pragma unroll
  for (int i = 0; i < 3; ++i) to_modes(v[i], v[i + 3], v[i + 6], v[i], v[i + 3], v[i + 6]);
}
template <typename T>
__device__ __forceinline__ void plane_from_modes(T (&v)[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) from_modes(v[i], v[i + 3], v[i + 6], v[i], v[i + 3], v[i + 6]);
#pragma unroll
  for (int j = 0; j < 3; ++j) from_modes(v[3 * j], v[3 * j + 1], v[3 * j + 2], v[3 * j], v[3 * j + 1], v[3 * j + 2]);
}

// r = (alpha_K M + eta_K viscous) a in the modes of one 3D cell; mass: the alpha_K-scaled dm
template <typename T>
__device__ __forceinline__ void modal_A3(const T (&a)[3][27], T (&r)[3][27], T eta, const T (&mass)[10],
                                         const ModalCoef<T>& m) {
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int q = i + 3 * j + 9 * k;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const T d = q == 0 ? mass[0] : fma(eta, m.dk[c][q], mass[modal_class(i, j, k)]);
          r[c][q] = d * a[c][q];
        }
      }
  // pairs of components (u, v) along axes (u, v), third axis p: mode (0|1, 1|2) of u with (+1, -1) of v
  constexpr int st[3] = {1, 3, 9};
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int u = p == 0 ? 1 : 0, v = p == 2 ? 1 : 2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T g1 = eta * m.dc[p][k], g2 = T(2) * g1, g4 = T(4) * g1, g8 = T(8) * g1;
      const int b = k * st[p], su = st[u], sv = st[v];
      r[u][b + sv] = fma(g1, a[v][b + su], r[u][b + sv]);
      r[v][b + su] = fma(g1, a[u][b + sv], r[v][b + su]);
      r[u][b + 2 * sv] = fma(g4, a[v][b + su + sv], r[u][b + 2 * sv]);
      r[v][b + su + sv] = fma(g2, a[u][b + 2 * sv], r[v][b + su + sv]);
      r[u][b + su + sv] = fma(g2, a[v][b + 2 * su], r[u][b + su + sv]);
      r[v][b + 2 * su] = fma(g4, a[u][b + su + sv], r[v][b + 2 * su]);
      r[u][b + su + 2 * sv] = fma(g8, a[v][b + 2 * su + sv], r[u][b + su + 2 * sv]);
      r[v][b + 2 * su + sv] = fma(g8, a[u][b + su + 2 * sv], r[v][b + 2 * su + sv]);
    }
  }
}

// r -= B^T beta (beta: the pressure's modes p0 + p1, p1 - p0 per axis, index i + 2 j + 4 k)
template <typename T>
__device__ __forceinline__ void modal_BT3(const T (&beta)[8], T (&r)[3][27], const ModalCoef<T>& m) {
  constexpr int st[3] = {1, 3, 9}, sp[3] = {1, 2, 4};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = q & 1, j = (q >> 1) & 1, k = q >> 2;
      const bool hi = (q & sp[a]) != 0;
      const int t = i + 3 * j + 9 * k + st[a];
      r[a][t] = fma(hi ? -m.g23[a] : -m.g2[a], beta[q], r[a][t]);
    }
}
// gamma = -(div a) against the pressure's modes
template <typename T>
__device__ __forceinline__ void modal_B3(const T (&a)[3][27], T (&gamma)[8], const ModalCoef<T>& m) {
  constexpr int st[3] = {1, 3, 9}, sp[3] = {1, 2, 4};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = q & 1, j = (q >> 1) & 1, k = q >> 2;
    T s = T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) s = fma((q & sp[c]) != 0 ? -m.g3[c] : -m.g2[c], a[c][i + 3 * j + 9 * k + st[c]], s);
    gamma[q] = s;
  }
}

}  // namespace gs
