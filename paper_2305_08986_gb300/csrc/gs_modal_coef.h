// Coefficients of the cell operators in the cells' Legendre modes (gs_modal.cuh): host arithmetic only.
//
// Every cell of a level has the same coefficients, so their rounding does not average out: it is a relative change of
// the operator that all cells share.  They are therefore formed as unevaluated sums of two doubles (about 106 bits,
// Dekker 1971) and rounded once: FP64 coefficients are the nearest doubles (formed in doubles they were up to 2.4
// half-units off).  The FP32 coefficients of the 2D viscous block keep their remainder as a second float (dl), which
// the kernels add before the product with eta is rounded: rounded alone they raised the error of A x by up to a fifth
// (37 x 41 cells 5.7e-8 -> 6.8e-8 relative to the norm, 5.9e-8 with the remainder; 3 x 3 sweeps 5.7e-8).
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define GS_HD __host__ __device__
#else
#define GS_HD
#endif

namespace gs {

// Coefficients of one level in 3D.  Mode index q = i + 3 j + 9 k, x fastest.
template <typename T>
struct ModalCoef {
  T dm[10];      // alpha prod h prod_a M_a w_a, by the numbers of 1s and 2s among the mode's indices
  T dk[3][27];   // component a: prod h sum_b (1 + [a = b]) K_b / h_b^2 prod_{c != b} M_c, times the w's
  T dc[3][3];    // coupling of the two components other than p: h_p M_k w_k / 36
  T g2[3], g3[3], g23[3];  // divergence: g_a / 2, g_a / 3, 2 g_a / 3 with g_a = prod_{b != a} h_b / 12
};

// Coefficients of one level in 2D, mode i + 3 j.
template <typename T>
struct Modal2 {
  T dm[6];               // alpha hx hy M_i M_j w_i w_j by modal2_class(i, j)
  T dk[9][2], dl[9][2];  // component a: hx hy sum_b (1 + [a = b]) K_b / h_b^2 M_other, times the w's; dl: what T leaves
  T g2[2], g3[2], g23[2];  // divergence: h_other / 24, h_other / 36, h_other / 18
};

// position of a 3D mode in dm: (number of indices equal to 1, number equal to 2)
GS_HD constexpr int modal_class(int i, int j, int k) {
  const int n1 = (i == 1) + (j == 1) + (k == 1), n2 = (i == 2) + (j == 2) + (k == 2);
  return n2 == 0 ? n1 : (n2 == 1 ? 4 + n1 : (n2 == 2 ? 7 + n1 : 9));
}
// position of a 2D mode (i, j) in dm (symmetric in i and j)
GS_HD constexpr int modal2_class(int i, int j) {
  const int lo = i < j ? i : j, hi = i < j ? j : i;
  return lo == 0 ? hi : (lo == 1 ? 2 + hi : 5);
}

struct TwoSum { double hi, lo; };  // hi + lo, |lo| at most half a unit of hi
inline TwoSum two_sum(double big, double small) {
  const double s = big + small;
  return {s, small - (s - big)};
}
inline TwoSum operator*(TwoSum a, double b) {
  const double p = a.hi * b;
  return two_sum(p, std::fma(a.lo, b, std::fma(a.hi, b, -p)));
}
inline TwoSum operator/(TwoSum a, double b) {
  const double q = a.hi / b;
  return two_sum(q, (std::fma(-q, b, a.hi) + a.lo) / b);
}
inline TwoSum operator+(TwoSum a, TwoSum b) {  // of the same sign
  const double s = a.hi + b.hi, t = s - a.hi;
  return two_sum(s, (a.hi - (s - t)) + (b.hi - t) + (a.lo + b.lo));
}

namespace modal {
// 1D matrices M = diag(1/36, 1/12, 1/45), K = diag(0, 1, 4/3) and the output weights w = 1, 1, 2 as ratios
constexpr double kM[3] = {36.0, 12.0, 45.0}, kK[3] = {0.0, 3.0, 4.0}, kW[3] = {1.0, 1.0, 2.0};

inline TwoSum mass(int dim, const double* h, double alpha, const int* ix) {
  TwoSum m{alpha, 0.0};
  for (int a = 0; a < dim; ++a) m = m * h[a] * kW[ix[a]] / kM[ix[a]];
  return m;
}
// (component c)  prod h sum_b (1 + [b = c]) K_b / h_b^2 prod_{e != b} M_e, times the w's
inline TwoSum viscous(int dim, const double* h, int c, const int* ix) {
  TwoSum s{0.0, 0.0};
  for (int b = 0; b < dim; ++b) {
    TwoSum t{(b == c ? 2.0 : 1.0) * kK[ix[b]], 0.0};
    if (t.hi == 0.0) continue;
    t = t / 3.0 / h[b];
    for (int e = 0; e < dim; ++e) {
      t = t * kW[ix[e]];
      if (e != b) t = t * h[e] / kM[ix[e]];
    }
    s = s.hi == 0.0 ? t : s + t;
  }
  return s;
}
inline TwoSum divergence(int dim, const double* h, int a) {
  TwoSum g{1.0, 0.0};
  for (int b = 0; b < dim; ++b)
    if (b != a) g = g * h[b] / 12.0;
  return g;
}
template <typename T>
inline T rounded(TwoSum s) { return (T)s.hi; }
template <typename T>
inline T remainder(TwoSum s) { return (T)((s.hi - (double)(T)s.hi) + s.lo); }
}  // namespace modal

// alpha: of the level, or 1 where the cells carry their own
template <typename T>
inline ModalCoef<T> make_modal(const double* h, double alpha) {
  ModalCoef<T> m{};
  for (int k = 0; k < 3; ++k)
    for (int j = 0; j < 3; ++j)
      for (int i = 0; i < 3; ++i) {
        const int ix[3] = {i, j, k};
        m.dm[modal_class(i, j, k)] = modal::rounded<T>(modal::mass(3, h, alpha, ix));
        for (int c = 0; c < 3; ++c) m.dk[c][i + 3 * j + 9 * k] = modal::rounded<T>(modal::viscous(3, h, c, ix));
      }
  for (int p = 0; p < 3; ++p)
    for (int k = 0; k < 3; ++k)
      m.dc[p][k] = modal::rounded<T>(TwoSum{h[p], 0.0} * modal::kW[k] / modal::kM[k] / 36.0);
  for (int a = 0; a < 3; ++a) {
    const TwoSum g = modal::divergence(3, h, a);
    m.g2[a] = modal::rounded<T>(g * 0.5);
    m.g3[a] = modal::rounded<T>(g / 3.0);
    m.g23[a] = modal::rounded<T>(g * 2.0 / 3.0);
  }
  return m;
}

template <typename T>
inline Modal2<T> make_modal2(const double* h, double alpha) {
  Modal2<T> m{};
  for (int j = 0; j < 3; ++j)
    for (int i = 0; i < 3; ++i) {
      const int ix[2] = {i, j};
      m.dm[modal2_class(i, j)] = modal::rounded<T>(modal::mass(2, h, alpha, ix));
      for (int c = 0; c < 2; ++c) {
        const TwoSum v = modal::viscous(2, h, c, ix);
        m.dk[i + 3 * j][c] = modal::rounded<T>(v);
        m.dl[i + 3 * j][c] = modal::remainder<T>(v);
      }
    }
  for (int a = 0; a < 2; ++a) {
    const TwoSum g = modal::divergence(2, h, a);
    m.g2[a] = modal::rounded<T>(g * 0.5);
    m.g3[a] = modal::rounded<T>(g / 3.0);
    m.g23[a] = modal::rounded<T>(g * 2.0 / 3.0);
  }
  return m;
}

}  // namespace gs
