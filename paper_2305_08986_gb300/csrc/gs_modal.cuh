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

// product kept apart from the sums around it (a contraction there could differ from kernel to kernel)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// (alpha mass + eta viscous) coefficient of mode q >= 1, component c; ms: the mass part.  FP32: with the remainder of
// the viscous coefficient (gs_modal_coef.h).
__device__ __forceinline__ float modal2_diag(const Modal2<float>& m, int q, int c, float eta, float ms) {
  return fmaf(eta, m.dk[q][c], fmaf(eta, m.dl[q][c], ms));
}
__device__ __forceinline__ double modal2_diag(const Modal2<double>& m, int q, int c, double eta, double ms) {
  return fma(eta, m.dk[q][c], ms);
}

// r += coupling of the two components in the modes of one 2D cell: mode (0|1, 1|2) of component x with (+1, -1) of
// component y, products E E = 1/36, ...
template <typename T>
__device__ __forceinline__ void modal2_couple(const T (&a)[2][9], T (&r)[2][9], T eta) {
  const T g1 = mul_rn(eta, T(1.0 / 36.0)), g2 = T(2) * g1, g4 = T(4) * g1, g8 = T(8) * g1;
  r[0][3] = fma(g1, a[1][1], r[0][3]);
  r[1][1] = fma(g1, a[0][3], r[1][1]);
  r[0][6] = fma(g4, a[1][4], r[0][6]);
  r[1][4] = fma(g2, a[0][6], r[1][4]);
  r[0][4] = fma(g2, a[1][2], r[0][4]);
  r[1][2] = fma(g4, a[0][4], r[1][2]);
  r[0][7] = fma(g8, a[1][5], r[0][7]);
  r[1][5] = fma(g8, a[0][7], r[1][5]);
}

// ---- pairs of FP32 values (one instruction, each half rounded as the scalar operation) -------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack2(f32x2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ void to_modes2(f32x2& x0, f32x2& x1, f32x2& x2) {  // x2 - x0 as x0 (-1) + x2: exact product
  const f32x2 s = add2(x0, x2), d = fma2(x0, pack2(-1.f, -1.f), x2);
  x0 = fma2(pack2(4.f, 4.f), x1, s);
  x2 = fma2(pack2(-2.f, -2.f), x1, s);
  x1 = d;
}
__device__ __forceinline__ void from_modes2(f32x2& r0, f32x2& r1, f32x2& r2) {
  const f32x2 t = fma2(pack2(0.5f, 0.5f), r2, r0), y1 = fma2(r2, pack2(-1.f, -1.f), mul2(pack2(4.f, 4.f), r0));
  r0 = fma2(r1, pack2(-1.f, -1.f), t);
  r2 = add2(t, r1);
  r1 = y1;
}
// y = (alpha_K M + eta_K viscous) x of one 2D cell in FP32, the two components in the halves of pairs: the sums of
// cell_modal2 with the same roundings (the same bits) in about 100 instead of 165 instructions.  For the strip kernel: A x
// 1280 x 210 7.74 -> 7.48 us, smoother call 1280 x 224 58.8 -> 57.1 us; small gains, because it waits for its staged rows
// and barriers more than it issues (51 % of the issue slots).  The tile kernels of small meshes keep the scalar form
// (32 x 32 smoother call: 16.1 us, 16.4 us with pairs).
__device__ __forceinline__ void cell_modal2_pair(const float (&x)[2][9], float (&y)[2][9], float eta, float alpha,
                                                 const Modal2<float>& m) {
  f32x2 v[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) v[q] = pack2(x[0][q], x[1][q]);
#pragma unroll
  for (int j = 0; j < 3; ++j) to_modes2(v[3 * j], v[3 * j + 1], v[3 * j + 2]);
#pragma unroll
  for (int i = 0; i < 3; ++i) to_modes2(v[i], v[i + 3], v[i + 6]);
  float a[2][9], r[2][9];
  const f32x2 e = pack2(eta, eta);
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const float ms = mul_rn(alpha, m.dm[modal2_class(q % 3, q / 3)]);
    const f32x2 mm = pack2(ms, ms);
    unpack2(v[q], a[0][q], a[1][q]);
    const f32x2 d = q == 0 ? mm : fma2(e, pack2(m.dk[q][0], m.dk[q][1]), fma2(e, pack2(m.dl[q][0], m.dl[q][1]), mm));
    unpack2(mul2(d, v[q]), r[0][q], r[1][q]);
  }
  modal2_couple(a, r, eta);
#pragma unroll
  for (int q = 0; q < 9; ++q) v[q] = pack2(r[0][q], r[1][q]);
#pragma unroll
  for (int i = 0; i < 3; ++i) from_modes2(v[i], v[i + 3], v[i + 6]);
#pragma unroll
  for (int j = 0; j < 3; ++j) from_modes2(v[3 * j], v[3 * j + 1], v[3 * j + 2]);
#pragma unroll
  for (int q = 0; q < 9; ++q) unpack2(v[q], y[0][q], y[1][q]);
}

// One 2D cell: y = (alpha_K M + eta_K viscous) x + B^T p, pb = B x (nodal values in and out; the blocks
// by the flags), every sum in the cell's modes.  alpha: factor of the mass term (alpha_K or 1).
template <bool WA, bool WBT, bool WB, typename T>
__device__ __forceinline__ void cell_modal2(const T (&x)[2][9], const T (&p)[4], T (&y)[2][9], T (&pb)[4], T eta, T alpha,
                                            const Modal2<T>& m) {
  T a[2][9], r[2][9];
  if (WA || WB) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int q = 0; q < 9; ++q) a[c][q] = x[c][q];
      plane_to_modes(a[c]);
    }
  }
  if (WA) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const T ms = mul_rn(alpha, m.dm[modal2_class(q % 3, q / 3)]);
        r[c][q] = mul_rn(q == 0 ? ms : modal2_diag(m, q, c, eta, ms), a[c][q]);
      }
    modal2_couple(a, r, eta);
  } else if (WBT) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int q = 0; q < 9; ++q) r[c][q] = T(0);
  }
  if (WBT) {
    const T s0 = p[0] + p[1], d0 = p[1] - p[0], s1 = p[2] + p[3], d1 = p[3] - p[2];
    const T b00 = s0 + s1, b10 = d0 + d1, b01 = s1 - s0, b11 = d1 - d0;
    r[0][1] = fma(-m.g2[0], b00, r[0][1]);
    r[0][4] = fma(-m.g2[0], b01, r[0][4]);
    r[0][2] = fma(-m.g23[0], b10, r[0][2]);
    r[0][5] = fma(-m.g23[0], b11, r[0][5]);
    r[1][3] = fma(-m.g2[1], b00, r[1][3]);
    r[1][4] = fma(-m.g2[1], b10, r[1][4]);
    r[1][6] = fma(-m.g23[1], b01, r[1][6]);
    r[1][7] = fma(-m.g23[1], b11, r[1][7]);
  }
  if (WA || WBT) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      plane_from_modes(r[c]);
#pragma unroll
      for (int q = 0; q < 9; ++q) y[c][q] = r[c][q];
    }
  }
  if (WB) {
    const T c00 = fma(-m.g2[0], a[0][1], mul_rn(-m.g2[1], a[1][3]));
    const T c01 = fma(-m.g2[0], a[0][4], mul_rn(-m.g3[1], a[1][6]));
    const T c10 = fma(-m.g3[0], a[0][2], mul_rn(-m.g2[1], a[1][4]));
    const T c11 = fma(-m.g3[0], a[0][5], mul_rn(-m.g3[1], a[1][7]));
    const T s0 = c00 - c01, s1 = c00 + c01, d0 = c10 - c11, d1 = c10 + c11;  // y = 0 / 1: modes along x
    pb[0] = s0 - d0;
    pb[1] = s0 + d0;
    pb[2] = s1 - d1;
    pb[3] = s1 + d1;
  }
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
