// The two halves of a level in the pressure-Laplacian V-cycle (Cahouet-Chabard term), each in one launch, for the
// smoother of degree 2 with one smoothing step (the defaults):
//   down  x0 = D^-1 b / theta;  x = x0 + c1 x0 + c2 D^-1 (b - K x0);  b_c = R (b - K x)
//   up    x <- x + P e;  d = D^-1 (b - K x) / theta, x <- x + d;  x <- x + c1 d + c2 D^-1 (b - K x)
// (K: the operator of gs_q1tile.cu, R / P: bilinear transfers; entries with a mask are zero throughout.)
//
// The levels of this cycle hold 328 to 290,000 nodes, and a launch costs 2.5 to 3 us whatever it holds, so the
// cycle was bound by its launches, seven per level.  A CTA evaluates a box of nodes with the halo that the
// following stages need (3 nodes down, 2 up) in shared memory and repeats the halo's work of its neighbours:
// 1.9 (2D) or 6 (3D) node evaluations per node instead of one, against five launches and as many passes over memory.
// Pressure V-cycle on the 1280 x 224 hierarchy (FP32, six levels): 99.9 -> 54.9 us; channel solve 38.8 -> 37.0 ms.
//
// The repeated evaluations are worth it while launches bound the level (q1cycle_max_nodes in gs_kernels.h).  One cycle
// with the finest level in two launches / in seven, us:
//   2D FP32  512^2 66 / 78, 2048^2 312 / 375: every level in two
//   2D FP64  320^2 136 / 138, 384^2 169 / 166, 512^2 223 / 212, 768^2 366 / 333: up to 2^17 nodes
//   3D FP32  48^3 75 / 82, 56^3 78 / 82, 64^3 105 / 103, 80^3 148 / 135: up to 2^18 nodes
//   3D FP64  8^3 66 / 49, 32^3 244 / 208 (all levels in seven: 172): the FP64 pipe bounds even the smallest; none
#include "gs_kernels.h"

namespace gs {
namespace {

template <int DIM>
struct Box;  // coarse nodes per CTA; the fine box is twice as wide
template <>
struct Box<2> { static constexpr int C0 = 16, C1 = 4, C2 = 1; };
template <>
struct Box<3> { static constexpr int C0 = 4, C1 = 4, C2 = 2; };

// window of F + 2 H - (H == 3) nodes per axis, starting H nodes below the box
template <int DIM, int H>
struct Win {
  using B = Box<DIM>;
  static constexpr int X0 = 2 * B::C0 + 2 * H - (H == 3), X1 = 2 * B::C1 + 2 * H - (H == 3),
                       X2 = DIM == 3 ? 2 * B::C2 + 2 * H - (H == 3) : 1;
  static constexpr int XY = X0 * X1, N = XY * X2;
};

// (K x)(p) from the window: sx nodes, sc cell scalars (at the cell's lowest node); sums as in gs_q1tile.cu
template <typename T, int DIM, class W>
__device__ __forceinline__ T apply(const T* sx, const T* sc, int p, const T* kc) {
  T acc = T(0);
#pragma unroll
  for (int cz = 0; cz < (DIM == 3 ? 2 : 1); ++cz)
#pragma unroll
    for (int cy = 0; cy < 2; ++cy)
#pragma unroll
      for (int cx = 0; cx < 2; ++cx) {
        const int qa = 1 - cx, qb = 1 - cy, qc = 1 - cz;
        const int lc = p - qa - W::X0 * qb - (DIM == 3 ? W::XY * qc : 0);
        T cellsum = T(0);
#pragma unroll
        for (int rc = 0; rc < (DIM == 3 ? 2 : 1); ++rc)
#pragma unroll
          for (int rb = 0; rb < 2; ++rb)
#pragma unroll
            for (int ra = 0; ra < 2; ++ra) {
              const T pa = qa == ra ? T(2) : T(1), pb = qb == rb ? T(2) : T(1);
              const T ka = qa == ra ? T(1) : T(-1), kb = qb == rb ? T(1) : T(-1);
              T w;
              if (DIM == 2) {
                w = kc[0] * ka * pb + kc[1] * pa * kb;
              } else {
                const T pc = qc == rc ? T(2) : T(1), kk = qc == rc ? T(1) : T(-1);
                w = kc[0] * ka * pb * pc + kc[1] * pa * kb * pc + kc[2] * pa * pb * kk;
              }
              cellsum += w * sx[lc + ra + W::X0 * rb + W::XY * rc];
            }
        acc += sc[lc] * cellsum;
      }
  return acc;
}

// f(p, i0, i1, i2) on the window nodes with lo <= i < X - hi along every axis
template <int DIM, class W, int LO, int HI, class F>
__device__ __forceinline__ void for_nodes(F&& f) {
  constexpr int E0 = W::X0 - LO - HI, E1 = W::X1 - LO - HI, E2 = DIM == 3 ? W::X2 - LO - HI : 1;
  for (int i = threadIdx.x; i < E0 * E1 * E2; i += 256) {
    const int i0 = LO + i % E0, i1 = LO + (i / E0) % E1, i2 = DIM == 3 ? LO + i / (E0 * E1) : 0;
    f(i0 + W::X0 * i1 + W::XY * i2, i0, i1, i2);
  }
}

template <int DIM>
struct Origin {
  int c[3];  // the box's first coarse node
  __device__ __forceinline__ Origin(const Geom& gc, int blk) {
    using B = Box<DIM>;
    const int nb0 = (gc.npn[0] + B::C0 - 1) / B::C0, nb1 = (gc.npn[1] + B::C1 - 1) / B::C1;
    c[0] = blk % nb0 * B::C0;
    c[1] = blk / nb0 % nb1 * B::C1;
    c[2] = DIM == 3 ? blk / (nb0 * nb1) * B::C2 : 0;
  }
};

// b and D^-1 of the window's nodes (0 and -1 outside the mesh and on masked nodes) and its cell scalars
template <typename T, int DIM, class W, int H>
__device__ __forceinline__ void stage(const Q1CycleArgs<T>& A, const int* c, T* sb, T* sd, T* sc) {
  const Geom& g = A.gf;
  for_nodes<DIM, W, 0, 0>([&](int p, int i0, int i1, int i2) {
    const int I = 2 * c[0] - H + i0, J = 2 * c[1] - H + i1, K = DIM == 3 ? 2 * c[2] - H + i2 : 0;
    bool in = I >= 0 && I < g.npn[0] && J >= 0 && J < g.npn[1];
    if (DIM == 3) in = in && K >= 0 && K < g.npn[2];
    T b = T(0), d = T(-1), s = T(0);
    if (in) {
      const long long q = I + (long long)g.npn[0] * (J + (long long)g.npn[1] * K);
      if (!A.mf[q]) {
        b = A.b[q];
        d = A.dinv[q];
      }
      if (I < g.n[0] && J < g.n[1] && (DIM == 2 || K < g.n[2])) {
        const long long cell = I + (long long)g.n[0] * (J + (long long)g.n[1] * K);
        if (!cell_void(g, cell)) s = A.w ? A.w[cell] : T(1);
      }
    }
    sb[p] = b;
    sd[p] = d;
    sc[p] = s;
  });
}

template <typename T, int DIM>
struct Q1DownK {
  using Args = Q1CycleArgs<T>;
  using B = Box<DIM>;
  using W = Win<DIM, 3>;
  static constexpr int THREADS = 256, MINB = 1;
  static constexpr size_t SMEM = sizeof(T) * 5 * W::N;
  static __device__ __forceinline__ void body(const Args& A, int blk, int) {
    extern __shared__ __align__(16) unsigned char q1_smem[];
    T* sb = reinterpret_cast<T*>(q1_smem);
    T *sd = sb + W::N, *sc = sd + W::N, *s0 = sc + W::N, *s1 = s0 + W::N;
    const Origin<DIM> o(A.gc, blk);
    stage<T, DIM, W, 3>(A, o.c, sb, sd, sc);
    __syncthreads();
    for_nodes<DIM, W, 0, 0>([&](int p, int, int, int) { s0[p] = sd[p] * sb[p] * A.inv_theta; });
    __syncthreads();
    const Geom& g = A.gf;
    for_nodes<DIM, W, 1, 1>([&](int p, int i0, int i1, int i2) {
      T x = T(0);
      if (sd[p] >= T(0)) {
        T dn = A.c2 * sd[p] * (sb[p] - apply<T, DIM, W>(s0, sc, p, A.kc));
        dn += A.c1 * s0[p];
        x = s0[p] + dn;
      }
      s1[p] = x;
      if (i0 >= 3 && i0 < W::X0 - 2 && i1 >= 3 && i1 < W::X1 - 2 && (DIM == 2 || (i2 >= 3 && i2 < W::X2 - 2))) {
        const int I = 2 * o.c[0] - 3 + i0, J = 2 * o.c[1] - 3 + i1, K = DIM == 3 ? 2 * o.c[2] - 3 + i2 : 0;
        if (I < g.npn[0] && J < g.npn[1] && (DIM == 2 || K < g.npn[2]))
          A.x[I + (long long)g.npn[0] * (J + (long long)g.npn[1] * K)] = x;
      }
    });
    __syncthreads();
    for_nodes<DIM, W, 2, 2>([&](int p, int, int, int) {  // s0 <- residual
      s0[p] = sd[p] >= T(0) ? sb[p] - apply<T, DIM, W>(s1, sc, p, A.kc) : T(0);
    });
    __syncthreads();
    const int t = threadIdx.x;
    if (t >= B::C0 * B::C1 * B::C2) return;
    const int a0 = t % B::C0, a1 = (t / B::C0) % B::C1, a2 = DIM == 3 ? t / (B::C0 * B::C1) : 0;
    const int I = o.c[0] + a0, J = o.c[1] + a1, K = o.c[2] + a2;
    if (I >= A.gc.npn[0] || J >= A.gc.npn[1] || (DIM == 3 && K >= A.gc.npn[2])) return;
    const long long q = I + (long long)A.gc.npn[0] * (J + (long long)A.gc.npn[1] * K);
    T acc = T(0);
    if (!A.mc[q]) {
      const int p = (3 + 2 * a0) + W::X0 * (3 + 2 * a1) + (DIM == 3 ? W::XY * (3 + 2 * a2) : 0);
#pragma unroll
      for (int k = (DIM == 3 ? -1 : 0); k < (DIM == 3 ? 2 : 1); ++k)
#pragma unroll
        for (int j = -1; j < 2; ++j)
#pragma unroll
          for (int i = -1; i < 2; ++i) {
            const T w = (i ? T(0.5) : T(1)) * (j ? T(0.5) : T(1)) * (k ? T(0.5) : T(1));
            acc += w * s0[p + i + W::X0 * j + W::XY * k];
          }
    }
    A.bc[q] = acc;
    if (A.sd) {  // the coarse level's smoother from zero (coarse_mode 1)
      const T v = A.sdinv[q] * acc * A.s_inv_theta;
      A.sd[q] = v;
      A.sx[q] = v;
    }
  }
};

template <typename T, int DIM>
struct Q1UpK {
  using Args = Q1CycleArgs<T>;
  using W = Win<DIM, 2>;
  static constexpr int THREADS = 256, MINB = 1;
  static constexpr size_t SMEM = sizeof(T) * 6 * W::N;
  static __device__ __forceinline__ void body(const Args& A, int blk, int) {
    extern __shared__ __align__(16) unsigned char q1_smem[];
    T* sb = reinterpret_cast<T*>(q1_smem);
    T *sd = sb + W::N, *sc = sd + W::N, *s0 = sc + W::N, *s1 = s0 + W::N, *sdir = s1 + W::N;
    const Origin<DIM> o(A.gc, blk);
    const Geom &g = A.gf, &gc = A.gc;
    stage<T, DIM, W, 2>(A, o.c, sb, sd, sc);
    __syncthreads();
    for_nodes<DIM, W, 0, 0>([&](int p, int i0, int i1, int i2) {  // x + P e
      T x = T(0);
      if (sd[p] >= T(0)) {  // a node of the mesh without a mask
        const int I = 2 * o.c[0] - 2 + i0, J = 2 * o.c[1] - 2 + i1, K = DIM == 3 ? 2 * o.c[2] - 2 + i2 : 0;
        T acc = T(0);
#pragma unroll
        for (int k = 0; k < (DIM == 3 ? 2 : 1); ++k) {
          if (k && !(K & 1)) continue;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            if (j && !(J & 1)) continue;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if (i && !(I & 1)) continue;
              const long long cq = ((I >> 1) + i) + (long long)gc.npn[0] * (((J >> 1) + j) + (long long)gc.npn[1] * ((K >> 1) + k));
              if (A.mc[cq]) continue;
              const T w = (I & 1 ? T(0.5) : T(1)) * (J & 1 ? T(0.5) : T(1)) * (K & 1 ? T(0.5) : T(1));
              acc += w * A.e[cq];
            }
          }
        }
        x = A.x[I + (long long)g.npn[0] * (J + (long long)g.npn[1] * K)] + acc;
      }
      s0[p] = x;
    });
    __syncthreads();
    for_nodes<DIM, W, 1, 1>([&](int p, int, int, int) {
      T x = T(0), dn = T(0);
      if (sd[p] >= T(0)) {
        dn = A.inv_theta * sd[p] * (sb[p] - apply<T, DIM, W>(s0, sc, p, A.kc));
        x = s0[p] + dn;
      }
      sdir[p] = dn;
      s1[p] = x;
    });
    __syncthreads();
    for_nodes<DIM, W, 2, 2>([&](int p, int i0, int i1, int i2) {
      const int I = 2 * o.c[0] - 2 + i0, J = 2 * o.c[1] - 2 + i1, K = DIM == 3 ? 2 * o.c[2] - 2 + i2 : 0;
      if (I >= g.npn[0] || J >= g.npn[1] || (DIM == 3 && K >= g.npn[2])) return;
      T x = T(0);
      if (sd[p] >= T(0)) {
        T dn = A.c2 * sd[p] * (sb[p] - apply<T, DIM, W>(s1, sc, p, A.kc));
        dn += A.c1 * sdir[p];
        x = s1[p] + dn;
      }
      A.xout[I + (long long)g.npn[0] * (J + (long long)g.npn[1] * K)] = x;
    });
  }
};

template <typename T, int DIM>
cudaError_t launch_half(int up, const Q1CycleArgs<T>& a, cudaStream_t st) {
  using B = Box<DIM>;
  const long long nblk = (long long)((a.gc.npn[0] + B::C0 - 1) / B::C0) * ((a.gc.npn[1] + B::C1 - 1) / B::C1) *
                         (DIM == 3 ? (a.gc.npn[2] + B::C2 - 1) / B::C2 : 1);
  if (up) return submit<Q1UpK<T, DIM>>(a, nblk, Q1UpK<T, DIM>::SMEM, st);
  return submit<Q1DownK<T, DIM>>(a, nblk, Q1DownK<T, DIM>::SMEM, st);
}
}  // namespace

template <typename T>
cudaError_t launch_q1cycle(int up, const Q1CycleArgs<T>& a, cudaStream_t st) {
  return a.gf.dim == 2 ? launch_half<T, 2>(up, a, st) : launch_half<T, 3>(up, a, st);
}
template cudaError_t launch_q1cycle<float>(int, const Q1CycleArgs<float>&, cudaStream_t);
template cudaError_t launch_q1cycle<double>(int, const Q1CycleArgs<double>&, cudaStream_t);

}  // namespace gs
