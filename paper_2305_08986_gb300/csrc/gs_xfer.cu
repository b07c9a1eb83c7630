// Transfers between velocity levels: P = Q2 interpolation of the coarse field at the fine nodes (Sec. 4, nested
// meshes); R = P^T.  1D weights: fine 2C <- coarse C (1); fine 4c+1 <- (3/8, 3/4, -1/8) on coarse (2c, 2c+1, 2c+2);
// fine 4c+3 <- (-1/8, 3/4, 3/8).  Constrained fine rows and constrained coarse columns are removed.
//
// A CTA takes one component of a box of nodes: it stages the window of input nodes that the box touches in shared
// memory, constrained ones as zero, and applies the 1D weights along one axis after the other.  Node by node, a
// coarse node took up to 25 (2D) or 125 (3D) products with a constraint test and a load each, in FP64 at 2
// operations per SM and clock; this way it takes about 4 operations per axis, and a test and a load per input node.
// Channel solve 37.0 -> 36.1 ms; FP64 V-cycle of the 1280 x 224 extension mesh 1861 -> 1807 us; batch of six mixed
// solves 49 -> 47 ms.
#include "gs_kernels.h"

namespace gs {
namespace {

template <typename T>
struct XferArgs {
  Geom gf, gc;
  const T* in;
  T* out;
  // start of the coarse level's Chebyshev smoother from zero, fused into the restriction that produces its
  // right-hand side: d = x = dinv * rc * inv_theta (the expression of launch_cheb_init0); d == NULL: none
  const T* dinv;
  T inv_theta;
  T* d;
  T* x;
};

constexpr int TPB = 256;

template <int DIM>
struct Box;
template <>
struct Box<2> { static constexpr int C0 = 32, C1 = 8, C2 = 1; };  // coarse nodes (restriction: one per thread)
template <>
struct Box<3> { static constexpr int C0 = 8, C1 = 8, C2 = 4; };

template <int DIM>
__device__ __forceinline__ void split(const int* ext, int s0, int s1, int s2, int blk, int& comp, int (&o)[3]) {
  comp = blk % DIM;
  blk /= DIM;
  const int n0 = (ext[0] + s0 - 1) / s0, n1 = (ext[1] + s1 - 1) / s1;
  o[0] = blk % n0 * s0;
  o[1] = blk / n0 % n1 * s1;
  o[2] = DIM == 3 ? blk / (n0 * n1) * s2 : 0;
}

// window of E0 x E1 x E2 nodes from node (w0, w1, w2) of one component; 0 outside the mesh and on constrained nodes
template <typename T, int DIM, int E0, int E1, int E2>
__device__ __forceinline__ void stage(const Geom& g, const T* v, int w0, int w1, int w2, T* s) {
  for (int i = threadIdx.x; i < E0 * E1 * E2; i += TPB) {
    const int I = w0 + i % E0, J = w1 + (i / E0) % E1, K = DIM == 3 ? w2 + i / (E0 * E1) : 0;
    bool in = I >= 0 && I < g.nv[0] && J >= 0 && J < g.nv[1];
    if (DIM == 3) in = in && K >= 0 && K < g.nv[2];
    T x = T(0);
    if (in) {
      const long long node = I + (long long)g.nv[0] * (J + (long long)g.nv[1] * K);
      if (!vnode_constrained(g, node, I, J, K)) x = ldg(v + node);
    }
    s[i] = x;
  }
}

// restriction along one axis to a coarse node of the given parity; s: its fine node, st: stride of the axis
template <typename T>
__device__ __forceinline__ T restrict1(const T* s, int st, bool odd) {
  const T in = s[-st] + s[st];
  if (odd) return fma(T(0.75), in, s[0]);
  return fma(T(-0.125), s[-3 * st] + s[3 * st], fma(T(0.375), in, s[0]));
}
// interpolation along one axis to fine offset i of the box; s: the box's first coarse node
template <typename T>
__device__ __forceinline__ T prolong1(const T* s, int st, int i) {
  if (!(i & 1)) return s[(i >> 1) * st];
  const T* c = s + 2 * (i >> 2) * st;
  const bool lo = (i & 3) == 1;  // near the cell's first node
  return fma(T(0.375), lo ? c[0] : c[2 * st], fma(T(0.75), c[st], T(-0.125) * (lo ? c[2 * st] : c[0])));
}

template <typename T, int DIM>
struct RestrictK {
  using Args = XferArgs<T>;
  using B = Box<DIM>;
  static constexpr int THREADS = TPB, MINB = 1;
  // window from fine node 2 o - 3
  static constexpr int E0 = 2 * B::C0 + 5, E1 = 2 * B::C1 + 5, E2 = DIM == 3 ? 2 * B::C2 + 5 : 1;
  static constexpr int NW = E0 * E1 * E2, NX = B::C0 * E1 * E2, NY = DIM == 3 ? B::C0 * B::C1 * E2 : 0;
  static constexpr size_t SMEM = sizeof(T) * (NW + NX + NY);
  static __device__ __forceinline__ void body(const Args& a, int blk, int) {
    extern __shared__ __align__(16) unsigned char xfer_smem[];
    T* sw = reinterpret_cast<T*>(xfer_smem);
    T *sx = sw + NW, *sy = sx + NX;
    const Geom &gf = a.gf, &gc = a.gc;
    int comp, o[3];
    split<DIM>(gc.nv, B::C0, B::C1, B::C2, blk, comp, o);
    stage<T, DIM, E0, E1, E2>(gf, a.in + comp * gf.Nv, 2 * o[0] - 3, 2 * o[1] - 3, 2 * o[2] - 3, sw);
    __syncthreads();
    for (int i = threadIdx.x; i < NX; i += TPB) {  // box origins are even: parities are those of the offsets
      const int a0 = i % B::C0, r = i / B::C0;
      sx[i] = restrict1(sw + E0 * r + 2 * a0 + 3, 1, a0 & 1);
    }
    __syncthreads();
    const int t = threadIdx.x, a0 = t % B::C0, a1 = (t / B::C0) % B::C1, a2 = DIM == 3 ? t / (B::C0 * B::C1) : 0;
    T v;
    if (DIM == 2) {
      v = restrict1(sx + a0 + B::C0 * (2 * a1 + 3), B::C0, a1 & 1);
    } else {
      for (int i = t; i < NY; i += TPB) {
        const int b0 = i % B::C0, b1 = (i / B::C0) % B::C1, k = i / (B::C0 * B::C1);
        sy[i] = restrict1(sx + b0 + B::C0 * (2 * b1 + 3 + E1 * k), B::C0, b1 & 1);
      }
      __syncthreads();
      v = restrict1(sy + a0 + B::C0 * (a1 + B::C1 * (2 * a2 + 3)), B::C0 * B::C1, a2 & 1);
    }
    const int I = o[0] + a0, J = o[1] + a1, K = o[2] + a2;
    if (I >= gc.nv[0] || J >= gc.nv[1] || (DIM == 3 && K >= gc.nv[2])) return;
    const long long node = I + (long long)gc.nv[0] * (J + (long long)gc.nv[1] * K);
    if (vnode_constrained(gc, node, I, J, K)) v = T(0);
    const long long i = comp * gc.Nv + node;
    a.out[i] = v;
    if (a.d) {
      const T s = a.dinv[i] * v * a.inv_theta;
      a.d[i] = s;
      a.x[i] = s;
    }
  }
};

template <typename T, int DIM>
struct ProlongAddK {
  using Args = XferArgs<T>;
  static constexpr int THREADS = TPB, MINB = 1;
  // fine nodes of the box (multiples of 4) and its window of coarse nodes
  static constexpr int F0 = DIM == 2 ? 64 : 16, F1 = 16, F2 = DIM == 3 ? 8 : 1;
  static constexpr int E0 = F0 / 2 + 1, E1 = F1 / 2 + 1, E2 = DIM == 3 ? F2 / 2 + 1 : 1;
  static constexpr int NW = E0 * E1 * E2, NX = F0 * E1 * E2, NY = DIM == 3 ? F0 * F1 * E2 : 0;
  static constexpr size_t SMEM = sizeof(T) * (NW + NX + NY);
  static __device__ __forceinline__ void body(const Args& a, int blk, int) {
    extern __shared__ __align__(16) unsigned char xfer_smem[];
    T* sw = reinterpret_cast<T*>(xfer_smem);
    T *sx = sw + NW, *sy = sx + NX;
    const Geom &gf = a.gf, &gc = a.gc;
    int comp, o[3];
    split<DIM>(gf.nv, F0, F1, F2, blk, comp, o);
    stage<T, DIM, E0, E1, E2>(gc, a.in + comp * gc.Nv, o[0] / 2, o[1] / 2, o[2] / 2, sw);
    __syncthreads();
    for (int i = threadIdx.x; i < NX; i += TPB) sx[i] = prolong1(sw + E0 * (i / F0), 1, i % F0);
    __syncthreads();
    if (DIM == 3) {
      for (int i = threadIdx.x; i < NY; i += TPB) {
        const int i0 = i % F0, i1 = (i / F0) % F1, k = i / (F0 * F1);
        sy[i] = prolong1(sx + i0 + F0 * E1 * k, F0, i1);
      }
      __syncthreads();
    }
    for (int i = threadIdx.x; i < F0 * F1 * F2; i += TPB) {
      const int i0 = i % F0, i1 = (i / F0) % F1, i2 = DIM == 3 ? i / (F0 * F1) : 0;
      const int I = o[0] + i0, J = o[1] + i1, K = o[2] + i2;
      if (I >= gf.nv[0] || J >= gf.nv[1] || (DIM == 3 && K >= gf.nv[2])) continue;
      const long long node = I + (long long)gf.nv[0] * (J + (long long)gf.nv[1] * K);
      if (vnode_constrained(gf, node, I, J, K)) continue;
      a.out[comp * gf.Nv + node] += DIM == 2 ? prolong1(sx + i0, F0, i1) : prolong1(sy + i0 + F0 * i1, F0 * F1, i2);
    }
  }
};

template <template <typename, int> class K, typename T, int DIM>
cudaError_t launch(const XferArgs<T>& a, const int* ext, int s0, int s1, int s2, cudaStream_t st) {
  const long long n = (long long)((ext[0] + s0 - 1) / s0) * ((ext[1] + s1 - 1) / s1) * (DIM == 3 ? (ext[2] + s2 - 1) / s2 : 1);
  return submit<K<T, DIM>>(a, DIM * n, K<T, DIM>::SMEM, st);
}
}  // namespace

template <typename T>
cudaError_t launch_restrict(const Geom& gf, const Geom& gc, const T* rf, T* rc, cudaStream_t st, const T* dinv,
                            T inv_theta, T* d, T* x) {
  const XferArgs<T> a{gf, gc, rf, rc, dinv, inv_theta, d, x};
  if (gf.dim == 2) return launch<RestrictK, T, 2>(a, gc.nv, Box<2>::C0, Box<2>::C1, Box<2>::C2, st);
  return launch<RestrictK, T, 3>(a, gc.nv, Box<3>::C0, Box<3>::C1, Box<3>::C2, st);
}

template <typename T>
cudaError_t launch_prolong_add(const Geom& gf, const Geom& gc, const T* xc, T* xf, cudaStream_t st) {
  const XferArgs<T> a{gf, gc, xc, xf, nullptr, T(0), nullptr, nullptr};
  using P2 = ProlongAddK<T, 2>;
  using P3 = ProlongAddK<T, 3>;
  if (gf.dim == 2) return launch<ProlongAddK, T, 2>(a, gf.nv, P2::F0, P2::F1, P2::F2, st);
  return launch<ProlongAddK, T, 3>(a, gf.nv, P3::F0, P3::F1, P3::F2, st);
}

#define INST(T)                                                                                                    \
  template cudaError_t launch_restrict<T>(const Geom&, const Geom&, const T*, T*, cudaStream_t, const T*, T, T*, T*); \
  template cudaError_t launch_prolong_add<T>(const Geom&, const Geom&, const T*, T*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace gs
