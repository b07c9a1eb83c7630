// Transfers between velocity levels: P = Q2 interpolation of the coarse field at the fine nodes (Sec. 4, nested
// meshes); R = P^T.  1D weights: fine 2C <- coarse C (1); fine 4c+1 <- (3/8, 3/4, -1/8) on coarse (2c, 2c+1, 2c+2);
// fine 4c+3 <- (-1/8, 3/4, 3/8).  Constrained fine rows and constrained coarse columns are removed.
//
// Node by node, a coarse node takes up to 25 (2D) or 125 (3D) products with a constraint test and a load each, in FP64
// at 2 operations per SM and clock; applied along one axis after the other the weights take about 4 operations per axis,
// and a test and a load per input node.
//
// Interpolation, and restriction in FP64: a CTA takes one component of a box of nodes, stages the window of input nodes
// that the box touches in shared memory, constrained ones as zero, and applies the weights axis by axis.
//
// Restriction in FP32: a warp takes one component of 29 coarse columns (lanes 2 .. 30; the others hold the halo) and
// marches along the last axis.  A lane loads the two fine nodes at its column of each fine row, takes the neighbours'
// along x by shuffles and keeps the last five rows (3D: planes, each restricted along y first) in registers: about 35
// (2D) or 110 (3D) instructions per coarse node and no barrier; the boxes take 250 and 900, because the window's nodes
// are dealt out to the threads one by one.  Fine mesh 1536^2 FP32: 34 us (boxes 83, node by node 64); 96^3: 95 (226, 215);
// 32^3: 10.6 (16.5, 23).  In FP64 the march repeats each row's restriction along x for the 2.5 coarse lines (3D) that use
// it, on a pipe of 2 operations per SM and clock, and the boxes stay: 32^3 40 us (march 56), 512^2 24 (29).
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
  int seg;  // restriction: coarse rows (3D: planes) a warp marches
};

constexpr int TPB = 256;

template <int DIM>
struct Box;  // coarse nodes of a restriction in boxes, one per thread
template <>
struct Box<2> { static constexpr int C0 = 32, C1 = 8, C2 = 1; };
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

// restriction along one axis to a coarse node of the given parity from the fine nodes at offsets -3, -1, 0, 1, 3
template <typename T>
__device__ __forceinline__ T restrict1(T m3, T m1, T c, T p1, T p3, bool odd) {
  const T in = m1 + p1;
  if (odd) return fma(T(0.75), in, c);
  return fma(T(-0.125), m3 + p3, fma(T(0.375), in, c));
}
// the same from shared memory; s: the coarse node's fine node, st: stride of the axis
template <typename T>
__device__ __forceinline__ T restrict_at(const T* s, int st, bool odd) {
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
struct RestrictMarchK {
  using Args = XferArgs<T>;
  static constexpr int THREADS = TPB, MINB = 1, COLS = 29;
  static __device__ __forceinline__ void body(const Args& a, int blk, int) {
    const Geom &gf = a.gf, &gc = a.gc;
    const int lane = threadIdx.x & 31, strips = (gc.nv[0] + COLS - 1) / COLS, last = gc.nv[DIM - 1];
    const int segs = (last + a.seg - 1) / a.seg, lines = DIM == 3 ? gc.nv[1] : 1;
    long long w = (long long)blk * (TPB / 32) + (threadIdx.x >> 5);
    if (w >= (long long)strips * lines * segs * DIM) return;
    const int I = (int)(w % strips) * COLS + lane - 2;
    w /= strips;
    const int Jc = DIM == 3 ? (int)(w % lines) : 0;
    w /= lines;
    const int L0 = (int)(w % segs) * a.seg, L1 = min(L0 + a.seg, last), comp = (int)(w / segs);
    const T* const v = a.in + comp * gf.Nv + 2 * I;
    const int nf0 = gf.nv[0], nf1 = gf.nv[1];
    const bool in0 = I >= 0 && 2 * I < nf0, in1 = I >= 0 && 2 * I + 1 < nf0;
    const unsigned f = gf.faces;
    const bool con0 = in0 && (((f & 1u) && I == 0) || ((f & 2u) && 2 * I == nf0 - 1));  // 2 I + 1 is on no x face
    const bool oddI = I & 1;
    // fine row (J, K) restricted along x; 0 outside the mesh, constrained nodes as zero
    auto row = [&](int J, int K) {
      bool in = J >= 0 && J < nf1, con = ((f & 4u) && J == 0) || ((f & 8u) && J == nf1 - 1);
      if (DIM == 3) {
        in = in && K >= 0 && K < gf.nv[2];
        con = con || ((f & 16u) && K == 0) || ((f & 32u) && K == gf.nv[2] - 1);
      }
      const long long at = (long long)nf0 * (J + (long long)nf1 * K);
      T c = T(0), p1 = T(0);
      if (gf.vmask) {
        const uint8_t* m = gf.vmask + 2 * I + at;
        if (in && in0 && !m[0]) c = ldg(v + at);
        if (in && in1 && !m[1]) p1 = ldg(v + at + 1);
      } else if (in && !con) {
        if (in0 && !con0) c = ldg(v + at);
        if (in1) p1 = ldg(v + at + 1);
      }
      const T m1 = __shfl_up_sync(0xffffffffu, p1, 1), m3 = __shfl_up_sync(0xffffffffu, p1, 2);
      const T p3 = __shfl_down_sync(0xffffffffu, p1, 1);
      return restrict1(m3, m1, c, p1, p3, oddI);
    };
    // 3D: fine plane K restricted along x and y; 2D: fine row K
    auto line = [&](int K) {
      if (DIM == 2) return row(K, 0);
      const int J = 2 * Jc;
      const bool odd = Jc & 1;
      const T m1 = row(J - 1, K), c = row(J, K), p1 = row(J + 1, K);
      const T m3 = odd ? T(0) : row(J - 3, K), p3 = odd ? T(0) : row(J + 3, K);
      return restrict1(m3, m1, c, p1, p3, odd);
    };
    const bool own = lane >= 2 && lane < 2 + COLS && I < gc.nv[0];
    T m3 = line(2 * L0 - 3), m1 = line(2 * L0 - 1), p1 = line(2 * L0 + 1);
#pragma unroll(DIM == 2 ? 4 : 1)
    for (int L = L0; L < L1; ++L) {
      const T c = line(2 * L), p3 = line(2 * L + 3);
      T r = restrict1(m3, m1, c, p1, p3, L & 1);
      m3 = m1;
      m1 = p1;
      p1 = p3;
      if (!own) continue;
      const int J = DIM == 3 ? Jc : L, K = DIM == 3 ? L : 0;
      const long long node = I + (long long)gc.nv[0] * (J + (long long)gc.nv[1] * K);
      if (vnode_constrained(gc, node, I, J, K)) r = T(0);
      const long long i = comp * gc.Nv + node;
      a.out[i] = r;
      if (a.d) {
        const T s = a.dinv[i] * r * a.inv_theta;
        a.d[i] = s;
        a.x[i] = s;
      }
    }
  }
};

template <typename T, int DIM>
struct RestrictBoxK {
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
      sx[i] = restrict_at(sw + E0 * r + 2 * a0 + 3, 1, a0 & 1);
    }
    __syncthreads();
    const int t = threadIdx.x, a0 = t % B::C0, a1 = (t / B::C0) % B::C1, a2 = DIM == 3 ? t / (B::C0 * B::C1) : 0;
    T v;
    if (DIM == 2) {
      v = restrict_at(sx + a0 + B::C0 * (2 * a1 + 3), B::C0, a1 & 1);
    } else {
      for (int i = t; i < NY; i += TPB) {
        const int b0 = i % B::C0, b1 = (i / B::C0) % B::C1, k = i / (B::C0 * B::C1);
        sy[i] = restrict_at(sx + b0 + B::C0 * (2 * b1 + 3 + E1 * k), B::C0, b1 & 1);
      }
      __syncthreads();
      v = restrict_at(sy + a0 + B::C0 * (a1 + B::C1 * (2 * a2 + 3)), B::C0 * B::C1, a2 & 1);
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
    // 2D: the fine values that the correction is added to are on their way while it is interpolated (bit k of `free`: a
    // free node).  At the end they were one memory latency more in a call of three (FP64, 64^2: 4.5 -> 3.9 us).
    constexpr int NF = F0 * F1 * F2 / TPB, RF = TPB / F0;  // nodes per thread, 2D: RF rows apart
    T fine[DIM == 2 ? NF : 1];
    unsigned free = 0;
    const int f0 = threadIdx.x % F0, f1 = threadIdx.x / F0;
    T* const out = a.out + comp * gf.Nv + o[0] + f0 + (long long)gf.nv[0] * (o[1] + f1);
    if constexpr (DIM == 2) {
#pragma unroll
      for (int k = 0; k < NF; ++k) {
        const int I = o[0] + f0, J = o[1] + f1 + RF * k;
        if (I < gf.nv[0] && J < gf.nv[1] && !vnode_constrained(gf, I + (long long)gf.nv[0] * J, I, J, 0)) {
          free |= 1u << k;
          fine[k] = out[RF * k * (long long)gf.nv[0]];
        }
      }
    }
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
    if constexpr (DIM == 2) {
#pragma unroll
      for (int k = 0; k < NF; ++k)
        if ((free >> k) & 1u) out[RF * k * (long long)gf.nv[0]] = fine[k] + prolong1(sx + f0, F0, f1 + RF * k);
    } else {
      for (int i = threadIdx.x; i < F0 * F1 * F2; i += TPB) {
        const int i0 = i % F0, i1 = (i / F0) % F1, i2 = i / (F0 * F1);
        const int I = o[0] + i0, J = o[1] + i1, K = o[2] + i2;
        if (I >= gf.nv[0] || J >= gf.nv[1] || K >= gf.nv[2]) continue;
        const long long node = I + (long long)gf.nv[0] * (J + (long long)gf.nv[1] * K);
        if (vnode_constrained(gf, node, I, J, K)) continue;
        a.out[comp * gf.Nv + node] += prolong1(sy + i0 + F0 * i1, F0 * F1, i2);
      }
    }
  }
};

template <typename T, int DIM>
cudaError_t restrict_dim(XferArgs<T> a, cudaStream_t st) {
  const int* n = a.gc.nv;
  if constexpr (sizeof(T) == 8) {
    using B = Box<DIM>;
    const long long boxes = (long long)((n[0] + B::C0 - 1) / B::C0) * ((n[1] + B::C1 - 1) / B::C1) *
                            (DIM == 3 ? (n[2] + B::C2 - 1) / B::C2 : 1);
    return submit<RestrictBoxK<T, DIM>>(a, DIM * boxes, RestrictBoxK<T, DIM>::SMEM, st);
  } else {
    // rows a warp marches: as many as leave 16 warps per SM, but at most 16 (the three rows of the halo are then a tenth
    // of those that it loads)
    using K = RestrictMarchK<T, DIM>;
    const long long lines = (long long)((n[0] + K::COLS - 1) / K::COLS) * (DIM == 3 ? n[1] : 1) * DIM;
    const long long seg = lines * n[DIM - 1] / (16 * 152);
    a.seg = (int)(seg < 1 ? 1 : (seg > 16 ? 16 : seg));
    const long long warps = lines * ((n[DIM - 1] + a.seg - 1) / a.seg);
    return submit<K>(a, (warps + TPB / 32 - 1) / (TPB / 32), 0, st);
  }
}
template <typename T, int DIM>
cudaError_t prolong_dim(const XferArgs<T>& a, cudaStream_t st) {
  using K = ProlongAddK<T, DIM>;
  const int* n = a.gf.nv;
  const long long boxes = (long long)((n[0] + K::F0 - 1) / K::F0) * ((n[1] + K::F1 - 1) / K::F1) *
                          (DIM == 3 ? (n[2] + K::F2 - 1) / K::F2 : 1);
  return submit<K>(a, DIM * boxes, K::SMEM, st);
}
}  // namespace

template <typename T>
cudaError_t launch_restrict(const Geom& gf, const Geom& gc, const T* rf, T* rc, cudaStream_t st, const T* dinv,
                            T inv_theta, T* d, T* x) {
  const XferArgs<T> a{gf, gc, rf, rc, dinv, inv_theta, d, x, 0};
  return gf.dim == 2 ? restrict_dim<T, 2>(a, st) : restrict_dim<T, 3>(a, st);
}

template <typename T>
cudaError_t launch_prolong_add(const Geom& gf, const Geom& gc, const T* xc, T* xf, cudaStream_t st) {
  const XferArgs<T> a{gf, gc, xc, xf, nullptr, T(0), nullptr, nullptr, 0};
  return gf.dim == 2 ? prolong_dim<T, 2>(a, st) : prolong_dim<T, 3>(a, st);
}

#define INST(T)                                                                                                    \
  template cudaError_t launch_restrict<T>(const Geom&, const Geom&, const T*, T*, cudaStream_t, const T*, T, T*, T*); \
  template cudaError_t launch_prolong_add<T>(const Geom&, const Geom&, const T*, T*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace gs
