// 3D kernel for the blocks A, B^T and B of the saddle operator (Eq. "stokes-discrete-block") on
// Cartesian Q2-Q1 hexahedra: y = K x, y = b - K x and the fused Chebyshev step, in the cells' Legendre
// modes (gs_modal.cuh).
//
// Work decomposition.  A CTA evaluates a patch of px x py cells of the (x, y) plane, one thread per cell
// column, and marches it up a segment of cell layers.  Patches and segments overlap by one cell: the
// first cell along an axis (except at the mesh boundary) is evaluated for its contributions only, so
// every node is written by exactly one thread, without atomics.  Along z a thread keeps in registers
// the (x, y)-modes of its top node plane, which is the bottom plane of its next cell, and the output
// modes that its cell leaves on that plane; per layer it reads two node planes, transforms 2 x 9 node
// lines along x and y and 9 along z, and completes two node planes.  Along x and y a cell leaves its
// values on the right and top node lines (5 per plane and component) in shared memory, where the
// neighbour that owns the node picks them up behind one barrier per layer (two buffers).  Every node
// sums its cells as ((own + left) + below) + below-left, each term already holding the layer below,
// so the result does not depend on the patch or segment shape.
//
// The patches cover one more column than there are cells along x and y: its threads evaluate nothing and write the
// mesh's last node lines from their neighbours' contributions, like any other node.  Written by the last cells
// instead, those lines took a serial chain of loads and stores in a few CTAs, which the whole launch waited for
// (SMs busy 61 % of the time; 64^3, 4 Chebyshev steps, FP32: 453 -> 318 us; FP64 saddle 37 x 29 x 41: 225 -> 210 us).
//
// Nothing is staged: the 27 + 27 node values a thread reads per layer are shared with its neighbours through L1.  The
// overlap, the columns of the last node lines and partly filled patches cost 1.4 lane-layers per cell of the mesh on 64^3
// and 1.9 on 37 x 29 x 41 (FP64: 4 x 30 columns, 5 layers, 130 CTAs).
#pragma once
#include "gs_modal.cuh"

namespace gs {

template <typename T>
struct March3Args {
  TileArgs<T> t;
  ModalCoef<T> m;
  int px, py;      // threads (cells) of a patch along x and y
  int np0, np1;    // patches along x and y
  int layers;      // evaluated cell layers per segment
  int skip;        // warps without a column only keep the barriers
};

namespace march3 {
template <typename T>
struct Cfg {
  static constexpr int NT = 128;   // threads per CTA
  static constexpr int MINB = 2;   // CTAs per SM: 8 warps at 255 registers; 12 at 168 spilled (4 Chebyshev steps, 64^3: 23 % slower)
  static constexpr double SHARE = sizeof(T) == 4 ? 0.5 : 0.9;  // of an SM's issue (FP64: pipe) slots a CTA takes
};

// values per thread: exchanged with the neighbours per layer; epilogue operands of the 8 nodes a cell owns
template <bool WU, bool WB>
constexpr int exchange_values() { return (WU ? 30 : 0) + (WB ? 3 : 0); }
template <int MODE, bool WU>
constexpr int operand_values() { return !WU || MODE == TILE_APPLY ? 0 : (MODE == TILE_CHEB ? 96 : 24); }

// Element `off` bytes after a base that is uniform in the CTA (32-bit offsets within a node plane).
template <typename T>
__device__ __forceinline__ T* at(T* base, unsigned off) {
  return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(base) + off);
}
// Asynchronous copies of an element of a node row and, with `two`, its successor into value slots of this thread.
template <typename T, int SLOT>
__device__ __forceinline__ void cp_async2(unsigned smem, const T* gmem, bool two) {
  constexpr int S = (int)sizeof(T);
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n cp.async.ca.shared.global [%0], [%1], %4;\n"
               " @p cp.async.ca.shared.global [%0+%3], [%1+%4], %4;\n}\n" ::"r"(smem), "l"(gmem), "r"((unsigned)two),
               "n"(SLOT * S), "n"(S) : "memory");
}

template <typename T, int MODE, bool WA, bool WBT, bool WB>
__device__ __forceinline__ void body(const March3Args<T>& M, int bid) {
  constexpr bool NEED_U = WA || WB, WU = WA || WBT;
  constexpr int NT = Cfg<T>::NT, NX = exchange_values<WU, WB>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sx = reinterpret_cast<T*>(smem_raw);  // [buffer][value][thread]
  T* so = sx + 2 * NX * NT + threadIdx.x;   // [operand value][thread]
  const unsigned so32 = (unsigned)__cvta_generic_to_shared(so);
  constexpr bool EB = WU && MODE != TILE_APPLY, ED = WU && MODE == TILE_CHEB;
  const TileArgs<T>& A = M.t;
  const Geom& g = A.g;
  const bool raw = A.raw != 0;
  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int nv0 = g.nv[0], np0 = g.npn[0];
  const long long Nv = g.Nv, vplane = (long long)nv0 * g.nv[1], pplane = (long long)np0 * g.npn[1];
  const int tid = threadIdx.x, PX = M.px;
  const int p0 = bid % M.np0, p1 = (bid / M.np0) % M.np1, sg = bid / (M.np0 * M.np1);
  const int tx = tid % PX, ty = tid / PX;
  const int c0 = p0 * (PX - 1) + tx, c1 = p1 * (M.py - 1) + ty;
  const bool here = ty < M.py && c0 <= n0 && c1 <= n1;  // c0 = n0, c1 = n1: the mesh's last node lines
  const bool in = here && c0 < n0 && c1 < n1;           // a cell of the mesh
  const bool left = tx > 0, below = ty > 0;       // neighbours in the patch
  const bool own = here && (left || p0 == 0) && (below || p1 == 0);
  const bool two0 = c0 < n0, two1 = c1 < n1;      // node columns / rows owned besides the first
  const int zs = sg * (M.layers - 1), ze = min(n2, zs + M.layers);
  const int zend = ze == n2 ? n2 + 1 : ze;  // one extra pass after the mesh's last layer completes the top node plane
  // In a launch with other meshes' blocks a warp without a column (a patch may hold fewer than 128) only keeps the
  // barriers: its arithmetic would take their issue slots (64 systems of 16^3: 127 -> 117 ms).  Alone it runs along, and
  // its instruction fetches serve the others: 4 Chebyshev steps on 8^3, FP32, take 32 us, and 39 us without it.
  if (M.skip && !__any_sync(0xffffffffu, here)) {
    for (int c2 = zs; c2 < zend; ++c2) __syncthreads();
    return;
  }
  // byte offsets in a plane (planes are below 4 GB): the cell's three node rows (threads without a cell read some
  // cell of the mesh), and the two node rows a thread writes
  const long long vcol = 2 * min(c0, n0) + (long long)nv0 * (2 * min(c1, n1));
  unsigned orow[3], wrow[2];
  {
    const long long rcol = 2 * min(c0, n0 - 1) + (long long)nv0 * (2 * min(c1, n1 - 1));
#pragma unroll
    for (int j = 0; j < 3; ++j) orow[j] = (unsigned)((rcol + (long long)nv0 * j) * (long long)sizeof(T));
#pragma unroll
    for (int j = 0; j < 2; ++j) wrow[j] = (unsigned)((vcol + (long long)nv0 * j) * (long long)sizeof(T));
  }
  const long long pcol = c0 + (long long)np0 * c1;

  // constrained local nodes of a node plane (bit la + 3 lb)
  unsigned fxy = 0;
  if ((g.faces & 1u) && c0 == 0) fxy |= 0x049u;
  if ((g.faces & 2u) && c0 >= n0 - 1) fxy |= c0 == n0 ? 0x049u : 0x124u;
  if ((g.faces & 4u) && c1 == 0) fxy |= 0x007u;
  if ((g.faces & 8u) && c1 >= n1 - 1) fxy |= c1 == n1 ? 0x007u : 0x1C0u;
  auto plane_mask = [&](int K) -> unsigned {
    if (!here || raw) return 0u;
    if (g.vmask) {
      unsigned m = 0;
      const uint8_t* vm = g.vmask + vplane * K + vcol;
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if ((two0 || q % 3 == 0) && (two1 || q / 3 == 0)) m |= vm[q % 3 + nv0 * (q / 3)] ? 1u << q : 0u;
      return m;
    }
    if (((g.faces & 16u) && K == 0) || ((g.faces & 32u) && K == 2 * n2)) return 0x1FFu;
    return fxy;
  };
  // the column's nodes on node plane K, constrained columns entering as zero
  auto load_plane = [&](int K, unsigned pm, T (&v)[3][9]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* base = A.xu + (c * Nv + vplane * K);
#pragma unroll
      for (int q = 0; q < 9; ++q) v[c][q] = ldg(at(base, orow[q / 3]) + q % 3);
    }
    if (__any_sync(0xffffffffu, pm != 0)) {
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if ((pm >> q) & 1u) v[0][q] = v[1][q] = v[2][q] = T(0);
    }
  };
  auto load_pplane = [&](int K, T (&b)[4]) {
    T p[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long i = pcol + pplane * K + (q & 1) + np0 * (q >> 1);
      p[q] = in && !(!raw && pnode_constrained(g, i)) ? A.xp[i] : T(0);
    }
    const T s0 = p[0] + p[1], d0 = p[1] - p[0], s1 = p[2] + p[3], d1 = p[3] - p[2];
    b[0] = s0 + s1;
    b[1] = d0 + d1;
    b[2] = s1 - s0;
    b[3] = d1 - d0;
  };

  T cin[3][9], cout[3][9];  // bottom plane: input modes, output modes left by the layer below
  T pin[4], pout[4];
  unsigned pmb = plane_mask(2 * zs);
  if (NEED_U) load_plane(2 * zs, pmb, cin);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (NEED_U) plane_to_modes(cin[c]);
#pragma unroll
    for (int q = 0; q < 9; ++q) cout[c][q] = T(0);
  }
  if (WBT) load_pplane(zs, pin);
#pragma unroll
  for (int q = 0; q < 4; ++q) pout[q] = T(0);

  // per-cell data of the column's cell in layer k (loaded one layer ahead)
  struct CellData {
    T eta, alpha;
    bool active;  // in the mesh and no obstacle
  };
  auto load_cell = [&](int k) {
    CellData d{T(0), T(1), in};
    if (in) {
      const long long i = c0 + (long long)n0 * (c1 + (long long)n1 * k);
      if (WA) d.eta = A.eta[i];
      if (WA && A.alpha) d.alpha = A.alpha[i];
      if (cell_void(g, i)) d.active = false;
    }
    return d;
  };
  CellData next = load_cell(zs);
  T xm[3][9], xt[3][9];  // the layer's middle and top node planes
  unsigned pmm = plane_mask(2 * zs + 1), pmt = plane_mask(2 * zs + 2);

#pragma unroll 1
  for (int c2 = zs; c2 < zend; ++c2) {
    T bot[3][9], mid[3][9], pb[4];
    const unsigned cmm = pmm, cmt = pmt;  // this layer's masks
    const bool writes = own && !(c2 == zs && zs > 0);  // not the layer below the segment's own
    // Epilogue operands of the eight nodes an owned cell writes: copied to this thread's own slots of
    // shared memory while the layer is computed (no registers held, no barrier needed).
    if (EB && writes) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int j = 0; j < 4; ++j) {  // node rows: plane j >> 1, row j & 1
          if (j >= 2 && c2 == n2) break;
          if ((j & 1) && !two1) continue;
          const long long base = c * Nv + vplane * (2 * c2 + (j >> 1));
          const unsigned o = so32 + (c * 8 + 2 * j) * NT * (unsigned)sizeof(T);
          cp_async2<T, NT>(o, at(A.bu + base, wrow[j & 1]), two0);
          if (ED) {
            cp_async2<T, NT>(o + 24 * NT * sizeof(T), at(A.dinv + base, wrow[j & 1]), two0);
            cp_async2<T, NT>(o + 72 * NT * sizeof(T), at(A.xu + base, wrow[j & 1]), two0);
            if (A.use_d) cp_async2<T, NT>(o + 48 * NT * sizeof(T), at((const T*)A.d + base, wrow[j & 1]), two0);
          }
        }
    }
    asm volatile("cp.async.commit_group;\n" ::);
    if (c2 < n2) {
      const CellData cell = next;
      const bool idle = __any_sync(0xffffffffu, !cell.active);
      if (c2 + 1 < ze) next = load_cell(c2 + 1);
      T a[3][27], r[3][27];
      if (NEED_U) {
        load_plane(2 * c2 + 1, cmm, xm);
        load_plane(2 * c2 + 2, cmt, xt);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          plane_to_modes(xm[c]);
          plane_to_modes(xt[c]);
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            to_modes(cin[c][q], xm[c][q], xt[c][q], a[c][q], a[c][q + 9], a[c][q + 18]);
            cin[c][q] = xt[c][q];
          }
        }
      }
      if (c2 + 1 < ze) {
        pmm = plane_mask(2 * c2 + 3);
        pmt = plane_mask(2 * c2 + 4);
      }
      if (WA) {
        T mass[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) mass[i] = cell.alpha * M.m.dm[i];
        modal_A3(a, r, cell.eta * A.c.eta_scale, mass, M.m);
      } else if (WU) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int q = 0; q < 27; ++q) r[c][q] = T(0);
      }
      if (WBT) {
        T tp[4], beta[8];
        load_pplane(c2 + 1, tp);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          beta[q] = pin[q] + tp[q];
          beta[q + 4] = tp[q] - pin[q];
          pin[q] = tp[q];
        }
        modal_BT3(beta, r, M.m);
      }
      if (WB) {
        T gm[8];
        modal_B3(a, gm, M.m);
        if (idle && !cell.active) {
#pragma unroll
          for (int q = 0; q < 8; ++q) gm[q] = T(0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          pb[q] = (gm[q] - gm[q + 4]) + pout[q];
          pout[q] = gm[q] + gm[q + 4];
        }
      }
      if (WU) {
        if (idle && !cell.active) {  // obstacle cells contribute nothing (in raw mode their nodes may hold values)
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int q = 0; q < 27; ++q) r[c][q] = T(0);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int q = 0; q < 9; ++q) {
            T y0, y2;
            from_modes(r[c][q], r[c][q + 9], r[c][q + 18], y0, mid[c][q], y2);
            bot[c][q] = y0 + cout[c][q];
            cout[c][q] = y2;
          }
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          bot[c][q] = cout[c][q];
          mid[c][q] = T(0);
        }
#pragma unroll
      for (int q = 0; q < 4; ++q) pb[q] = pout[q];
    }

    // nodal values of the two planes; those on the right and top node lines go to the neighbours
    T* slot = sx + ((c2 - zs) & 1) * (NX * NT) + tid;
    if (WU) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        plane_from_modes(bot[c]);
        plane_from_modes(mid[c]);
        constexpr int ex[5] = {2, 5, 8, 6, 7};
#pragma unroll
        for (int e = 0; e < 5; ++e) {
          slot[(c * 5 + e) * NT] = bot[c][ex[e]];
          slot[(15 + c * 5 + e) * NT] = mid[c][ex[e]];
        }
      }
    }
    T pv[4];
    if (WB) {
      const T s0 = pb[0] - pb[2], s1 = pb[0] + pb[2], d0 = pb[1] - pb[3], d1 = pb[1] + pb[3];
      pv[0] = s0 - d0;
      pv[1] = s0 + d0;
      pv[2] = s1 - d1;
      pv[3] = s1 + d1;
#pragma unroll
      for (int e = 0; e < 3; ++e) slot[(NX - 3 + e) * NT] = pv[e + 1];
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    if (writes) {
      if (WU) {
#pragma unroll
        for (int pl = 0; pl < 2; ++pl) {
          if (pl == 1 && c2 == n2) break;
          const unsigned pm = pl == 0 ? pmb : cmm;
          T out[3][4], od[3][4], xin[3][4];
          if (!ED && WA && pm) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if ((two0 || !(q & 1)) && (two1 || q < 2))
                  xin[c][q] = ldg(at(A.xu + (c * Nv + vplane * (2 * c2 + pl)), wrow[q >> 1]) + (q & 1));
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            T (&v)[9] = pl == 0 ? bot[c] : mid[c];
            const T* s = slot + (pl * 15 + c * 5) * NT;
            if (left) {
              v[0] += s[-1];
              v[3] += s[NT - 1];
            }
            if (below) {
              v[0] += s[3 * NT - PX];
              v[1] += s[4 * NT - PX];
            }
            if (left && below) v[0] += s[2 * NT - PX - 1];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int lq = (q & 1) + 3 * (q >> 1);
              const bool con = (pm >> lq) & 1u;
              const T* o = so + (c * 8 + pl * 4 + q) * NT;
              if (ED) xin[c][q] = o[72 * NT];
              const T ax = con ? (WA ? xin[c][q] : T(0)) : v[lq];
              if (MODE == TILE_APPLY) {
                out[c][q] = ax;
              } else if (MODE == TILE_RESID) {
                out[c][q] = o[0] - ax;
              } else {
                T dn = A.c2 * o[24 * NT] * (o[0] - ax);
                if (A.use_d) dn += A.c1 * o[48 * NT];
                od[c][q] = dn;
                out[c][q] = xin[c][q] + dn;
              }
            }
          }
          T* y = ED ? A.xout : A.yu;
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if ((!two0 && (q & 1)) || (!two1 && q >= 2)) continue;
              const long long base = c * Nv + vplane * (2 * c2 + pl);
              at(y + base, wrow[q >> 1])[q & 1] = out[c][q];
              if (ED) at(A.d + base, wrow[q >> 1])[q & 1] = od[c][q];
            }
        }
      }
      if (WB) {
        const T* s = slot + (NX - 3) * NT;
        if (left) pv[0] += s[-1];
        if (below) pv[0] += s[NT - PX];
        if (left && below) pv[0] += s[2 * NT - PX - 1];
        const long long i = pcol + pplane * c2;
        const bool con = !raw && pnode_constrained(g, i);
        const T bx = con ? (WBT ? A.xp[i] : T(0)) : pv[0];
        A.yp[i] = MODE == TILE_RESID ? A.bp[i] - bx : bx;
      }
    }
    pmb = cmt;
  }
}

template <typename T, int MODE, bool WA, bool WBT, bool WB>
struct March3K {
  using Args = March3Args<T>;
  static constexpr int THREADS = Cfg<T>::NT, MINB = Cfg<T>::MINB;
  static __device__ __forceinline__ void body(const Args& a, int blk, int) { march3::body<T, MODE, WA, WBT, WB>(a, blk); }
};

}  // namespace march3
}  // namespace gs
