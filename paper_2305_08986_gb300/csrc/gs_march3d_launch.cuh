// Launcher of the 3D march kernel (gs_march3d.cuh), one translation unit per precision.
#pragma once
#include "gs_march3d.cuh"
#include "gs_march3d_shape.h"
#include "gs_occ.cuh"

namespace gs {
namespace march3 {

template <typename T, int MODE, bool WA, bool WBT, bool WB>
cudaError_t launch(const TileArgs<T>& a, cudaStream_t st) {
  using K = March3K<T, MODE, WA, WBT, WB>;
  constexpr size_t smem = sizeof(T) * (2 * exchange_values<WA || WBT, WB>() + operand_values<MODE, WA || WBT>()) * Cfg<T>::NT;
  const bool shared = current_recorder() != nullptr;  // recorded into a launch of several meshes
  thread_local Answers shapes;
  const Shape& s = shapes.find({{a.g.n[0], a.g.n[1], a.g.n[2]}, Cfg<T>::NT, sm_count(), ctas_per_sm<K>(smem),
                                a.shape == 1 ? 4 : a.g.n[2], Cfg<T>::SHARE, shared});
  if (s.px < 1) return cudaErrorInvalidValue;
  March3Args<T> m;
  m.t = a;
  m.m = *a.m3;
  m.px = s.px;
  m.py = s.py;
  m.np0 = s.np0;
  m.np1 = s.np1;
  m.layers = s.layers;
  m.skip = shared;
  return submit<K>(m, (long long)s.np0 * s.np1 * s.segs, smem, st);
}

template <typename T>
cudaError_t dispatch(int mode, int ops, const TileArgs<T>& a, cudaStream_t st) {
  if (ops == OPS_A) {
    if (mode == TILE_APPLY) return launch<T, TILE_APPLY, true, false, false>(a, st);
    if (mode == TILE_RESID) return launch<T, TILE_RESID, true, false, false>(a, st);
    return launch<T, TILE_CHEB, true, false, false>(a, st);
  }
  if (mode == TILE_CHEB) return cudaErrorInvalidValue;
  const bool ap = mode == TILE_APPLY;
  switch (ops) {
    case OPS_BT: return ap ? launch<T, TILE_APPLY, false, true, false>(a, st) : launch<T, TILE_RESID, false, true, false>(a, st);
    case OPS_B: return ap ? launch<T, TILE_APPLY, false, false, true>(a, st) : launch<T, TILE_RESID, false, false, true>(a, st);
    case OPS_A | OPS_BT | OPS_B:
      return ap ? launch<T, TILE_APPLY, true, true, true>(a, st) : launch<T, TILE_RESID, true, true, true>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace march3
}  // namespace gs
