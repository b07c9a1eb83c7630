// Launcher of the 3D march kernel (gs_march3d.cuh), one translation unit per precision.
#pragma once
#include "gs_march3d.cuh"
#include "gs_occ.cuh"

namespace gs {
namespace march3 {

// Patch and segment shape for a mesh of `cells` cells.  Patches of px x py <= NT threads covering an axis of n
// cells with overlap 1 number ceil((n - 1) / (px - 1)); px is then shrunk to the least that gives that
// number.  For every patch shape the segments are cut so that the grid is one, two or three waves of the
// resident CTAs (or single layers, where that is less), and the shape with the least estimated time is
// taken: evaluated layers per CTA times the waves, a partly filled wave counting by the share of an
// SM's issue (FP64: pipe) slots that its CTAs take, kShare per CTA.
struct Shape { int px, py, np0, np1, layers, segs; };

inline int cover(int n, int p) { return n <= p ? 1 : (n - 1 + p - 2) / (p - 1); }
inline int shrink(int n, int k) { return k == 1 ? n : (n - 1 + k - 1) / k + 1; }

template <typename T>
Shape choose(const int* cells, int sms, int resident, int max_layers) {
  const int n[3] = {cells[0] + 1, cells[1] + 1, cells[2]};  // the columns of the last node lines included
  const double kShare = sizeof(T) == 4 ? 0.5 : 0.9;
  Shape best{};
  double best_cost = 0.0;
  auto wave = [&](int k) { const double t = k * kShare; return t > 1.0 ? t : 1.0; };
  for (int q = 2; q <= Cfg<T>::NT / 2; ++q) {
    Shape s;
    s.np0 = cover(n[0], q);
    s.px = shrink(n[0], s.np0);
    if (s.px > q || s.px < 1) continue;
    const int pymax = Cfg<T>::NT / s.px;
    if (pymax < 2) continue;
    s.np1 = cover(n[1], pymax);
    s.py = shrink(n[1], s.np1);
    if (s.px * s.py > Cfg<T>::NT) continue;
    const int patches = s.np0 * s.np1;
    for (int w = 1; w <= 2 * resident + 1; ++w) {  // w CTAs per SM, and single layers
      long long segs = w > 2 * resident ? n[2] : (long long)w * sms / patches;
      if (segs < 1) segs = 1;
      s.layers = segs >= n[2] ? 2 : shrink(n[2], (int)segs);
      if (s.layers > max_layers) s.layers = max_layers;
      if (s.layers > n[2]) s.layers = n[2];
      s.segs = cover(n[2], s.layers < 2 ? 2 : s.layers);
      const long long ctas = (long long)patches * s.segs;
      const int per_sm = (int)((ctas + sms - 1) / sms);
      const double cost = (s.layers + 0.5) * ((per_sm / resident) * wave(resident) + (per_sm % resident ? wave(per_sm % resident) : 0.0));
      if (best_cost == 0.0 || cost < best_cost) {
        best_cost = cost;
        best = s;
      }
    }
  }
  return best;
}

template <typename T, int MODE, bool WA, bool WBT, bool WB>
cudaError_t launch(const TileArgs<T>& a, cudaStream_t st) {
  using K = March3K<T, MODE, WA, WBT, WB>;
  constexpr size_t smem = sizeof(T) * (2 * exchange_values<WA || WBT, WB>() + operand_values<MODE, WA || WBT>()) * Cfg<T>::NT;
  const Shape s = choose<T>(a.g.n, sm_count(), ctas_per_sm<K>(smem), a.shape == 1 ? 4 : a.g.n[2]);
  if (s.px < 1) return cudaErrorInvalidValue;
  March3Args<T> m;
  m.t = a;
  m.m = *a.m3;
  m.px = s.px;
  m.py = s.py;
  m.np0 = s.np0;
  m.np1 = s.np1;
  m.layers = s.layers;
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
