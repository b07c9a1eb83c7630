// Patch and segment shape of the 3D march kernel (gs_march3d.cuh): host arithmetic only.
//
// Patches of px x py <= `threads` threads covering an axis of n columns with overlap 1 number
// ceil((n - 1) / (px - 1)); px is then shrunk to the least that gives that number.  For every patch shape the segments
// are cut so that the grid is one to 2 * resident CTAs per SM, or as short as they get (two evaluated layers, one owned),
// and the shape with the least estimated time is taken: evaluated layers per CTA times the waves, a partly filled wave
// counting by the share of an SM's issue (FP64: pipe) slots that its CTAs take, `share` per CTA.
//
// Small meshes fit one wave in many shapes of the same estimated time.  A mesh alone on the GPU takes the narrowest
// patches, which spread its loads over the most SMs; in a launch that holds the blocks of many meshes (`shared`) the work
// counts, and the shape that executes the least, warps times layers, is taken.  With the narrowest there as well, 18 of
// a CTA's 128 lanes held a column on 8^3 cells: 256 systems of 8^3 299 -> 79 ms, 128 of 12^3 364 -> 98 ms.
#pragma once

namespace gs {
namespace march3 {

struct Shape { int px, py, np0, np1, layers, segs; };

inline int cover(int n, int p) { return n <= p ? 1 : (n - 1 + p - 2) / (p - 1); }
inline int shrink(int n, int k) { return k == 1 ? n : (n - 1 + k - 1) / k + 1; }

// warps that hold a column times the layers they execute, over the whole grid
inline long long work(const Shape& s) {
  return (long long)s.np0 * s.np1 * s.segs * ((s.px * s.py + 31) / 32) * s.layers;
}

// cells: of the mesh.  max_layers: longest segment allowed (evaluated layers).  shared: with other meshes' blocks.
inline Shape choose(const int* cells, int threads, double share, int sms, int resident, int max_layers, bool shared) {
  const int n[3] = {cells[0] + 1, cells[1] + 1, cells[2]};  // the columns of the last node lines included
  Shape best{};
  double best_cost = 0.0;
  auto wave = [&](int k) { const double t = k * share; return t > 1.0 ? t : 1.0; };
  for (int q = 2; q <= threads / 2; ++q) {
    Shape s;
    s.np0 = cover(n[0], q);
    s.px = shrink(n[0], s.np0);
    if (s.px < q) continue;  // as for q = px
    const int pymax = threads / s.px;
    if (pymax < 2) continue;
    s.np1 = cover(n[1], pymax);
    s.py = shrink(n[1], s.np1);
    if (s.px * s.py > threads) continue;
    const int patches = s.np0 * s.np1;
    for (int w = 1; w <= 2 * resident + 1; ++w) {  // w CTAs per SM, and the shortest segments
      long long segs = w > 2 * resident ? n[2] : (long long)w * sms / patches;
      if (segs < 1) segs = 1;
      s.layers = segs >= n[2] ? 2 : shrink(n[2], (int)segs);
      if (s.layers > max_layers) s.layers = max_layers;
      if (s.layers > n[2]) s.layers = n[2];
      s.segs = cover(n[2], s.layers < 2 ? 2 : s.layers);
      const long long ctas = (long long)patches * s.segs;
      const int per_sm = (int)((ctas + sms - 1) / sms);
      const double cost = (s.layers + 0.5) * ((per_sm / resident) * wave(resident) + (per_sm % resident ? wave(per_sm % resident) : 0.0));
      if (best_cost == 0.0 || cost < best_cost || (shared && cost == best_cost && work(s) < work(best))) {
        best_cost = cost;
        best = s;
      }
    }
  }
  return best;
}

// The same from the last few answers of the calling thread: the search takes 3 to 5 us of a host core, as long as a
// small launch, and depends on its arguments alone.  (One list per kernel and thread; 32 entries hold the levels of
// several contexts.)
struct Query {
  int cells[3], threads, sms, resident, max_layers;
  double share;
  bool shared;
  bool operator==(const Query& o) const {
    return cells[0] == o.cells[0] && cells[1] == o.cells[1] && cells[2] == o.cells[2] && threads == o.threads &&
           sms == o.sms && resident == o.resident && max_layers == o.max_layers && share == o.share && shared == o.shared;
  }
};
struct Answers {
  static constexpr int N = 32;
  Query q[N] = {};
  Shape s[N] = {};
  int next = 0;
  long long searches = 0;
  const Shape& find(const Query& k) {
    for (int i = 0; i < N; ++i)
      if (q[i] == k) return s[i];  // an empty entry has threads = 0 and equals no query
    const int i = next;
    next = (next + 1) % N;
    searches++;
    q[i] = k;
    s[i] = choose(k.cells, k.threads, k.share, k.sms, k.resident, k.max_layers, k.shared);
    return s[i];
  }
};

}  // namespace march3
}  // namespace gs
