"""Host rule that cuts a 3D mesh into patches and segments (csrc/gs_march3d_shape.h), compiled for the host.

Every shape has to cover the mesh without an empty patch or segment, and on the small meshes that share a launch with
many others the executed work has to stay near the least: a layer of px x py columns takes ceil(px py / 32) warps, so
32 work / cells is the number of lane-layers per cell.  Three or less on cubes of 8 to 32 cells (the overlap of two
evaluated layers per owned one is 2, that of the columns and of partly filled warps up to 1.5)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# meshes with several patches along both axes, whose segments by size have more than four layers (the first in FP64 only)
SEVERAL_PATCHES = [(28, 64, 40), (33, 50, 60)]
DRIVER = r"""
#include <cstdio>
#include "gs_march3d_shape.h"
using namespace gs::march3;
int main() {
  int c[3], res, cap, shared;
  double share;
  while (std::scanf("%d %d %d %d %d %lf %d", c, c + 1, c + 2, &res, &cap, &share, &shared) == 7) {
    static Answers a;
    const Shape s = a.find({{c[0], c[1], c[2]}, 128, 152, res, cap, share, shared != 0});
    const Shape t = choose(c, 128, share, 152, res, cap, shared != 0);
    const bool same = s.px == t.px && s.py == t.py && s.layers == t.layers && s.segs == t.segs;
    std::printf("%d %d %d %d %d %d %lld %lld %d\n", s.px, s.py, s.np0, s.np1, s.layers, s.segs, work(s), a.searches, same);
  }
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    (d / "driver.cpp").write_text(DRIVER)
    exe = str(d / "driver")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2305_08986_gb300", "csrc"),
                    str(d / "driver.cpp"), "-o", exe], check=True)

    def run(queries):
        text = "".join("%d %d %d %d %d %g %d\n" % q for q in queries)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def test_shapes_cover_the_mesh(choose):
    sizes = [1, 2, 3, 5, 8, 13, 31, 64, 65, 127, 200]
    q = [(a, b, c, res, cap, share, shared) for a in sizes for b in sizes for c in sizes
         for res, share in ((1, 0.9), (2, 0.5), (2, 0.9)) for cap in (min(4, c), c)
         for shared in (0, 1)]
    for (a, b, c, _, cap, *_), (px, py, np0, np1, layers, segs, *_) in zip(q, choose(q)):
        assert 2 <= px and 2 <= py and px * py <= 128 and 1 <= layers <= cap
        for n, p, k in ((a + 1, px, np0), (b + 1, py, np1), (c, layers, segs)):
            step = max(p - 1, 1)
            assert (k - 1) * step + p >= n                    # the last one reaches the end
            assert k == 1 or (k - 2) * step + p < n            # and is not empty


def test_small_meshes_execute_little_beyond_their_cells(choose):
    q = [(n, n, n, 2, n, share, 1) for n in (8, 12, 16, 20, 24, 28, 32) for share in (0.5, 0.9)]
    for (n, *_), s in zip(q, choose(q)):
        assert 32 * s[6] <= 3 * n ** 3


def test_answers_are_kept_and_keyed_by_every_argument(choose):
    """One search per distinct query while they fit the list, the searched shape in every answer, also beyond it."""
    q = [(a, 24, c, res, cap, share, shared) for a in (8, 24) for c in (16, 64) for res, cap in ((2, c), (2, 4), (1, c))
         for share, shared in ((0.5, 0), (0.5, 1))]
    rows = choose(q * 5)
    assert len(set(q)) == len(q) <= 32 and rows[-1][7] == len(q)
    rows = choose([(n, n, n, 2, n, 0.5, 0) for n in list(range(8, 60)) * 2])
    assert all(r[8] for r in rows)


def test_larger_meshes_get_other_shapes_by_size_than_with_four_layers(choose):
    """What tests/test_gpu_march_shapes.py relies on."""
    for n in SEVERAL_PATCHES:
        for share in (0.5, 0.9):
            by_size, four = choose([n + (2, n[2], share, 0), n + (2, 4, share, 0)])
            assert by_size[2] > 1 and by_size[3] > 1 and four[4] <= 4
            if share == 0.9 or n != SEVERAL_PATCHES[0]:
                assert by_size[4] > 4
