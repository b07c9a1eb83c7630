"""Coefficients of the cell operators in Legendre modes (csrc/gs_modal_coef.h), compiled for the host, against exact
rationals: every FP64 coefficient is the nearest double, every FP32 one the nearest float, and the FP32 viscous
coefficients of 2D meshes are within 2^-47 of the exact value together with their remainders (24 bits each)."""
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRIVER = r"""
#include <cstdio>
#include "gs_modal_coef.h"
using namespace gs;
template <typename T, class M>
void print(const M& m) {
  const T* p = reinterpret_cast<const T*>(&m);
  for (size_t i = 0; i < sizeof(M) / sizeof(T); ++i) std::printf("%a ", (double)p[i]);
  std::printf("\n");
}
int main() {
  int dim;
  double h[3], alpha;
  while (std::scanf("%d %la %la %la %la", &dim, h, h + 1, h + 2, &alpha) == 5) {
    if (dim == 2) { print<double>(make_modal2<double>(h, alpha)); print<float>(make_modal2<float>(h, alpha)); }
    else { print<double>(make_modal<double>(h, alpha)); print<float>(make_modal<float>(h, alpha)); }
  }
}
"""
M, K, W = [Fr(1, 36), Fr(1, 12), Fr(1, 45)], [Fr(0), Fr(1), Fr(4, 3)], [1, 1, 2]
MESHES = [(2, (2.5 / 1280, 0.41 / 210), 1000.0), (2, (1 / 37, 1 / 41), 7.3), (2, (0.5 / 3, 0.75 / 1000), 0.0),
          (3, (1 / 37, 1 / 29, 1 / 41), 100.0), (3, (1 / 13, 1 / 14, 1 / 5), 3.7), (3, (1 / 64,) * 3, 0.0),
          (3, (0.001, 7.0, 0.3), 1e6)]


def _exact(dim, h, alpha):
    """{name: (exact rationals in the order of the struct)}"""
    h = [Fr(x) for x in h]
    modes = [(i, j, k) for k in range(3 if dim == 3 else 1) for j in range(3) for i in range(3)]
    prod = lambda it: Fr(1) * np.prod([Fr(x) for x in it], initial=Fr(1))
    dm = {}
    for ix in modes:
        n1, n2 = sum(q == 1 for q in ix[:dim]), sum(q == 2 for q in ix[:dim])
        dm[(n1, n2)] = Fr(alpha) * prod(h) * prod(M[q] * W[q] for q in ix[:dim])
    order = [(0, 0), (1, 0), (2, 0), (3, 0), (0, 1), (1, 1), (2, 1), (0, 2), (1, 2), (0, 3)] if dim == 3 else \
            [(0, 0), (1, 0), (0, 1), (2, 0), (1, 1), (0, 2)]

    def visc(c, ix):
        return sum((2 if b == c else 1) * K[ix[b]] / h[b] ** 2 * prod(M[ix[e]] for e in range(dim) if e != b)
                   for b in range(dim)) * prod(h) * prod(W[q] for q in ix[:dim])
    dk = [[visc(c, ix) for ix in modes] for c in range(dim)]
    ga = [prod(h[b] / 12 for b in range(dim) if b != a) for a in range(dim)]
    div = [g / 2 for g in ga] + [g / 3 for g in ga] + [2 * g / 3 for g in ga]
    if dim == 3:
        dc = [h[p] * M[k] * W[k] / 36 for p in range(3) for k in range(3)]
        return [dm[o] for o in order] + dk[0] + dk[1] + dk[2] + dc + div, None
    kk = [dk[c][q] for q in range(9) for c in range(2)]
    return [dm[o] for o in order] + kk, (kk, div)


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("coef")
    (d / "driver.cpp").write_text(DRIVER)
    exe = str(d / "driver")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2305_08986_gb300", "csrc"),
                    str(d / "driver.cpp"), "-o", exe], check=True)
    text = "".join("%d %s %s %s %s\n" % (dim, float(h[0]).hex(), float(h[1]).hex(),
                                         float(h[2] if dim == 3 else 1).hex(), float(a).hex()) for dim, h, a in MESHES)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    return [[float.fromhex(q) for q in line.split()] for line in out.splitlines()]


def _nearest(got, exact, dtype):
    g = dtype(got)
    assert float(g) == got
    lo, hi = (Fr(float(np.nextafter(g, dtype(s) * dtype(np.inf)))) for s in (-1, 1))
    e = abs(Fr(got) - exact)
    return e <= abs(lo - exact) and e <= abs(hi - exact)


@pytest.mark.parametrize("k", range(len(MESHES)))
@pytest.mark.parametrize("row,dtype", [(0, np.float64), (1, np.float32)])
def test_coefficients_are_rounded_once(rows, k, row, dtype):
    dim, h, alpha = MESHES[k]
    got = rows[2 * k + row]
    exact, rest = _exact(dim, h, alpha)
    for g, e in zip(got, exact):
        assert _nearest(g, e, dtype), (g, float(e))
    if rest is None:
        assert len(got) == len(exact)
        return
    kk, div = rest
    low = got[len(exact):len(exact) + 18]
    for hi, lo, e in zip(got[6:24], low, kk):
        assert abs(Fr(hi) + Fr(lo) - e) <= abs(e) / 2 ** (47 if row else 100)
    for g, e in zip(got[len(exact) + 18:], div):
        assert _nearest(g, e, dtype)
    assert len(got) == len(exact) + 18 + 6
