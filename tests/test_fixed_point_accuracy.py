"""The fixed-point element algebra (csrc/fixed.cuh, compiled here for the CPU)
against exact rational arithmetic where entries of one element differ in size:
edges and faces of a graded mesh, rows of Q z over several decades."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from tests.test_fixed_point import exact

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "fixed.cuh"
extern "C" int gram(const double* e, double* G) {
  int64_t g[6];
  int kg;
  if (!fx::geometry(reinterpret_cast<const double(*)[3]>(e), g, kg)) return 0;
  for (int i = 0; i < 6; ++i) G[i] = fx::to_double(g[i], kg);
  return 1;
}
extern "C" int kernel(const double* e, double a, double c20, double rdet, double* Q) {
  int64_t g[6];
  int kg;
  return fx::geometry(reinterpret_cast<const double(*)[3]>(e), g, kg) &&
         fx::face_kernel(g, kg, a, c20, rdet, [](double x) { return 1.0 / x; }, Q);
}
extern "C" int product(const double* Q, const double* z, double* e, unsigned* small) {
  return fx::product4(Q, z, e, small);
}
"""
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxa")
    src, so = d / "fx.cpp", d / "libfx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2509_11133_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def ptr(x):
    return x.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def graded(kind, inv, rng):
    """Edge vectors of a jittered element with one feature of size 1/inv, turned
    at random; differences of coordinates."""
    base = np.array([[[0, 0, 0], [1, 0, 0], [1, 1, 0], [1, 1, 1]], [[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]]],
                    float)[rng.integers(2)]
    P = base + 0.15 * rng.uniform(-1, 1, (4, 3))
    if kind == "one short edge":
        P[1] = P[0] + (P[1] - P[0]) / inv
    elif kind == "two short edges":
        P[1:3] = P[0] + (P[1:3] - P[0]) / inv
    elif kind == "flat":
        P[:, 2] /= inv
    elif kind == "needle":
        P[:, :2] /= inv
    R, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    P = rng.uniform(0, 1, 3) + 10.0 ** rng.uniform(-3, 0) * P @ R.T
    return np.ascontiguousarray(P[1:] - P[0])


@pytest.mark.parametrize("kind", ["one short edge", "two short edges", "flat", "needle"])
@pytest.mark.parametrize("inv", [1, 3, 8, 12, 24])
def test_gram_entries(lib, kind, inv):
    """Every entry of G_e to 2.05 x 2^-53 of |e_i||e_j|: the rounding to fp64, one
    unit; half a unit of the fixed scale, at most one on a diagonal entry 2^-7 of
    the largest and less on the others; and 0.31 for the components of an edge
    that are cut at 2^-60 of the largest (2 sqrt(3) 2^3.5 2^-60 for the shortest
    edge of 2^-3.5)."""
    rng = np.random.default_rng(inv)
    taken = 0
    for _ in range(200):
        e = graded(kind, inv, rng)
        G = np.zeros(6)
        if not lib.gram(ptr(e), ptr(G)):
            continue
        taken += 1
        E = [[Fraction(float(x)) for x in r] for r in e]
        ij = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
        ref = {p: sum(x * y for x, y in zip(E[p[0]], E[p[1]])) for p in ij}
        for n, (i, j) in enumerate(ij):
            scale = float(ref[i, i] * ref[j, j]) ** 0.5
            assert abs(float(Fraction(float(G[n])) - ref[i, j])) <= 2.05 * U * scale
    assert taken >= 150 or inv > 4  # the rest are left to fp64


# e (three edges), a, c/20, 1/|det E|: elements whose Q was off by 9.3 to 10.7 x
# 2^-53 of its largest entry without the low products of Y = adj(M) G T0^-1
HARD = """
0x1.9561ba82a07e7p-2 0x1.dae5897fb548p-5 0x1.c9ea7531d9978p-3 0x1.972cc0cfb6618p-4 0x1.8f8c2a2304d8ap-2 0x1.b6e17524bbdf8p-3 0x1.21d3571bec14p-3 0x1.0f883f9ae7818p-4 0x1.fba1cbb304d08p-2 0x1.cdf15f3789537p-2 0x1.a94e01d67dabfp-13 0x1.0f48cc2612c6ap+4
0x1.9cc8aa31521ap-7 0x1.897ae9b8b18p-10 0x1.73f3c1fb74p-13 0x1.991b9c2b8e2cp-6 0x1.e589b4d28fd6p-6 0x1.8a540e77bf0bp-9 0x1.b092db12e15cp-6 0x1.cc52f8cf5915p-6 0x1.803bb4bfb7f9ap-6 0x1.d44ec52224243p+3 0x1.42cd70f8a22bp-7 0x1.1a67fdc4e4b79p+17
0x1.2304dfef43cp-14 0x1.02528414414p-11 0x1.372e4ed29p-15 -0x1.8b8ebbc280bp-13 0x1.4cb8e87081p-9 0x1.868123ee093p-9 0x1.15ca3ec0372ap-10 0x1.98b27ddaf42p-9 0x1.277a4a81a27p-9 0x1.b434e1085a4edp-2 0x1.9257e876084p-9 0x1.5597024a8d2e3p+29
0x1.0f2c915fd3418p-5 -0x1.0909b1505f61p-5 0x1.91a6e76812p-12 0x1.eb0a1da33048p-9 -0x1.f09dcc3da2dep-6 0x1.bbf798ad3b48p-9 0x1.26ba5814858cp-8 -0x1.2125055313edp-5 0x1.2f2029f088bdp-6 0x1.cee20a90a00bdp-4 0x1.49f261455c3c8p-6 0x1.2fdf960a4a796p+16
0x1.5da048293224p-7 0x1.000daa255228p-8 -0x1.25762759958p-9 0x1.114646b2b0fp-7 0x1.61d66d1003dp-9 -0x1.27b72f33448p-12 0x1.44b7f2d595cp-8 0x1.18bd77e1dbfp-9 -0x1.bf75c0f214p-12 0x1.f468f18deee99p-3 0x1.a03d7881631a4p-8 0x1.00203304e30a7p+27
-0x1.201252cf296ap-4 -0x1.02c8e6225254p-6 0x1.21ca8a0adbb1p-6 -0x1.fe0f695b1c7ap-5 -0x1.1aeaa0a41954ap-3 -0x1.c1b8fad895c4p-8 -0x1.ae79deb360b1p-5 -0x1.452601dc3ff36p-3 0x1.e179c2bea91dp-5 0x1.74422163603dp+0 0x1.05de68724f06fp-11 0x1.8c7368072b8acp+10
"""


@pytest.mark.parametrize("row", HARD.split("\n")[1:-1], ids=range(6))
def test_condensation_of_hard_elements(lib, row):
    """Q to 8 x 2^-53 of its largest entry: the scalar's fp64 operations (five:
    the constant, two products, a reciprocal, det M's conversion), the rounding to
    fp64, and less than one each for det M (2^-54.7) and for the sums."""
    v = np.array([float.fromhex(x) for x in row.split()])
    e, (a, c20, rdet) = np.ascontiguousarray(v[:9]), v[9:]
    Q = np.zeros(10)
    D = ctypes.c_double
    assert lib.kernel(ptr(e), D(a), D(c20), D(rdet), ptr(Q)) == 1
    ref = exact(e.reshape(3, 3), a, c20, rdet)
    big = max(abs(x) for x in ref)
    assert max(abs(Fraction(float(q)) - x) for q, x in zip(Q, ref)) <= Fraction(8 * U) * big


def test_condensation_of_needles(lib):
    """The same bound on elements that are nearly collinear or coplanar off the axes."""
    rng = np.random.default_rng(2)
    taken = 0
    for i in range(200):
        e = graded(("needle", "flat")[i % 2], float(rng.uniform(4, 40)), rng)
        rdet = 1.0 / abs(np.linalg.det(e))
        a = float(np.exp(rng.standard_normal()))
        c20 = a / float((e ** 2).sum(1).max()) * 10.0 ** rng.uniform(-12, -1)
        Q = np.zeros(10)
        D = ctypes.c_double
        if not lib.kernel(ptr(e), D(a), D(c20), D(rdet), ptr(Q)):
            continue
        taken += 1
        ref = exact(e, a, c20, rdet)
        big = max(abs(x) for x in ref)
        assert max(abs(Fraction(float(q)) - x) for q, x in zip(Q, ref)) <= Fraction(8 * U) * big
    assert taken >= 60


@pytest.mark.parametrize("spread", [0, 1, 2, 4, 8])
def test_product_rows(lib, spread):
    """Each row of Q z that is not marked for fp64, to 8 x 2^-53 of its own terms:
    one for the rounding to fp64, one for half a unit of the sum (2^-60 of
    max|Q| max|z|, of which the row's largest term is at least 2^-7), and two
    (a unit) for each of the three other terms if an operand of it is cut.  The
    root mean square stays below fp64's own chain, and most rows are taken."""
    rng = np.random.default_rng(spread)
    at = [[0, 1, 2, 3], [1, 4, 5, 6], [2, 5, 7, 8], [3, 6, 8, 9]]
    taken, err, err64 = 0, [], []
    n = 500
    for _ in range(n):
        Q = rng.uniform(-2, 2, 10) * 10.0 ** rng.uniform(-spread, 0, 10)
        z = rng.uniform(-2, 2, 4) * 10.0 ** rng.uniform(-spread, 0, 4)
        e, small = np.zeros(4), ctypes.c_uint(0)
        assert lib.product(ptr(Q), ptr(z), ptr(e), ctypes.byref(small)) == 1
        for k in range(4):
            if small.value >> k & 1:
                continue
            taken += 1
            f = [Fraction(float(Q[at[k][m]])) * Fraction(float(z[m])) for m in range(4)]
            terms = float(sum(abs(x) for x in f))
            chain = 0.0
            for x in f:  # the fma chain: each sum rounded once
                chain = float(Fraction(chain) + x)
            err.append(abs(float(Fraction(float(e[k])) - sum(f))) / terms)
            err64.append(abs(float(Fraction(chain) - sum(f))) / terms)
    assert max(err) <= 8 * U
    assert np.mean(np.square(err)) <= np.mean(np.square(err64))
    assert taken >= (4 * n if spread == 0 else n) * 0.9
