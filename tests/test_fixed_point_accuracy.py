"""The fixed-point element algebra (csrc/fixed.cuh, compiled here for the CPU)
against exact rational arithmetic where entries of one element differ in size:
edges and faces of a graded mesh, rows of Q z over several decades."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

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
