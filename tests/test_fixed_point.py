"""The fixed-point element algebra (csrc/fixed.cuh, compiled here for the CPU)
against exact rational arithmetic, over the forms it accepts -- regular,
jittered, random and anisotropic elements, nine decades of size, reaction terms
up to a quarter of the diffusion -- and the elements it leaves to fp64.

Bound.  Q is the exact expression of the given 1/|det E| with three fp64
roundings in its scalar and its own rounding below 2^-53 of the largest entry:
within 8 x 2^-53 of that.
"""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "fixed.cuh"
extern "C" int run(const double* e, double a, double c20, double rdet, double* Q) {
  int64_t g[6];
  int kg;
  const double(*E)[3] = reinterpret_cast<const double(*)[3]>(e);
  if (!fx::geometry(E, g, kg)) return 0;
  return fx::face_kernel(g, kg, a, c20, rdet, [](double x) { return 1.0 / x; }, Q) ? 2 : 1;
}
extern "C" int product(const double* Q, const double* z, double* e) { return fx::product4(Q, z, e); }
extern "C" double there_and_back(double x, int k) { return fx::to_double(fx::from_double(x, k), k - 60); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "libfx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-static-libubsan", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2509_11133_gb300", "csrc"),
                    str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    D = ctypes.c_double
    L.run.argtypes = [ctypes.POINTER(D), D, D, D, ctypes.POINTER(D)]
    L.product.argtypes = [ctypes.POINTER(D)] * 3
    L.there_and_back.argtypes, L.there_and_back.restype = [D, ctypes.c_int], D
    return L


def run(lib, e, a, c20):
    e = np.ascontiguousarray(e, dtype=np.float64)
    P = ctypes.POINTER(ctypes.c_double)
    Q = np.zeros(10)
    rdet = 1.0 / (abs(np.linalg.det(e)) or 1.0) if np.isfinite(e).all() else 1.0
    return lib.run(e.ctypes.data_as(P), a, c20, rdet, Q.ctypes.data_as(P)), rdet, Q


def exact(e, a, c20, rdet):
    E = [[Fraction(float(x)) for x in r] for r in e]
    a, c20, rdet = Fraction(float(a)), Fraction(float(c20)), Fraction(float(rdet))
    G = [[sum(x * y for x, y in zip(r, s)) for s in E] for r in E]
    M = [[a * (2 if i == j else 1) + c20 * G[i][j] for j in range(3)] for i in range(3)]
    T = [[G[i][j] - sum(G[i]) / 4 for j in range(3)] for i in range(3)]
    cof = lambda i, j: (M[(i + 1) % 3][(j + 1) % 3] * M[(i + 2) % 3][(j + 2) % 3] -
                        M[(i + 1) % 3][(j + 2) % 3] * M[(i + 2) % 3][(j + 1) % 3])
    A = [[cof(j, i) for j in range(3)] for i in range(3)]
    s = Fraction(2, 3) * rdet / sum(M[0][j] * A[j][0] for j in range(3))
    Y = [[s * sum(A[i][k] * T[k][j] for k in range(3)) for j in range(3)] for i in range(3)]
    V = [[Fraction(0)] * 4 for _ in range(4)]  # D0' Y D0, D0 = [-1 | I]
    for i in range(3):
        for j in range(3):
            V[i + 1][j + 1] += Y[i][j]
            V[0][j + 1] -= Y[i][j]
            V[i + 1][0] -= Y[i][j]
            V[0][0] += Y[i][j]
    o = (3, 1, 2, 0)
    return [V[o[k]][o[m]] for k in range(4) for m in range(k, 4)]


def elements(kind, n=150):
    rng = np.random.default_rng(11)
    base = np.array([[[1, 0, 0], [1, 1, 0], [1, 1, 1]], [[.5, 0, 0], [.5, .5, 0], [.625, .375, .25]],
                     [[1, 0, 0], [0, 1, 0], [0, 0, 1]], [[1, 1, -1], [1, -1, 1], [-1, 1, 1]]])
    for i in range(n):
        e = base[i % 4].copy()
        if kind == "jittered":
            e += 0.2 * rng.uniform(-1, 1, (3, 3))
        elif kind == "random":
            e = rng.standard_normal((3, 3))
        elif kind == "anisotropic":
            e = (e + 0.2 * rng.uniform(-1, 1, (3, 3))) * np.array([1.0, 0.4, 0.1])
        elif kind == "edge of a binade":
            e = e * np.nextafter(1.0, [0.0, 2.0, 1.0][i % 3])
        h = 10.0 ** rng.uniform(-6, 3)
        o = rng.uniform(0, 1, 3) * h
        e = ((o + h * e) - o)  # the rounding of a difference of coordinates
        a = [1.0, 1e4, float(np.exp(rng.standard_normal()))][i % 3]
        g = float((e ** 2).sum(1).max())
        yield e, a, a / g * 10.0 ** rng.uniform(-20, -1)


@pytest.mark.parametrize("kind", ["regular", "jittered", "random", "anisotropic", "edge of a binade"])
def test_against_rationals(lib, kind):
    taken = 0
    for e, a, c20 in elements(kind):
        code, rdet, Q = run(lib, e, a, c20)
        if code == 2:
            taken += 1
            ref = exact(e, a, c20, rdet)
            big = max(abs(x) for x in ref)
            assert max(abs(Fraction(float(q)) - x) for q, x in zip(Q, ref)) <= Fraction(8 * 2.0 ** -53) * big
    assert taken >= 60


@pytest.mark.parametrize("spread", [0, 3, 30])
def test_product(lib, spread):
    """Rows of Q z over `spread` decades of entries: 2^-53.9 of max|Q| max|z|, then rounded."""
    rng = np.random.default_rng(spread)
    P = ctypes.POINTER(ctypes.c_double)
    at = [[0, 1, 2, 3], [1, 4, 5, 6], [2, 5, 7, 8], [3, 6, 8, 9]]
    for i in range(300):
        Q = rng.uniform(-2, 2, 10) * 10.0 ** rng.uniform(-spread, 0, 10) * 10.0 ** rng.uniform(-30, 30)
        z = rng.uniform(-2, 2, 4) * 10.0 ** rng.uniform(-spread, 0, 4) * 10.0 ** rng.uniform(-30, 30)
        if i % 5 == 0:
            Q[i % 10], z[i % 4] = 0.0, np.nextafter(2.0, 0) * 2.0 ** 3
        e = np.zeros(4)
        assert lib.product(Q.ctypes.data_as(P), z.ctypes.data_as(P), e.ctypes.data_as(P)) == 1
        scale = Fraction(float(np.abs(Q).max())) * Fraction(float(np.abs(z).max()))
        for k in range(4):
            ref = sum(Fraction(float(Q[at[k][m]])) * Fraction(float(z[m])) for m in range(4))
            assert abs(Fraction(float(e[k])) - ref) <= Fraction(2.0 ** -53.9) * scale + Fraction(2.0 ** -53) * abs(ref)
    for bad in (np.nan, np.inf):
        Q[3] = bad
        assert lib.product(Q.ctypes.data_as(P), z.ctypes.data_as(P), e.ctypes.data_as(P)) == 0
    assert lib.product(np.zeros(10).ctypes.data_as(P), z.ctypes.data_as(P), e.ctypes.data_as(P)) == 0


def test_left_to_fp64(lib):
    e = np.array([[1.0, 0, 0], [1, 1, 0], [1, 1, 1]])
    assert run(lib, e, 1.0, 0.05)[0] == 2
    for bad in (np.nan, np.inf, -np.inf):
        b = e.copy()
        b[1, 2] = bad
        assert run(lib, b, 1.0, 0.05)[0] == 0
    assert run(lib, np.zeros((3, 3)), 1.0, 0.05)[0] == 0
    assert run(lib, e * [1, 1, 0], 1.0, 0.05)[0] == 0           # no extent along a coordinate
    assert run(lib, e * [1, 1, 1 / 64], 1.0, 0.05)[0] == 0      # an extent below 1/16 of the largest
    assert run(lib, e * [[1], [1 / 64], [1]], 1.0, 0.05)[0] == 0  # an edge below it
    assert run(lib, e * 1e120, 1.0, 0.05)[0] == 0               # out of the exponent range
    assert run(lib, e, 1e-3, 0.05)[0] == 1                      # the reaction term dominates
    assert run(lib, e, 5e-324, 0.05)[0] == 1


@pytest.mark.parametrize("k", [-300, -3, 0, 1, 52, 300])
def test_conversions(lib, k):
    rng = np.random.default_rng(k + 1000)
    assert lib.there_and_back(0.0, k) in (0.0, math.ldexp(1.0, k - 60))  # below one unit
    for x in list(rng.uniform(-2, 2, 200)) + [1.0, -1.0, np.nextafter(2.0, 0), 2.0 ** -8, -2.0 ** -8 * 1.25]:
        y = math.ldexp(x, k)
        if abs(x) >= 2.0 ** -8:
            assert lib.there_and_back(y, k) == y
        else:
            assert abs(lib.there_and_back(y, k) - y) <= math.ldexp(1.0, k - 60) + abs(y) * 2.0 ** -53
