// Per-element helpers shared by the assembly, recovery and adjoint kernels:
// the geometry record of the mesh and the condensation kernel Qf of one
// element (see assemble.cu for the derivation).
#pragma once

#include "dw.cuh"
#include "fixed.cuh"
#include "ph_internal.cuh"

namespace ph_elem {

__device__ __forceinline__ int comp(int4 v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }
__device__ __forceinline__ unsigned short comps(ushort4 v, int k) {
  return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
}

// Index of (k, m), k <= m, in the packed upper triangle 00 01 02 03 11 12 13 22 23 33.
__host__ __device__ constexpr int ut(int k, int m) {
  return k <= m ? (k * 7 - k * k) / 2 + m : (m * 7 - m * m) / 2 + k;
}

struct Geo {
  double g00, g01, g02, g11, g12, g22;  // G_e
  double adet, rdet;
};

// The edge vectors E = rows P_i - P_0 (i = 1..3) of tet [P0 P1 P2 P3].
__device__ __forceinline__ void edge_vectors(const double* __restrict__ coord, int4 v, double e[3][3]) {
  const double* p0 = coord + 3 * (int64_t)v.x;
  const double* p1 = coord + 3 * (int64_t)v.y;
  const double* p2 = coord + 3 * (int64_t)v.z;
  const double* p3 = coord + 3 * (int64_t)v.w;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    e[0][d] = p1[d] - p0[d];
    e[1][d] = p2[d] - p0[d];
    e[2][d] = p3[d] - p0[d];
  }
}

// |det E| in fp64 (the sign bit cleared).
__device__ __forceinline__ double abs_det(const double e[3][3]) {
  const double det = e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) +
                     e[0][1] * (e[1][2] * e[2][0] - e[1][0] * e[2][2]) +
                     e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]);
  return ph::neg_if(det, __double2hiint(det) < 0);
}

// G_e = E E' in fp64 (00 01 02 11 12 22), for the elements that fx::geometry
// leaves out.
__device__ __forceinline__ void gram(const double e[3][3], double g[6]) {
  g[0] = e[0][0] * e[0][0] + e[0][1] * e[0][1] + e[0][2] * e[0][2];
  g[1] = e[0][0] * e[1][0] + e[0][1] * e[1][1] + e[0][2] * e[1][2];
  g[2] = e[0][0] * e[2][0] + e[0][1] * e[2][1] + e[0][2] * e[2][2];
  g[3] = e[1][0] * e[1][0] + e[1][1] * e[1][1] + e[1][2] * e[1][2];
  g[4] = e[1][0] * e[2][0] + e[1][1] * e[2][1] + e[1][2] * e[2][2];
  g[5] = e[2][0] * e[2][0] + e[2][1] * e[2][1] + e[2][2] * e[2][2];
}

// The geometry record of element t as stored: g and its scale.
struct Record {
  int64_t g[6];
  int kg;  // PH_GEXP_F64: g holds doubles
};
__device__ __forceinline__ Record load_record(const double* __restrict__ geo, const int32_t* __restrict__ gexp,
                                              int64_t t) {
  const longlong2* p = reinterpret_cast<const longlong2*>(geo + PH_GEO_STRIDE * t);
  const longlong2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
  return Record{{a.x, a.y, b.x, b.y, c.x, c.y}, __ldg(gexp + t)};
}
// The same in fp64.
__device__ __forceinline__ Geo to_f64(const Record& r, double2 vol) {
  double g[6];
#pragma unroll
  for (int i = 0; i < 6; ++i)
    g[i] = r.kg == PH_GEXP_F64 ? __longlong_as_double(r.g[i]) : fx::to_double(r.g[i], r.kg);
  return Geo{g[0], g[1], g[2], g[3], g[4], g[5], vol.x, vol.y};
}

// Qf (face-indexed, packed upper triangle) times sc = sc6/6.
__device__ __forceinline__ void face_kernel(const Geo& G, double a, double c20, double sc6, double Q[10]) {
  const double a2 = a + a;
  const double m00 = fma(c20, G.g00, a2), m11 = fma(c20, G.g11, a2), m22 = fma(c20, G.g22, a2);
  const double m01 = fma(c20, G.g01, a), m02 = fma(c20, G.g02, a), m12 = fma(c20, G.g12, a);
  double A00 = fma(m11, m22, -m12 * m12);
  double A01 = fma(m02, m12, -m01 * m22);
  double A02 = fma(m01, m12, -m02 * m11);
  double A11 = fma(m00, m22, -m02 * m02);
  double A12 = fma(m01, m02, -m00 * m12);
  double A22 = fma(m00, m11, -m01 * m01);
  const double detM = fma(m00, A00, fma(m01, A01, m02 * A02));
  const double s = (sc6 * G.rdet) * ph::rcp_newton(detM);  // sc * 6/|det E| / det M
  A00 *= s; A01 *= s; A02 *= s; A11 *= s; A12 *= s; A22 *= s;
  // G_e T0^-1 = G_e - (G_e 1) 1'/4 (T0 = I + 1 1'; one fma per entry, the quarter being exact)
  const double r0 = (G.g00 + G.g01) + G.g02, r1 = (G.g01 + G.g11) + G.g12, r2 = (G.g02 + G.g12) + G.g22;
  const double t00 = fma(-0.25, r0, G.g00), t01 = fma(-0.25, r0, G.g01), t02 = fma(-0.25, r0, G.g02);
  const double t10 = fma(-0.25, r1, G.g01), t11 = fma(-0.25, r1, G.g11), t12 = fma(-0.25, r1, G.g12);
  const double t20 = fma(-0.25, r2, G.g02), t21 = fma(-0.25, r2, G.g12), t22 = fma(-0.25, r2, G.g22);
  // Y = adj(M) G_e T0^-1 (symmetric): upper triangle
  const double y00 = fma(A00, t00, fma(A01, t10, A02 * t20));
  const double y01 = fma(A00, t01, fma(A01, t11, A02 * t21));
  const double y02 = fma(A00, t02, fma(A01, t12, A02 * t22));
  const double y11 = fma(A01, t01, fma(A11, t11, A12 * t21));
  const double y12 = fma(A01, t02, fma(A11, t12, A12 * t22));
  const double y22 = fma(A02, t02, fma(A12, t12, A22 * t22));
  // Qv = D0' Y D0; faces 0,1,2,3 sit opposite vertices 3,1,2,0
  const double c0 = y00 + y01 + y02, c1 = y01 + y11 + y12, c2 = y02 + y12 + y22;
  Q[ut(0, 0)] = y22;
  Q[ut(0, 1)] = y02;
  Q[ut(0, 2)] = y12;
  Q[ut(0, 3)] = ph::negate(c2);
  Q[ut(1, 1)] = y00;
  Q[ut(1, 2)] = y01;
  Q[ut(1, 3)] = ph::negate(c0);
  Q[ut(2, 2)] = y11;
  Q[ut(2, 3)] = ph::negate(c1);
  Q[ut(3, 3)] = c0 + c1 + c2;
}

// The condensation kernel Qf/9 of an element from its record: fixed point
// (fixed.cuh), or fp64 for the elements it leaves out.
__device__ __forceinline__ void element_kernel(const Record& r, double2 vol, double a, double c20, double Q[10]) {
  const auto rcp = [](double x) { return ph::rcp_newton(x); };
  if (r.kg == PH_GEXP_F64 || !fx::face_kernel(r.g, r.kg, a, c20, vol.y, rcp, Q))
    face_kernel(to_f64(r, vol), a, c20, 6.0 / 9.0, Q);
}

using ph::neg_if;


// Local matrices, condensation and scatter of element t (Section 4.2-4.3,
// Eq. schur): the body of the assembly kernels (one thread per element).
// UD, GN, FAC: u_D and g_N given, the factor wanted (constants of the plain
// kernels, the problem's in the batched one).
__device__ __forceinline__ void assemble_element(bool UD, bool GN, bool FAC, int64_t t, const double* __restrict__ geo,
                                                 const int32_t* __restrict__ gexp, const double2* __restrict__ vol,
                                                 const int4* __restrict__ tface, const int4* __restrict__ tmult,
                                                 const int4* __restrict__ tpos, const ushort4* __restrict__ trel,
                                                 const double* __restrict__ face_area, const double* __restrict__ a,
                                                 double c20, double six_over_c, const double* __restrict__ f_face,
                                                 const double* __restrict__ uD, const double* __restrict__ gN,
                                                 double* __restrict__ values, double* __restrict__ rhs,
                                                 double* __restrict__ factor, unsigned* status) {
  const double at = __ldg(a + t);
  if (!ph::pos_finite(at)) {
    ph_flag(status, PH_ERR_ARG);
    return;
  }
  const double2 vt = __ldg(vol + t);  // |det E|, 1/|det E|
  const Record R = load_record(geo, gexp, t);
  const int4 tf = __ldg(tface + t);
  const int4 tm = __ldg(tmult + t);
  int F[4];
  bool neg[4];
  double ar[4], h[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    F[k] = comp(tf, k) & PH_ID_MASK;
    neg[k] = comp(tf, k) < 0;
    ar[k] = __ldg(face_area + F[k]);
  }
  const double q4 = vt.x * (1.0 / 24.0);  // |T| / 4
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    h[k] = q4 * __ldg(f_face + F[k]);
    if (GN && comp(tm, k) == PH_NO_MULT) h[k] = fma(ar[k], __ldg(gN + F[k]), h[k]);
  }
  double Q[10];
  element_kernel(R, vt, at, c20, Q);
  if (FAC) {
    double2* fo = reinterpret_cast<double2*>(factor + 10 * t);
    fo[0] = make_double2(Q[0], Q[1]);
    fo[1] = make_double2(Q[2], Q[3]);
    fo[2] = make_double2(Q[4], Q[5]);
    fo[3] = make_double2(Q[6], Q[7]);
    fo[4] = make_double2(Q[8], Q[9]);
  }
  const double icT = vt.y * six_over_c;  // 1/(c|T|)
  const double hs = (h[0] + h[1]) + (h[2] + h[3]);
  const double base = icT * hs;
  // condensed block S[k][m] = d_k d_m (1/(c|T|) + Qf/9), each entry once, as
  // d_k (Q_km d_m + e_m) with d = sigma |F| (sign on the bit pattern) and
  // e_m = d_m / (c|T|): 4 + 2 per entry FP64 operations.  (In fixed point too,
  // from the integers behind Q: 24 FP64 operations fewer but 800 integer
  // instructions more, 2.31 -> 2.62 ms at 17.9M tets.)
  double d[4], e4[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[k] = neg_if(ar[k], neg[k]);
    e4[k] = icT * d[k];
  }
  double S[10];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int m = k; m < 4; ++m) S[ut(k, m)] = d[k] * fma(Q[ut(k, m)], d[m], e4[m]);
  const int4 tp = __ldg(tpos + t);
  const ushort4 tr = __ldg(trel + t);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int mk = comp(tm, k);
    if (mk == PH_NO_MULT) continue;
    const int l = mk & PH_ID_MASK;
    const bool bnd = mk < 0;
    // g_k = -d_k (h'sum/(c|T|) + (Qf h')_k / 9)
    double e = base;
#pragma unroll
    for (int m = 0; m < 4; ++m) e = fma(Q[ut(k, m)], h[m], e);
    double g = neg_if(ar[k] * e, !neg[k]);
    if (UD && bnd) g = fma(ar[k], __ldg(uD + F[k]), g);  // b_D = |F| u_D(Ct_F)
    const int pd = comp(tp, k);
    if (bnd) {
      values[pd] = S[ut(k, k)];
      rhs[l] = g;
    } else {
      atomicAdd(values + pd, S[ut(k, k)]);
      atomicAdd(rhs + l, g);
    }
    const unsigned rel = comps(tr, k);
    int idx = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (m == k) continue;
      if (comp(tm, m) != PH_NO_MULT) {
        const int off = ((int)(rel << (28 - 4 * idx))) >> 28;  // sign-extend 4 bits
        values[pd + off] = S[ut(k, m)];
      }
      ++idx;
    }
  }
}

__device__ __forceinline__ void store_u(double* __restrict__ u, int64_t t, const double U[4]) {
  // vertex j holds U of the face opposite it: j = 0,1,2,3 <- k = 3,1,2,0
  double2* out = reinterpret_cast<double2*>(u + 4 * t);
  out[0] = make_double2(U[3], U[1]);
  out[1] = make_double2(U[2], U[0]);
}

// z'_k = |T|/4 f(Ct_k) + |F_k| g(Ct_k) [Neumann] + d_k Lambda_k
__device__ __forceinline__ void recovery_load(bool GN, double q4, int4 tf, int4 tm, const double* __restrict__ face_area,
                                              const double* __restrict__ f_face, const double* __restrict__ gN,
                                              const double* __restrict__ lambda, double z[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int F = comp(tf, k) & PH_ID_MASK;
    const int mk = comp(tm, k);
    const double ar = __ldg(face_area + F);
    double zk = q4 * __ldg(f_face + F);
    if (mk == PH_NO_MULT) {
      if (GN) zk = fma(ar, __ldg(gN + F), zk);
    } else {
      zk = fma(neg_if(ar, comp(tf, k) < 0), __ldg(lambda + (mk & PH_ID_MASK)), zk);
    }
    z[k] = zk;
  }
}

// Recovery of element t from the element factor Qf/9 stored by the assembly
// (Algorithm 1, second loop): U[o(k)] = z'sum/(c|T|) - 3 (Qf/9 z')_k.  The
// body of the plain and the batched recovery kernels.
// FIXED: the product in fixed point (fixed.cuh), 18 FP64 operations instead of
// 34, which bound the kernel (17.9M tets: 1.09 -> 0.745 ms).  A row that it leaves
// out (one in some hundreds of random fields) reads its factor again: held in
// registers for that, the kernel took 0.96 ms.
// (GN, FIXED: constants of the plain kernels, the problem's in the batched one.)
__device__ __forceinline__ void recover_element_factored(bool GN, bool FIXED, int64_t t,
                                                         const double2* __restrict__ vol,
                                                         const int4* __restrict__ tface,
                                                         const int4* __restrict__ tmult,
                                                         const double* __restrict__ face_area,
                                                         const double* __restrict__ factor, double six_over_c,
                                                         const double* __restrict__ f_face,
                                                         const double* __restrict__ gN,
                                                         const double* __restrict__ lambda, double* __restrict__ u) {
  const double2 vt = __ldg(vol + t);
  double z[4];
  recovery_load(GN, vt.x * (1.0 / 24.0), __ldg(tface + t), __ldg(tmult + t), face_area, f_face, gN, lambda, z);
  const double2* fp = reinterpret_cast<const double2*>(factor + 10 * t);
  const double2 q0 = __ldg(fp), q1 = __ldg(fp + 1), q2 = __ldg(fp + 2), q3 = __ldg(fp + 3), q4 = __ldg(fp + 4);
  const double Q[10] = {q0.x, q0.y, q1.x, q1.y, q2.x, q2.y, q3.x, q3.y, q4.x, q4.y};
  const double icT = vt.y * six_over_c;
  const double zs = icT * ((z[0] + z[1]) + (z[2] + z[3]));
  double e[4], U[4];
  if (FIXED) {
    unsigned rows;  // to form in fp64, as the other branch does
    if (!fx::product4(Q, z, e, &rows)) rows = 0xF;
    while (rows) {
      const int k = __ffs(rows) - 1;
      rows &= rows - 1;
      double s = 0.0;
#pragma unroll
      for (int m = 0; m < 4; ++m) s = fma(__ldg(factor + 10 * t + ut(k, m)), z[m], s);
#pragma unroll
      for (int j = 0; j < 4; ++j) e[j] = j == k ? s : e[j];
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      e[k] = 0.0;
#pragma unroll
      for (int m = 0; m < 4; ++m) e[k] = fma(Q[ut(k, m)], z[m], e[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) U[k] = fma(-3.0, e[k], zs);
  store_u(u, t, U);
}

// The same recovery with the product (Qf/9) z' in double-word arithmetic on
// the FP32 pipe (dw.cuh): the factor and z' become float pairs scaled by the
// element's largest binade of each, each row sum returns to fp64 exactly
// scaled.  z', its sum and the final combination stay fp64: they are the
// terms whose rounding bounds the result when a Lambda that is not a
// solution makes them cancel, and the pairs' ~2^-47 lands on the smaller
// (Qf z')/3 (a factor c h^2/a below them).  18 FP64 operations per element
// instead of 34.  Elements whose binades leave the pairs' range take the fp64
// product.
template <bool GN>
__device__ __forceinline__ void recover_element_factored_dw(int64_t t, const double2* __restrict__ vol,
                                                            const int4* __restrict__ tface,
                                                            const int4* __restrict__ tmult,
                                                            const double* __restrict__ face_area,
                                                            const double* __restrict__ factor, double six_over_c,
                                                            const double* __restrict__ f_face,
                                                            const double* __restrict__ gN,
                                                            const double* __restrict__ lambda,
                                                            double* __restrict__ u) {
  using namespace dw;
  const double2 vt = __ldg(vol + t);
  double z[4];
  recovery_load(GN, vt.x * (1.0 / 24.0), __ldg(tface + t), __ldg(tmult + t), face_area, f_face, gN, lambda, z);
  const double2* fp = reinterpret_cast<const double2*>(factor + 10 * t);
  const double2 q0 = __ldg(fp), q1 = __ldg(fp + 1), q2 = __ldg(fp + 2), q3 = __ldg(fp + 3), q4 = __ldg(fp + 4);
  const double Q[10] = {q0.x, q0.y, q1.x, q1.y, q2.x, q2.y, q3.x, q3.y, q4.x, q4.y};
  const double icT = vt.y * six_over_c;
  const double zs = icT * ((z[0] + z[1]) + (z[2] + z[3]));
  int kq = -1023, kz = -1023;
#pragma unroll
  for (int i = 0; i < 10; ++i) kq = max(kq, exponent(Q[i]));
#pragma unroll
  for (int m = 0; m < 4; ++m) kz = max(kz, exponent(z[m]));
  double U[4];
  if (kq > -900 && kq < 900 && kz > -900 && kz < 900 && kq + kz > -1000 && kq + kz < 1000) {
    f2 qd[10], zd[4];
#pragma unroll
    for (int i = 0; i < 10; ++i) qd[i] = from_double(Q[i], -kq);
#pragma unroll
    for (int m = 0; m < 4; ++m) zd[m] = from_double(z[m], -kz);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      f2 v = mul(qd[ut(k, 0)], zd[0]);
#pragma unroll
      for (int m = 1; m < 4; ++m) v = add(v, mul(qd[ut(k, m)], zd[m]));
      U[k] = fma(-3.0, to_double(v, kq + kz), zs);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double e = 0.0;
#pragma unroll
      for (int m = 0; m < 4; ++m) e = fma(Q[ut(k, m)], z[m], e);
      U[k] = fma(-3.0, e, zs);
    }
  }
  store_u(u, t, U);
}

}  // namespace ph_elem
