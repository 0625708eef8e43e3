// Fixed-point evaluation of the element algebra on the integer pipe.
//
// On this part FP64 issues 1.75 operations per clock per SM and the integer
// pipe about 100 (a 32 x 32 -> 64 bit multiply-add, IMAD.WIDE: 14).  The edge
// Gram matrix of an element and the 3x3 algebra of its condensation kernel
// (assemble.cu) are sums of products of numbers of similar size, so they are
// formed here in 64-bit integers with one power of two per element: a product
// of two such numbers takes three IMAD.WIDE (0.2 clocks, against 0.57 for a
// DFMA) on a pipe that the FP64 kernels leave idle.  The results return to fp64
// rounded to nearest.
//
// A number is an int64 v with |v| < 2^61 (up to 2^62 where noted) and a scale
// known per element.  A product uses v = h 2^32 + l with l a signed 32-bit
// integer: sum of v w = 2^64 sum(h h') + 2^32 sum(h l' + l h') + sum(l l'),
// and the last sum, below 2^62 per term, is left out where the result keeps no bits
// below it, and kept (mac_wide) where the sum is shifted further: left out of Y
// (a shift of 6) it cost Q up to 10.7 x 2^-53 of its largest entry, now 4.4 at worst
// and 1.2 rms at most over the shapes that are accepted; fp64: 22 and 3.4.
// Sums of at most three products do not overflow with |v|, |w| <= 2^61:
// |h l'| <= 2^60, six of them 2^62.6.  The high sum may be shifted past 2^63 on
// the way (two's complement): only the final value has to fit.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace fx {

struct Half {
  int h, l;  // v = h 2^32 + l
};
FX_HD Half split(int64_t v) {
  const int l = (int)(uint32_t)(uint64_t)v;
  return Half{(int)((uint32_t)((uint64_t)v >> 32) + ((uint32_t)l >> 31)), l};
}

struct Acc {
  int64_t hh = 0, x = 0;
  FX_HD Acc() {}
  // rounds shifted(., s) to nearest
  FX_HD explicit Acc(int s) : x((int64_t)1 << (31 - s)) {}
};
FX_HD void mac(Acc& a, Half v, Half w) {
  a.hh += (int64_t)v.h * w.h;
  a.x += (int64_t)v.h * w.l;
  a.x += (int64_t)v.l * w.h;
}
// the same with the low product kept (its upper half)
FX_HD void mac_wide(Acc& a, Half v, Half w) {
  a.x += ((int64_t)v.l * w.l) >> 32;
  mac(a, v, w);
}
// the sum of products times 2^(s - 64), 0 <= s < 32
FX_HD int64_t shifted(const Acc& a, int s) { return (int64_t)((uint64_t)a.hh << s) + (a.x >> (32 - s)); }

// v w 2^(s - 64), rounded, with the low product kept
FX_HD int64_t mul_wide(Half v, Half w, int s) {
  Acc a(s);
  mac_wide(a, v, w);
  return shifted(a, s);
}

#ifdef __CUDA_ARCH__
__device__ __forceinline__ int clz64(uint64_t v) { return __clzll((long long)v); }
__device__ __forceinline__ uint64_t bits_of(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double of_bits(uint64_t b) { return __longlong_as_double((long long)b); }
#else
inline int clz64(uint64_t v) { return v ? __builtin_clzll(v) : 64; }
inline uint64_t bits_of(double x) {
  uint64_t b;
  __builtin_memcpy(&b, &x, 8);
  return b;
}
inline double of_bits(uint64_t b) {
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
}
#endif

// floor(log2 |x|) of a normal x
FX_HD int exponent(double x) { return (int)((bits_of(x) >> 52) & 0x7FF) - 1023; }

// x 2^(60 - k), truncated: |x| < 2^(k+1), so the result is below 2^61
FX_HD int64_t from_double(double x, int k) {
  const uint64_t b = bits_of(x);
  const int64_t m = (int64_t)(((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 8);
  const int d = k + 1023 - (int)((b >> 52) & 0x7FF);
  const int64_t v = m >> (d < 63 ? d : 63);
  const int64_t s = (int64_t)b >> 63;
  return (v ^ s) - s;
}

// v 2^k rounded to nearest (ties away from zero); v 2^k a normal double
FX_HD double to_double(int64_t v, int k) {
  const int64_t s = v >> 63;
  const uint64_t u = (uint64_t)((v ^ s) - s);
  if (u == 0) return 0.0;
  const int z = clz64(u);
  const uint64_t n = u << z;  // top bit set
  // biased exponent 63 - z + k + 1023; the mantissa's leading bit adds one to
  // the exponent field, and a carry of the rounding propagates into it
  const uint64_t e = (uint64_t)(int64_t)(63 - z + k + 1022) << 52;
  return of_bits((e + (n >> 11) + ((n >> 10) & 1)) | ((uint64_t)s << 63));
}

// ---------------------------------------------------------------------------
// Geometry: G = E E' (00 01 02 11 12 22) of the edge vectors E (rows P_i - P_0)
// as g = v 2^kg with the largest diagonal entry in [2^59, 2^60].  A component of E
// within 2^-7 of the largest converts exactly, the low products are kept, and the
// sum is rounded to nearest: half a unit of 2^kg.  False when the element is left
// to fp64, because the common scale would cost its small entries bits that fp64
// keeps: a squared edge below 2^-7 of the largest (kShort; at 2^-7 half a unit is
// 2^-53 of the entry), or an edge, or the extent along a coordinate, below 2^-4 of
// the largest edge component (kSpread); or for an exponent out of range (NaN and
// infinity among them).  So every entry is as accurate as in fp64, over regular,
// jittered, flat, needle and short-edged elements against binary128: diagonal
// entries to 0.6 x 2^-53 (rms; 0.7 at most for a shape) where fp64 has 0.8, 1.5
// against 2.9 at worst, and with them the contraction with adj(G) of the gradient
// (median, 90th and 99th percentile of the error 0.7 to 1.0 of fp64's).
// |det E| and the face areas stay fp64: they carry the leading term d d'/(c|T|) of
// H, whose last bit an ill-conditioned solve amplifies by 1e7, and rounding them
// otherwise, if better, would move such solutions.
// ---------------------------------------------------------------------------
constexpr int kSpread = 4, kShort = 7;

FX_HD bool geometry(const double e[3][3], int64_t g[6], int& kg) {
  uint32_t m[3][3];
  for (int i = 0; i < 3; ++i)
    for (int d = 0; d < 3; ++d) m[i][d] = (uint32_t)(bits_of(e[i][d]) >> 32) & 0x7FFFFFFFu;
  uint32_t all = 0, least = 0x7FFFFFFFu;
  for (int i = 0; i < 3; ++i) {
    uint32_t r = m[i][0], c = m[0][i];
    for (int d = 1; d < 3; ++d) {
      r = r > m[i][d] ? r : m[i][d];
      c = c > m[d][i] ? c : m[d][i];
    }
    all = all > r ? all : r;
    least = least < r ? least : r;
    least = least < c ? least : c;
  }
  const int top = (int)(all >> 20), k = top - 1023;
  if (k < -300 || k > 300 || top - (int)(least >> 20) > kSpread) return false;
  Half h[3][3];
  for (int i = 0; i < 3; ++i)
    for (int d = 0; d < 3; ++d) h[i][d] = split(from_double(e[i][d], k));
  Acc a[6];
  for (int d = 0; d < 3; ++d) {
    mac_wide(a[0], h[0][d], h[0][d]);
    mac_wide(a[1], h[0][d], h[1][d]);
    mac_wide(a[2], h[0][d], h[2][d]);
    mac_wide(a[3], h[1][d], h[1][d]);
    mac_wide(a[4], h[1][d], h[2][d]);
    mac_wide(a[5], h[2][d], h[2][d]);
  }
  int64_t most = a[0].hh > a[3].hh ? a[0].hh : a[3].hh, fewest = a[0].hh < a[3].hh ? a[0].hh : a[3].hh;
  most = most > a[5].hh ? most : a[5].hh;  // in [2^56, 3 2^58]
  fewest = fewest < a[5].hh ? fewest : a[5].hh;
  if (fewest < most >> kShort) return false;
  const int s = clz64((uint64_t)most) - 4;
  for (int i = 0; i < 6; ++i) {
    a[i].x += (int64_t)1 << (31 - s);
    g[i] = shifted(a[i], s);
  }
  kg = 2 * k - 56 - s;
  return true;
}

// ---------------------------------------------------------------------------
// The condensation kernel Q = Qf/9 (face-indexed, packed upper triangle) of an
// element from its fixed-point G: with M = a T0 + (c/20) G (T0 = I + 1 1'),
//     Y = (6/9) / (|det E| det M) adj(M) G T0^-1,   G T0^-1 = G - (G 1) 1'/4,
// expanded to the faces as in face_kernel (element.cuh).  `rcp` is the fp64
// reciprocal.  False (fp64 takes the element) when (c/20) G exceeds a quarter
// of a, or an exponent leaves the range.
//
// Scales, with am = a 2^(59 - ka) in [2^59, 2^60): M < 2^61.1 in units of am's;
// A = adj(M) 2^-63 in [2^56.5, 2^59.4]; det M = D 2^58 with D in [2^58, 2^61.6];
// A' = A (6/9)/|det E|/D below 2^59; Y below 2^62.1 (its entries and the sums
// below are entries of a positive semidefinite 4x4 matrix whose diagonal
// |x_v|^2/a is bounded by 25/16 of the largest g_ii).
// ---------------------------------------------------------------------------
template <class R>
FX_HD bool face_kernel(const int64_t g[6], int kg, double a, double c20, double rdet, const R& rcp, double Q[10]) {
  const int ka = exponent(a), kc = exponent(c20), kr = exponent(rdet);
  const int sh = ka - kc - kg - 62, ky = kr - ka + kg - 1;
  if (sh < 1 || ka < -900 || ka > 900 || kc < -900 || kc > 900 || kr < -900 || kr > 900 || ky < -900 || ky > 900)
    return false;
  const int64_t am = from_double(a, ka) >> 1;
  const Half cm = split(from_double(c20, kc));
  int64_t M[6];
  for (int i = 0; i < 6; ++i) {
    Acc p;
    mac(p, cm, split(g[i]));
    M[i] = shifted(p, 1) >> (sh < 63 ? sh : 63);
  }
  M[0] += 2 * am;
  M[1] += am;
  M[2] += am;
  M[3] += 2 * am;
  M[4] += am;
  M[5] += 2 * am;
  const Half m00 = split(M[0]), m01 = split(M[1]), m02 = split(M[2]), m11 = split(M[3]), m12 = split(M[4]),
             m22 = split(M[5]);
  const Half n01 = split(-M[1]), n02 = split(-M[2]), n12 = split(-M[4]);
  const auto two = [](Half p, Half q, Half r, Half t) {
    Acc s;
    mac(s, p, q);
    mac(s, r, t);
    return split(shifted(s, 1));
  };
  const Half A00 = two(m11, m22, n12, m12), A01 = two(m02, m12, n01, m22), A02 = two(m01, m12, n02, m11);
  const Half A11 = two(m00, m22, n02, m02), A12 = two(m01, m02, n12, m00), A22 = two(m00, m11, n01, m01);
  Acc d(6);
  mac_wide(d, m00, A00);
  mac_wide(d, m01, A01);
  mac_wide(d, m02, A02);
  const int64_t D = shifted(d, 6);
  if (D <= 0) return false;
  const Half s = split(from_double((6.0 / 9.0 * rdet) * rcp(to_double(D, 0)), kr - 57));
  const Half B00 = split(mul_wide(A00, s, 7)), B01 = split(mul_wide(A01, s, 7)), B02 = split(mul_wide(A02, s, 7));
  const Half B11 = split(mul_wide(A11, s, 7)), B12 = split(mul_wide(A12, s, 7)), B22 = split(mul_wide(A22, s, 7));
  // G T0^-1 by rows
  const int64_t r0 = (g[0] + g[1] + g[2]) >> 2, r1 = (g[1] + g[3] + g[4]) >> 2, r2 = (g[2] + g[4] + g[5]) >> 2;
  const Half t00 = split(g[0] - r0), t01 = split(g[1] - r0), t02 = split(g[2] - r0);
  const Half t10 = split(g[1] - r1), t11 = split(g[3] - r1), t12 = split(g[4] - r1);
  const Half t20 = split(g[2] - r2), t21 = split(g[4] - r2), t22 = split(g[5] - r2);
  const auto three = [](Half p, Half q, Half r, Half t, Half u, Half v) {
    Acc y(6);
    mac_wide(y, p, q);
    mac_wide(y, r, t);
    mac_wide(y, u, v);
    return shifted(y, 6);
  };
  const int64_t y00 = three(B00, t00, B01, t10, B02, t20), y01 = three(B00, t01, B01, t11, B02, t21);
  const int64_t y02 = three(B00, t02, B01, t12, B02, t22), y11 = three(B01, t01, B11, t11, B12, t21);
  const int64_t y12 = three(B01, t02, B11, t12, B12, t22), y22 = three(B02, t02, B12, t12, B22, t22);
  const int64_t c0 = y00 + y01 + y02, c1 = y01 + y11 + y12, c2 = y02 + y12 + y22;
  Q[0] = to_double(y22, ky);
  Q[1] = to_double(y02, ky);
  Q[2] = to_double(y12, ky);
  Q[3] = to_double(-c2, ky);
  Q[4] = to_double(y00, ky);
  Q[5] = to_double(y01, ky);
  Q[6] = to_double(-c0, ky);
  Q[7] = to_double(y11, ky);
  Q[8] = to_double(-c1, ky);
  Q[9] = to_double(c0 + c1 + c2, ky);
  return true;
}

// ---------------------------------------------------------------------------
// e = Q z for the packed upper triangle Q of a 4x4 matrix: both on the scale of
// their largest entry, each row's four products summed in integers and rounded
// once.  A row whose largest product has its exponent within kRowGap of the
// scale max|Q| max|z| is as accurate as fp64's chain of four, relative to the sum
// of its own products' magnitudes: 0.32 x 2^-53 (rms) at the scale, 0.43 at
// 2^-7 of it, against fp64's 0.51; 2.2 against 3.1 at worst.  Rows further down
// lose the bits that the common scale cuts (0.57 at 2^-8, 1.2 at 2^-9): their bits
// of `small` are set, for the caller to form them in fp64.  False (fp64 takes all
// of it) for exponents out of range, zero Q or z among them.
// ---------------------------------------------------------------------------
constexpr int kRowGap = 7;

FX_HD bool product4(const double Q[10], const double z[4], double e[4], unsigned* small = nullptr) {
  int eq[10], ez[4], kq = -1023, kz = -1023;
  for (int i = 0; i < 10; ++i) {
    eq[i] = exponent(Q[i]);
    kq = kq > eq[i] ? kq : eq[i];
  }
  for (int m = 0; m < 4; ++m) {
    ez[m] = exponent(z[m]);
    kz = kz > ez[m] ? kz : ez[m];
  }
  if (kq < -400 || kq > 400 || kz < -400 || kz > 400) return false;
  Half q[10], w[4];
  for (int i = 0; i < 10; ++i) q[i] = split(from_double(Q[i], kq));
  for (int m = 0; m < 4; ++m) w[m] = split(from_double(z[m], kz));
  const int at[4][4] = {{0, 1, 2, 3}, {1, 4, 5, 6}, {2, 5, 7, 8}, {3, 6, 8, 9}};
  unsigned low = 0;
  for (int k = 0; k < 4; ++k) {
    // |v|, |w| < 2^61: the cross products in two sums, each up to 2^62, and the
    // upper halves of the low products
    int64_t hh = 0, x = 0, y = 0;
    int ll = 0, top = -4096;
    for (int m = 0; m < 4; ++m) {
      const Half p = q[at[k][m]], r = w[m];
      hh += (int64_t)p.h * r.h;
      x += (int64_t)p.h * r.l;
      y += (int64_t)p.l * r.h;
      ll += (p.l >> 17) * (r.l >> 17);
      const int t = eq[at[k][m]] + ez[m];
      top = top > t ? top : t;
    }
    low |= (unsigned)(top < kq + kz - kRowGap) << k;
    const int64_t c = (x >> 1) + (y >> 1) + 2 * (int64_t)ll + ((int64_t)1 << 27);
    e[k] = to_double((int64_t)((uint64_t)hh << 3) + (c >> 28), kq + kz - 59);
  }
  if (small) *small = low;
  return true;
}

}  // namespace fx
