// Mesh construction on the device: face-to-tetrahedron connectivity
// (Section 3.3), face / multiplier numbering, the CSR pattern of the condensed
// face system and per-element geometry.
//
// Connectivity.  The paper builds faces from edge-to-tet sparse maps
// (Listings EdgeNum2Tetra, FacesUp).  Here every local face becomes a key
// (v0 < v1 < v2) that is counting-sorted into buckets by its largest vertex v2
// (histogram, scan, scatter; mesh order keeps the scatter local; on refined
// meshes the largest vertex spreads keys more evenly than the smallest), and
// the keys of a bucket are matched against each other.  The result is the
// paper's numbering: a face's id is the rank of its first occurrence in
// (tet, local face) order and the tet of that occurrence is T+; it does not
// depend on the order of entries inside a bucket.
#include <math.h>
#include <string.h>

#include <functional>
#include <initializer_list>
#include <vector>


#include "element.cuh"
#include "ph_internal.cuh"

namespace {

__device__ __forceinline__ int comp(int4 v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// Local face k of T = [a b c d]: [a b c], [a c d], [a d b], [d c b] (Section 2.2).
__device__ __forceinline__ int3 local_face(int4 v, int k) {
  switch (k) {
    case 0: return make_int3(v.x, v.y, v.z);
    case 1: return make_int3(v.x, v.z, v.w);
    case 2: return make_int3(v.x, v.w, v.y);
    default: return make_int3(v.w, v.z, v.y);
  }
}

__device__ __forceinline__ int3 sort3(int3 a) {
  int x = a.x, y = a.y, z = a.z, t;
  if (y < x) { t = x; x = y; y = t; }
  if (z < y) { t = y; y = z; z = t; }
  if (y < x) { t = x; x = y; y = t; }
  return make_int3(x, y, z);
}

__device__ __forceinline__ bool valid_tet(int4 v, int64_t nC) {
  bool in = v.x >= 0 && v.y >= 0 && v.z >= 0 && v.w >= 0 && v.x < nC && v.y < nC && v.z < nC && v.w < nC;
  bool distinct = v.x != v.y && v.x != v.z && v.x != v.w && v.y != v.z && v.y != v.w && v.z != v.w;
  return in && distinct;
}

// True once an earlier kernel of this mesh recorded an error: the kernels
// after validation read ids produced by the earlier ones and must not touch
// memory through them then (the error is reported at the end of creation).
__device__ __forceinline__ bool failed(const unsigned* status) { return *status != 0; }

__device__ __forceinline__ bool valid_tri(int3 v, int64_t nC) {
  bool in = v.x >= 0 && v.y >= 0 && v.z >= 0 && v.x < nC && v.y < nC && v.z < nC;
  return in && v.x != v.y && v.x != v.z && v.y != v.z;
}

__device__ __forceinline__ int3 neumann_tri(const int32_t* nb, int64_t i) {
  return make_int3(nb[3 * i], nb[3 * i + 1], nb[3 * i + 2]);
}

// Bucket of a sorted face key (v0 < v1 < v2): the largest vertex and `sub`
// bits hashed from the other two, so a bucket holds about 2^-sub of the faces
// whose largest vertex is v2.  Hashing v0 as well as v1 matters: the faces
// around one edge (v1, v2) share both vertices, and bits of v1 alone leave
// them all in one bucket (long match scans).
__device__ __forceinline__ int64_t bucket_of(int3 s, int sub) {
  return ((int64_t)s.z << sub) | ((s.x ^ s.y) & ((1 << sub) - 1));
}

// Element geometry of tet t: the record (G_e, fixed point or fp64), its scale,
// |det E| and 1/|det E|.
__device__ __forceinline__ void tet_geom(const double* __restrict__ coord, int4 v, int64_t t, bool fixed,
                                         double* __restrict__ geo, int32_t* __restrict__ gexp,
                                         double2* __restrict__ vol, unsigned* status) {
  double e[3][3];
  ph_elem::edge_vectors(coord, v, e);
  const double adet = ph_elem::abs_det(e), rdet = ph::rcp_newton(adet);
  if (!ph::pos_finite(adet)) ph_flag(status, PH_ERR_DEGENERATE);
  ph_elem::Record r;
  if (!fixed || !fx::geometry(e, r.g, r.kg)) {
    double g[6];
    ph_elem::gram(e, g);
#pragma unroll
    for (int i = 0; i < 6; ++i) r.g[i] = __double_as_longlong(g[i]);
    r.kg = PH_GEXP_F64;
  }
  longlong2* o = reinterpret_cast<longlong2*>(geo + PH_GEO_STRIDE * t);
  o[0] = make_longlong2(r.g[0], r.g[1]);
  o[1] = make_longlong2(r.g[2], r.g[3]);
  o[2] = make_longlong2(r.g[4], r.g[5]);
  gexp[t] = r.kg;
  vol[t] = make_double2(adet, rdet);
}

// last p with off[p] <= i (off ascending, off[0] = 0)
__device__ __forceinline__ int problem_of(const int64_t* __restrict__ off, int32_t n, int64_t i) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// 1. histogram of face keys by bucket
__device__ __forceinline__ void face_count_item(int64_t i, const int4* __restrict__ tet, int64_t nE, int64_t nC, const int32_t* __restrict__ nb,
                             int64_t nN, int sub, int32_t* __restrict__ cnt, int4* __restrict__ tet_copy,
                             unsigned* status) {
  if (i < nE) {
    int4 v = tet[i];
    tet_copy[i] = v;  // the mesh's own copy of the input
    if (!valid_tet(v, nC)) { ph_flag(status, PH_ERR_ARG); return; }
#pragma unroll
    for (int k = 0; k < 4; ++k) atomicAdd(&cnt[bucket_of(sort3(local_face(v, k)), sub)], 1);
  } else if (i < nE + nN) {
    int3 f = neumann_tri(nb, i - nE);
    if (!valid_tri(f, nC)) { ph_flag(status, PH_ERR_ARG); return; }
    atomicAdd(&cnt[bucket_of(sort3(f), sub)], 1);
  }
}

__global__ void k_face_count(const int4* __restrict__ tet, int64_t nE, int64_t nC, const int32_t* __restrict__ nb,
                             int64_t nN, int sub, int32_t* __restrict__ cnt, int4* __restrict__ tet_copy,
                             unsigned* status) {
  face_count_item(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      tet, nE, nC, nb, nN, sub, cnt, tet_copy, status);
}

// 2. scatter keys into buckets: entry = (v0, v1, v2, slot), slot = 4t+k for
//    tet faces and 4nE+i for Neumann triples.  cnt counts down to 0.  The
//    same thread then computes the tet's geometry: G_e in fixed point on the
//    integer pipe (fixed.cuh), 22 FP64 operations where the fp64 record took
//    55 and bound the kernel.  Now the atomics, the scattered stores and the
//    geometry share it (17.9M tets: 1.94 -> 1.10 ms; 1.08 without the low
//    products, which cost graded elements accuracy).  Blocks of 128 threads, 6
//    per SM (80 registers): without those, 5 or 7 took 1.15 and 1.09 ms,
//    256-thread blocks at 96 registers 1.63; storing the entries after the
//    geometry instead of before it holds their stores back, 1.26.
constexpr int kFillThreads = 128;
template <bool GEO>
__device__ __forceinline__ void face_fill_item(int64_t i, const int4* __restrict__ tet, int64_t nE, int64_t nC, const int32_t* __restrict__ nb,
                            int64_t nN, int sub, const int32_t* __restrict__ start, int32_t* __restrict__ cnt,
                            int4* __restrict__ entries, int32_t* __restrict__ mate, const double* __restrict__ coord,
                            double* __restrict__ geo, int32_t* __restrict__ gexp, double2* __restrict__ vol,
                            const int64_t* __restrict__ toff, int32_t nprob, unsigned* status) {
  if (failed(status)) return;
  if (i < nE) {
    int4 v = tet[i];
    if (!valid_tet(v, nC)) return;
    int pos[4];  // four atomics in flight, then their stores
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t b = bucket_of(sort3(local_face(v, k)), sub);
      pos[k] = start[b] + atomicSub(&cnt[b], 1) - 1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int3 s = sort3(local_face(v, k));
      entries[pos[k]] = make_int4(s.x, s.y, s.z, (int)(4 * i + k));
    }
    reinterpret_cast<int4*>(mate)[i] = make_int4(-1, -1, -1, -1);  // no mate yet (boundary)
    if (!GEO) return;
    int64_t n = nE;  // tets of the tet's mesh
    if (toff) {
      const int p = problem_of(toff, nprob, i);
      n = toff[p + 1] - toff[p];
    }
    tet_geom(coord, v, i, n >= ph::kFixedMin, geo, gexp, vol, status);
  } else if (i < nE + nN) {
    int3 f = neumann_tri(nb, i - nE);
    if (!valid_tri(f, nC)) return;
    int3 s = sort3(f);
    const int64_t b = bucket_of(s, sub);
    int pos = start[b] + atomicSub(&cnt[b], 1) - 1;
    entries[pos] = make_int4(s.x, s.y, s.z, (int)i + 3 * (int)nE);  // slot 4nE + (i - nE)
  }
}

template <bool GEO>
__global__ void __launch_bounds__(kFillThreads, 6) k_face_fill(const int4* __restrict__ tet, int64_t nE, int64_t nC, const int32_t* __restrict__ nb,
                            int64_t nN, int sub, const int32_t* __restrict__ start, int32_t* __restrict__ cnt,
                            int4* __restrict__ entries, int32_t* __restrict__ mate, const double* __restrict__ coord,
                            double* __restrict__ geo, int32_t* __restrict__ gexp, double2* __restrict__ vol,
                            const int64_t* __restrict__ toff, int32_t nprob, unsigned* status) {
  face_fill_item<GEO>(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      tet, nE, nC, nb, nN, sub, start, cnt, entries, mate, coord, geo, gexp, vol, toff, nprob, status);
}

// Outcome of one entry's scan: a tet entry records its mate (and its mate's
// mate) or -2 for a Neumann triple; errors as in k_face_match.
__device__ __forceinline__ void settle_entry(int4 e, int ntet, int nt, int nn, int tm, int32_t* __restrict__ mate,
                                             unsigned* status) {
  if (e.w < ntet) {
    if (nt + nn >= 2) ph_flag(status, nn > 0 ? PH_ERR_ARG : PH_ERR_NONMANIFOLD);
    if (nt == 1) {
      mate[e.w] = tm;
      mate[tm] = e.w;
    } else if (nn == 1) {
      mate[e.w] = -2;
    }
  } else {
    if (nt != 1 || nn != 0) ph_flag(status, PH_ERR_ARG);
    else mate[tm] = -2;
  }
}

// k is an entry of e's bucket (same largest vertex) or the sentinel (-1, ...),
// which equals no entry
__device__ __forceinline__ void count_match(int4 k, int4 e, int ntet, int& nt, int& nn, int& tm) {
  if (k.x == e.x && k.y == e.y) {
    if (k.w < ntet) { ++nt; tm = k.w; } else { ++nn; }
  }
}

// 3. match equal keys inside a bucket.  A tet entry compares itself with the
//    LATER entries of its bucket only and writes both mates of a pair, so each
//    pair is found once (a second match marks a face in three tets, or a
//    Neumann triple on an interior face); Neumann entries (boundary only, few)
//    scan the whole bucket, themselves included (one Neumann hit taken off),
//    and must match exactly one tet entry.  Each thread takes two entries, i
//    and i + half, and scans their buckets in lockstep: two independent chains
//    of loads in flight per thread.  The kernel issues instructions at close
//    to the SM's rate, so the loop carries no more than the loads and
//    compares; the bucket hash keeps the scans short.
__device__ __forceinline__ void face_match_item(int64_t i0, const int4* __restrict__ entries, int64_t nent, const int32_t* __restrict__ start,
                             int sub, int64_t nE, int32_t* __restrict__ mate, unsigned* status) {
  const int64_t half = (nent + 1) >> 1;
  if (i0 >= half || failed(status)) return;
  const int64_t i1 = i0 + half;
  const bool has1 = i1 < nent;
  const int ntet = (int)(4 * nE);  // slots are int32
  const int4 none = make_int4(-1, -1, -1, -1);
  const int4 e0 = entries[i0];
  const int4 e1 = has1 ? entries[i1] : none;
  const int64_t b0 = bucket_of(make_int3(e0.x, e0.y, e0.z), sub);
  const int64_t b1 = has1 ? bucket_of(make_int3(e1.x, e1.y, e1.z), sub) : 0;
  const int end0 = start[b0 + 1], end1 = has1 ? start[b1 + 1] : 0;
  // tet entries scan the later entries of their bucket, Neumann entries all of it
  const bool nm0 = e0.w >= ntet, nm1 = has1 && e1.w >= ntet;
  int j0 = nm0 ? start[b0] : (int)i0 + 1;
  int j1 = has1 ? (nm1 ? start[b1] : (int)i1 + 1) : 0;
  int nt0 = 0, nn0 = nm0 ? -1 : 0, tm0 = -1, nt1 = 0, nn1 = nm1 ? -1 : 0, tm1 = -1;
  while (j0 < end0 || j1 < end1) {
    const int4 k0 = j0 < end0 ? entries[j0] : none;
    const int4 k1 = j1 < end1 ? entries[j1] : none;
    count_match(k0, e0, ntet, nt0, nn0, tm0);
    count_match(k1, e1, ntet, nt1, nn1, tm1);
    ++j0;
    ++j1;
  }
  settle_entry(e0, ntet, nt0, nn0, tm0, mate, status);
  if (has1) settle_entry(e1, ntet, nt1, nn1, tm1, mate, status);
}

__global__ void k_face_match(const int4* __restrict__ entries, int64_t nent, const int32_t* __restrict__ start,
                             int sub, int64_t nE, int32_t* __restrict__ mate, unsigned* status) {
  face_match_item(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      entries, nent, start, sub, nE, mate, status);
}

// 4. face bases: an exclusive scan of the number of first occurrences per tet,
//    which the scan itself counts from the mates (exclusive_scan's `mates`).
using ph::first_occurrence;

__device__ __forceinline__ int first_rank(int4 m, int s0, int k) {
  int r = 0;
  if (k > 0) r += first_occurrence(m.x, s0);
  if (k > 1) r += first_occurrence(m.y, s0 + 1);
  if (k > 2) r += first_occurrence(m.z, s0 + 2);
  return r;
}

// Face ids of tet t, given its tuple v, mates m, face base fb and, for each face
// it does not own, its owner's mates om[k] and face base ofb[k]; own(F, T-,
// tuple, kind) takes each face it owns (a first occurrence).  With tmult (no
// Neumann faces) also the slots' multiplier ids, l(F) = F.
template <class Own>
__device__ __forceinline__ void emit_tet(int64_t t, int4 v, int4 m, int fb, const int4 om[4], const int ofb[4],
                                         int4* __restrict__ tface, int4* __restrict__ tmult, const Own& own) {
  const int s0 = (int)(4 * t);
  int out[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int mk = comp(m, k);
    if (first_occurrence(mk, s0 + k)) {
      const int F = fb + first_rank(m, s0, k);
      out[k] = F;
      own(F, mk >= 0 ? (mk >> 2) : -1, local_face(v, k), mk >= 0 ? 0 : (mk == -1 ? 1 : 2));
    } else {
      const int t2 = mk >> 2, k2 = mk & 3;
      out[k] = (int)((unsigned)(ofb[k] + first_rank(om[k], 4 * t2, k2)) | 0x80000000u);
    }
  }
  tface[t] = make_int4(out[0], out[1], out[2], out[3]);
  if (tmult) {
    int o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = (int)((unsigned)(out[k] & PH_ID_MASK) | (comp(m, k) < 0 ? PH_BND_BIT : 0u));
    tmult[t] = make_int4(o[0], o[1], o[2], o[3]);
  }
}

// The owner's mates and face base for each face of a tet it does not own.
__device__ __forceinline__ void load_owners(int64_t t, int4 m, const int4* __restrict__ mate4,
                                            const int32_t* __restrict__ fbase, int4 om[4], int ofb[4]) {
  const int s0 = (int)(4 * t);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int mk = comp(m, k);
    if (!first_occurrence(mk, s0 + k)) {
      om[k] = mate4[mk >> 2];
      ofb[k] = fbase[mk >> 2];
    }
  }
}

// 5. per tet: face ids, and T+/T-, T+'s tuple, kind and non-Neumann flag of the
//    faces it owns (first occurrences).  Without Neumann faces (mult_iota
//    given) every face has a multiplier, l(F) = F, so the tet also writes its
//    slots' multiplier ids and, for the faces it owns, the row length 1 + 3
//    per tet of the face (7 interior, 4 boundary); k_tet_mult is not needed.
//    The faces owned by a block's tets are consecutive: they are staged in
//    shared memory and written in runs.  (Written by their tets, in up to 28
//    partly filled stores per warp, they bound the kernel by L1: 0.66 ms at
//    17.9M tets, now 0.47.)
constexpr int kEmitThreads = 256;

__global__ void __launch_bounds__(kEmitThreads) k_face_emit(
    const int4* __restrict__ tet, int64_t nE, const int4* __restrict__ mate4, const int32_t* __restrict__ fbase,
    int4* __restrict__ tface, int2* __restrict__ face_tet, int32_t* __restrict__ face_vtx,
    int8_t* __restrict__ face_kind, int32_t* __restrict__ flag, int32_t* __restrict__ mult_iota,
    int4* __restrict__ tmult, int32_t* __restrict__ rowlen, const unsigned* status) {
  __shared__ int2 s_tet[4 * kEmitThreads];
  __shared__ int32_t s_vtx[12 * kEmitThreads];
  __shared__ int8_t s_kind[4 * kEmitThreads];
  if (failed(status)) return;
  const int64_t first = blockIdx.x * (int64_t)kEmitThreads, t = first + threadIdx.x;
  const int base = fbase[first], count = fbase[min(first + kEmitThreads, nE)] - base;
  if (t < nE) {
    const int4 v = tet[t], m = mate4[t];
    const int fb = fbase[t];
    int4 om[4];
    int ofb[4];
    load_owners(t, m, mate4, fbase, om, ofb);
    emit_tet(t, v, m, fb, om, ofb, tface, mult_iota ? tmult : nullptr, [&](int F, int minus, int3 lf, int kind) {
      const int i = F - base;
      s_tet[i] = make_int2((int)t, minus);
      s_vtx[3 * i] = lf.x;
      s_vtx[3 * i + 1] = lf.y;
      s_vtx[3 * i + 2] = lf.z;
      s_kind[i] = (int8_t)kind;
    });
  }
  __syncthreads();
  const int nF = fbase[nE];
  for (int i = threadIdx.x; i < count; i += kEmitThreads) {
    const int F = base + i, kind = s_kind[i];
    face_tet[F] = s_tet[i];
    face_kind[F] = (int8_t)kind;
    if (flag) flag[F] = kind != 2;  // Neumann faces present: multipliers by a scan of the flags
    if (mult_iota) {                // none: l(F) = F
      mult_iota[F] = F;
      rowlen[F] = kind == 0 ? 7 : 4;
      if (F + 1 == nF) rowlen[F + 1] = 0;  // the scan reads one entry past the last row
    }
  }
  for (int i = threadIdx.x; i < 3 * count; i += kEmitThreads) face_vtx[3 * (int64_t)base + i] = s_vtx[i];
}

// The same for one tet, its faces written directly.
__device__ __forceinline__ void face_emit_item(int64_t t, const int4* tet, int64_t nE, const int4* mate4,
                                               const int32_t* fbase, int4* tface, int2* face_tet, int32_t* face_vtx,
                                               int8_t* face_kind, int32_t* flag, int32_t* mult_iota, int4* tmult,
                                               int32_t* rowlen, const unsigned* status) {
  if (failed(status)) return;
  const int nF = fbase[nE];
  const int4 m = mate4[t];
  int4 om[4];
  int ofb[4];
  load_owners(t, m, mate4, fbase, om, ofb);
  emit_tet(t, tet[t], m, fbase[t], om, ofb, tface, mult_iota ? tmult : nullptr, [&](int F, int minus, int3 lf, int kind) {
    face_tet[F] = make_int2((int)t, minus);
    face_vtx[3 * F] = lf.x;
    face_vtx[3 * F + 1] = lf.y;
    face_vtx[3 * F + 2] = lf.z;
    face_kind[F] = (int8_t)kind;
    if (flag) flag[F] = kind != 2;
    if (mult_iota) {
      mult_iota[F] = F;
      rowlen[F] = kind == 0 ? 7 : 4;
      if (F + 1 == nF) rowlen[F + 1] = 0;
    }
  });
}

// face area 1/2 |(P_z - P_x) x (P_y - P_x)| of the vertices p[0..2] = P_x, P_y,
// P_z
__device__ __forceinline__ double face_area(const double p[3][3]) {
  const double *x = p[0], *y = p[1], *z = p[2];
  double u0 = z[0] - x[0], u1 = z[1] - x[1], u2 = z[2] - x[2];
  double v0 = y[0] - x[0], v1 = y[1] - x[1], v2 = y[2] - x[2];
  double cx = u1 * v2 - u2 * v1, cy = u2 * v0 - u0 * v2, cz = u0 * v1 - u1 * v0;
  return ph::half_sqrt(cx * cx + cy * cy + cz * cz);
}

// Neumann faces get no multiplier.  Face counts are read on the device
// (d_tot[0] = nF), the grid covers the upper bound.
__device__ __forceinline__ void mult_fix_item(int64_t F, int32_t* __restrict__ face_mult, const int8_t* __restrict__ face_kind,
                           const int64_t* __restrict__ d_tot, int64_t nFmax, const unsigned* status) {
  if (F >= nFmax || F >= d_tot[0] || failed(status)) return;
  if (face_kind[F] == 2) face_mult[F] = -1;
}

__global__ void k_mult_fix(int32_t* __restrict__ face_mult, const int8_t* __restrict__ face_kind,
                           const int64_t* __restrict__ d_tot, int64_t nFmax, const unsigned* status) {
  mult_fix_item(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      face_mult, face_kind, d_tot, nFmax, status);
}

// 7. per-slot multiplier ids and row lengths: row l(F) = 1 + sum over F's
//    tets of (non-Neumann faces of the tet) - 1.
__device__ __forceinline__ void tet_mult_item(int64_t t, const int4* __restrict__ tface, int64_t nE, const int32_t* __restrict__ face_mult,
                           const int2* __restrict__ face_tet, int4* __restrict__ tmult, int32_t* __restrict__ rowlen,
                           const unsigned* status) {
  if (t >= nE || failed(status)) return;
  int4 tf = tface[t];
  int l[4], o[4];
  int mT = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    int F = comp(tf, k) & PH_ID_MASK;
    l[k] = face_mult[F];
    mT += l[k] >= 0;
    bool bnd = face_tet[F].y < 0;
    o[k] = l[k] < 0 ? PH_NO_MULT : (int)((unsigned)l[k] | (bnd ? PH_BND_BIT : 0u));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (l[k] >= 0) atomicAdd(&rowlen[l[k]], mT - 1 + (comp(tf, k) >= 0 ? 1 : 0));
  tmult[t] = make_int4(o[0], o[1], o[2], o[3]);
}

__global__ void k_tet_mult(const int4* __restrict__ tface, int64_t nE, const int32_t* __restrict__ face_mult,
                           const int2* __restrict__ face_tet, int4* __restrict__ tmult, int32_t* __restrict__ rowlen,
                           const unsigned* status) {
  tet_mult_item(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      tface, nE, face_mult, face_tet, tmult, rowlen, status);
}

// The other three local faces of a tet, m != k ascending, as multiplier ids
// (PH_NO_MULT, which sorts last, for Neumann faces or no tet).
__device__ __forceinline__ void other_mults(int4 tm, int k, int& o0, int& o1, int& o2) {
  int id[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int mj = comp(tm, j);
    id[j] = mj == PH_NO_MULT ? PH_NO_MULT : (mj & PH_ID_MASK);
  }
  o0 = k == 0 ? id[1] : id[0];
  o1 = k <= 1 ? id[2] : id[1];
  o2 = k <= 2 ? id[3] : id[2];
}

__device__ __forceinline__ void cswap(int& a, int& b) {
  const int lo = min(a, b), hi = max(a, b);
  a = lo;
  b = hi;
}

// number of entries of c[0..7) below x (the rank of x among distinct ids)
__device__ __forceinline__ int rank7(const int c[7], int x) {
  int r = 0;
#pragma unroll
  for (int i = 0; i < 7; ++i) r += c[i] < x;
  return r;
}

// 8. column indices of each row (ascending) and each slot's scatter positions:
//    tpos = diagonal, trel = rank offsets of the other three local faces (4-bit
//    two's complement, m != k ascending).
//    Row l(F) holds l(F) and the other non-Neumann faces of F's one or two
//    tets (all distinct): 7 candidates with PH_NO_MULT for absent ones, put in
//    order by a 16-comparator sorting network, all in registers.  The thread
//    also computes the face's area, whose 22 FP64 operations bound the kernel
//    (1.50 ms at 35.9M faces; with the product in fixed point 1.35, but see
//    fixed.cuh on the areas' last bits).  Its chains of gathers hide under the
//    FP64 pipe in any order: issuing all loads first changed nothing (1.49 ms
//    before).
// BATCH (a batched build): U holds the problems' offsets; the face's ids (in
// place), its column ids and positions are then local to its problem.
struct FillOffsets {
  const int64_t *toff, *voff;
  const long long* first;  // first face, multiplier, CSR entry
  int32_t n;
  int32_t* rowptr;  // the problems' own row pointers: L_p + 1 entries at first multiplier + p
};

template <bool BATCH, bool AREA>
__device__ __forceinline__ void row_fill_item(int64_t F, int2* __restrict__ face_tet, const int4* __restrict__ tface,
                           const int4* __restrict__ tmult, int32_t* __restrict__ face_mult,
                           const int64_t* __restrict__ d_tot, int64_t nFmax,
                           const int32_t* __restrict__ rowptr, int32_t* __restrict__ colind,
                           int32_t* __restrict__ tpos,
                           unsigned short* __restrict__ trel, const double* __restrict__ coord,
                           int32_t* __restrict__ face_vtx, double* __restrict__ area, const FillOffsets U,
                           unsigned* status) {
  if (F >= nFmax || F >= d_tot[0] || failed(status)) return;
  // every load whose address is known, before anything uses one
  const int2 ft = face_tet[F];
  const int l = face_mult[F];
  const int T[2] = {ft.x, ft.y};
  int vtx[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) vtx[j] = face_vtx[3 * F + j];
  int4 tf[2], tm[2];
#pragma unroll
  for (int side = 0; side < 2; ++side)
    if (T[side] >= 0) {
      tf[side] = tface[T[side]];
      tm[side] = tmult[T[side]];
    }
  double p[3][3];
  if (AREA)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int d = 0; d < 3; ++d) p[j][d] = coord[3 * (int64_t)vtx[j] + d];
  int base = 0, end = 0;
  if (l >= 0) {
    base = rowptr[l];
    end = rowptr[l + 1];
  }
  if (AREA) area[F] = face_area(p);
  int m0 = 0, z0 = 0;
  if (BATCH) {
    const int q = problem_of(U.toff, U.n, T[0]);
    const int t0 = (int)U.toff[q], v0 = (int)U.voff[q];
    m0 = (int)U.first[3 * q + 1];
    z0 = (int)U.first[3 * q + 2];
    face_tet[F] = make_int2(ft.x - t0, ft.y < 0 ? -1 : ft.y - t0);
#pragma unroll
    for (int j = 0; j < 3; ++j) face_vtx[3 * F + j] = vtx[j] - v0;
    if (l >= 0) {
      face_mult[F] = l - m0;
      if (l == m0) U.rowptr[l + q] = 0;
      U.rowptr[l + q + 1] = end - z0;
    }
  }
  if (l < 0) return;
  int k[2] = {0, 0};
  int o[2][3];
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    o[side][0] = o[side][1] = o[side][2] = PH_NO_MULT;
    if (T[side] < 0) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((comp(tf[side], j) & PH_ID_MASK) == F) k[side] = j;
    other_mults(tm[side], k[side], o[side][0], o[side][1], o[side][2]);
  }
  int c[7] = {l, o[0][0], o[0][1], o[0][2], o[1][0], o[1][1], o[1][2]};
  cswap(c[0], c[6]); cswap(c[2], c[3]); cswap(c[4], c[5]);
  cswap(c[0], c[2]); cswap(c[1], c[4]); cswap(c[3], c[6]);
  cswap(c[0], c[1]); cswap(c[2], c[5]); cswap(c[3], c[4]);
  cswap(c[1], c[2]); cswap(c[4], c[6]);
  cswap(c[2], c[3]); cswap(c[4], c[5]);
  cswap(c[1], c[2]); cswap(c[3], c[4]); cswap(c[5], c[6]);
  const int n = 7 - ((c[0] == PH_NO_MULT) + (c[1] == PH_NO_MULT) + (c[2] == PH_NO_MULT) + (c[3] == PH_NO_MULT) +
                     (c[4] == PH_NO_MULT) + (c[5] == PH_NO_MULT) + (c[6] == PH_NO_MULT));
  if (end - base != n) { ph_flag(status, PH_ERR_ARG); return; }
#pragma unroll
  for (int i = 0; i < 7; ++i)
    if (i < n) colind[base + i] = c[i] - m0;
  const int rl = rank7(c, l), diag = base + rl - z0;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    if (T[side] < 0) continue;
    unsigned bits = 0;
#pragma unroll
    for (int idx = 0; idx < 3; ++idx) {
      const int lm = o[side][idx];
      if (lm != PH_NO_MULT) bits |= ((unsigned)(rank7(c, lm) - rl) & 0xFu) << (4 * idx);
    }
    tpos[4 * (int64_t)T[side] + k[side]] = diag;
    trel[4 * (int64_t)T[side] + k[side]] = (unsigned short)bits;
  }
}

template <bool BATCH, bool AREA>
__global__ void __launch_bounds__(ph::kThreads, BATCH ? 4 : 5) k_row_fill(int2* __restrict__ face_tet, const int4* __restrict__ tface,
                           const int4* __restrict__ tmult, int32_t* __restrict__ face_mult,
                           const int64_t* __restrict__ d_tot, int64_t nFmax,
                           const int32_t* __restrict__ rowptr, int32_t* __restrict__ colind,
                           int32_t* __restrict__ tpos,
                           unsigned short* __restrict__ trel, const double* __restrict__ coord,
                           int32_t* __restrict__ face_vtx, double* __restrict__ area, const FillOffsets U,
                           unsigned* status) {
  row_fill_item<BATCH, AREA>(blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
      face_tet, tface, tmult, face_mult, d_tot, nFmax, rowptr, colind, tpos, trel, coord, face_vtx, area, U, status);
}


// ---------------------------------------------------------------------------
// Small meshes: the connectivity in one launch of one block, the geometry in
// another.  The nine launches above take 2.5 to 8 us each whatever they do (~60
// us with their gaps at 864 tets); here a phase costs its chain of L1 and L2
// trips.  The items are the kernels' own, so the result is theirs bit for bit.
// One block: a cluster would need the scans across its blocks, and the FP64
// work (97 operations per tet, 13 us on one SM at 864 tets) is what wants
// spreading, which k_small_geom does.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 1024;
constexpr int64_t kSmallTets = 1536, kSmallBuckets = 8192;

struct SmallMesh {
  const int4* tet_in;
  const double* coord_in;
  const int32_t* nb;
  int64_t nE, nC, nN;
  int sub;
  int64_t nbuckets;
  int32_t *cnt, *start, *newc, *flag, *rowlen;
  int4* entries;
  int32_t* mate;
  int64_t* d_tot;
  // the mesh's arrays
  double* coord;
  int4 *tet, *tface, *tmult;
  int2* face_tet;
  int32_t *face_vtx, *face_mult, *rowptr, *colind, *tpos;
  int8_t* face_kind;
  unsigned short* trel;
  double *geo, *face_area;
  int32_t* gexp;
  double2* vol;
  unsigned* status;
};

// Exclusive prefix sum of n values of in(i) into out, total returned, by the
// whole block (each thread a run of consecutive values).
template <class F>
__device__ __forceinline__ int small_scan(int64_t n, const F& in, int32_t* out) {
  __shared__ int warp_sum[kSmallThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t per = (n + kSmallThreads - 1) / kSmallThreads, lo = min(n, tid * per), hi = min(n, lo + per);
  int sum = 0;
  for (int64_t i = lo; i < hi; ++i) sum += in(i);
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) warp_sum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    int w = warp_sum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    warp_sum[lane] = w;
  }
  __syncthreads();
  const int total = warp_sum[kSmallThreads / 32 - 1];
  int run = inc - sum + (wid > 0 ? warp_sum[wid - 1] : 0);
  for (int64_t i = lo; i < hi; ++i) {
    const int v = in(i);  // out may be in's array: read before it is written
    out[i] = run;
    run += v;
  }
  __syncthreads();
  return total;
}

__global__ void __launch_bounds__(kSmallThreads) k_small_connect(const SmallMesh m) {
  const int tid = threadIdx.x;
  const int64_t nE = m.nE, nN = m.nN, nF4 = 4 * nE + nN;
  if (tid == 0) *m.status = 0;
  for (int64_t i = tid; i < m.nbuckets; i += kSmallThreads) m.cnt[i] = 0;
  for (int64_t i = tid; i < 3 * m.nC; i += kSmallThreads) m.coord[i] = m.coord_in[i];
  if (nN > 0)
    for (int64_t i = tid; i <= nF4; i += kSmallThreads) m.flag[i] = m.rowlen[i] = 0;
  __syncthreads();
  for (int64_t i = tid; i < nE + nN; i += kSmallThreads)
    face_count_item(i, m.tet_in, nE, m.nC, m.nb, nN, m.sub, m.cnt, m.tet, m.status);
  __syncthreads();
  if (failed(m.status)) {  // invalid ids: nothing may be read through them
    if (tid == 0) m.d_tot[0] = -1;
    return;
  }
  small_scan(m.nbuckets, [&](int64_t i) { return m.cnt[i]; }, m.start);
  for (int64_t i = tid; i < nE + nN; i += kSmallThreads)
    face_fill_item<false>(i, m.tet, nE, m.nC, m.nb, nN, m.sub, m.start, m.cnt, m.entries, m.mate, nullptr, nullptr,
                          nullptr, nullptr, nullptr, 0, m.status);
  __syncthreads();
  for (int64_t i = tid; i < (nF4 + 1) / 2; i += kSmallThreads)
    face_match_item(i, m.entries, nF4, m.start, m.sub, nE, m.mate, m.status);
  __syncthreads();
  const int4* mate4 = reinterpret_cast<const int4*>(m.mate);
  const int nF = small_scan(nE + 1, [&](int64_t i) { return i < nE ? ph::first_occurrences(mate4[i], (int)(4 * i)) : 0; },
                            m.newc);
  if (tid == 0) m.d_tot[0] = nF;
  for (int64_t i = tid; i < nE; i += kSmallThreads)
    face_emit_item(i, m.tet, nE, mate4, m.newc, m.tface, m.face_tet, m.face_vtx, m.face_kind, nN > 0 ? m.flag : nullptr,
                   nN > 0 ? nullptr : m.face_mult, m.tmult, m.rowlen, m.status);
  __syncthreads();
  int L = nF;
  if (nN > 0) {
    L = small_scan(nF + 1, [&](int64_t i) { return m.flag[i]; }, m.face_mult);
    for (int64_t F = tid; F < nF; F += kSmallThreads)
      mult_fix_item(F, m.face_mult, m.face_kind, m.d_tot, nF4, m.status);
    __syncthreads();
    for (int64_t t = tid; t < nE; t += kSmallThreads)
      tet_mult_item(t, m.tface, nE, m.face_mult, m.face_tet, m.tmult, m.rowlen, m.status);
    __syncthreads();
  }
  const int nnz = small_scan(L + 1, [&](int64_t i) { return m.rowlen[i]; }, m.rowptr);
  if (tid == 0) {
    m.d_tot[1] = L;
    m.d_tot[2] = nnz;
  }
  const FillOffsets none{nullptr, nullptr, nullptr, 0, nullptr};
  for (int64_t F = tid; F < nF; F += kSmallThreads)
    row_fill_item<false, false>(F, m.face_tet, m.tface, m.tmult, m.face_mult, m.d_tot, nF4, m.rowptr, m.colind, m.tpos,
                                m.trel, m.coord, m.face_vtx, m.face_area, none, m.status);
}

// The geometry of tet i < nE (also where a face did not match), or the area of
// face i - nE.
__global__ void __launch_bounds__(128) k_small_geom(const SmallMesh m) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nF = m.d_tot[0];
  if (nF < 0) return;
  if (i < m.nE) {
    tet_geom(m.coord, m.tet[i], i, m.nE >= ph::kFixedMin, m.geo, m.gexp, m.vol, m.status);
    return;
  }
  i -= m.nE;
  if (i >= nF || failed(m.status)) return;
  double p[3][3];
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int d = 0; d < 3; ++d) p[j][d] = m.coord[3 * (int64_t)m.face_vtx[3 * i + j] + d];
  m.face_area[i] = face_area(p);
}

__device__ __forceinline__ int shift_id(int x, int64_t off) {  // keep bit 31 (sigma / Dirichlet mark)
  return (int)(((unsigned)x & 0x80000000u) | (unsigned)((x & PH_ID_MASK) - (int)off));
}

// per tet of a batched build: local vertex ids, face ids, multiplier ids
// (k_row_fill has made the faces' and the CSR's local: separate passes over the
// 521M columns, 75M faces and 75M rows of 256 problems took 2.3, 0.7 and 0.4
// ms)
__global__ void k_rebase_tets(const FillOffsets o, int64_t nE, int4* __restrict__ tet, int4* __restrict__ tface,
                              int4* __restrict__ tmult, const unsigned* status) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nE || failed(status)) return;
  const int p = problem_of(o.toff, o.n, t);
  const int v = (int)o.voff[p];
  const int64_t f = o.first[3 * p], mo = o.first[3 * p + 1];
  const int4 a = tet[t];
  tet[t] = make_int4(a.x - v, a.y - v, a.z - v, a.w - v);
  const int4 b = tface[t];
  tface[t] = make_int4(shift_id(b.x, f), shift_id(b.y, f), shift_id(b.z, f), shift_id(b.w, f));
  const int4 c = tmult[t];
  int cm[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (cm[k] != PH_NO_MULT) cm[k] = shift_id(cm[k], mo);
  tmult[t] = make_int4(cm[0], cm[1], cm[2], cm[3]);
}

__global__ void k_face_centroid(const double* __restrict__ coord, const int32_t* __restrict__ face_vtx, int64_t nF,
                                double* __restrict__ out) {
  int64_t F = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (F >= nF) return;
  const double* x = coord + 3 * (int64_t)face_vtx[3 * F];
  const double* y = coord + 3 * (int64_t)face_vtx[3 * F + 1];
  const double* z = coord + 3 * (int64_t)face_vtx[3 * F + 2];
#pragma unroll
  for (int d = 0; d < 3; ++d) out[3 * F + d] = (x[d] + y[d] + z[d]) / 3.0;
}

struct Counters {
  int64_t total;
  unsigned status;
  unsigned pad;
};

}  // namespace

using namespace ph;

static void mesh_free(ph_mesh* m, cudaStream_t s) {
  if (!m) return;
  if (m->shared) {
    if (m->shared->refs.fetch_sub(1) == 1) {
      free_async(m->shared->arena, s);
      delete m->shared;
    }
  } else {
    free_async(m->arena, s);
  }
  delete m;
}

// Offsets of the problems of a batched build (the union mesh of
// ph_mesh_create_batch), one thread per problem.  Problem p owns tets
// [toff[p], toff[p+1]); its faces, multipliers and CSR entries are
// contiguous, and start at: the face of its first tet's first local face
// (always a first occurrence), the multiplier of the first non-Neumann face at
// or after it (Neumann faces have none; the walk may run into the next
// problem's faces, whose first multiplier is then this problem's end, which is
// also its start when it has no multiplier), and that row's first CSR entry.
// An empty problem gets -1 (the host takes the next problem's offsets).
__global__ void k_batch_offsets(const int4* __restrict__ tface, const int32_t* __restrict__ face_mult,
                                const int32_t* __restrict__ rowptr, const int64_t* __restrict__ d_tot,
                                const int64_t* __restrict__ toff, int32_t n, long long* __restrict__ out,
                                const unsigned* status) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  long long f0 = -1, m0 = -1, z0 = -1;
  if (toff[p + 1] > toff[p] && !failed(status)) {
    const int64_t nF = d_tot[0], L = d_tot[1];
    f0 = tface[toff[p]].x & PH_ID_MASK;
    int64_t F = f0;
    while (F < nF && face_mult[F] < 0) ++F;
    m0 = F < nF ? face_mult[F] : L;
    z0 = rowptr[m0];
  }
  out[3 * p] = f0;
  out[3 * p + 1] = m0;
  out[3 * p + 2] = z0;
}

// Hook of a batched build: the union's inputs, and the per-problem offsets,
// computed before the build's one synchronisation and read with it.
struct BatchCounts {
  // called once the mesh's own memory is allocated: sets the input arrays and
  // the pointers below.  (Memory of a mesh freed just before, its kernels still
  // running, is reused by the stream only if the largest block is asked for
  // first: with the inputs before it the pool mapped 14 GB anew, 5 ms a build.)
  std::function<ph_status(const double** coord, const int32_t** tet, const int32_t** neumann)> inputs;
  const int64_t *d_toff, *d_voff;  // n + 1 tet and vertex offsets (device)
  int32_t n;
  long long* d_counts;  // 3n: first face, multiplier, CSR entry of each problem
  long long* h_counts;  // 3n (host)
  int32_t* rowptr;      // out: the problems' row pointers (device, in the mesh's allocation)
};

// Synchronise and read n device int64 counters and the status word.
static ph_status read_counters(const int64_t* d_tot, int n, unsigned* d_status, cudaStream_t s, int64_t* tot,
                               unsigned* status) {
  cudaError_t e = cudaMemcpyAsync(tot, d_tot, sizeof(int64_t) * n, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(status, d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return cuda_status(e, "mesh_create sync");
}

#define PH_TRY(expr)                    \
  do {                                  \
    st = (expr);                        \
    if (st != PH_OK) goto fail;         \
  } while (0)
#define PH_CU(expr, what) PH_TRY(cuda_status((expr), what))

static ph_status mesh_build(const double* coord, int64_t nC, const int32_t* tet, int64_t nE, const int32_t* neumann,
                            int64_t nN, cudaStream_t s, ph_mesh** out, BatchCounts* bc, bool dw = false);

extern "C" ph_status ph_mesh_create(const double* coord, int64_t nC, const int32_t* tet, int64_t nE,
                                    const int32_t* neumann, int64_t nN, void* stream, ph_mesh** out) {
  return mesh_build(coord, nC, tet, nE, neumann, nN, (cudaStream_t)stream, out, nullptr);
}

extern "C" ph_status ph_mesh_create_dw(const double* coord, int64_t nC, const int32_t* tet, int64_t nE,
                                       const int32_t* neumann, int64_t nN, void* stream, ph_mesh** out) {
  return mesh_build(coord, nC, tet, nE, neumann, nN, (cudaStream_t)stream, out, nullptr, true);
}

static ph_status mesh_build(const double* coord, int64_t nC, const int32_t* tet, int64_t nE, const int32_t* neumann,
                            int64_t nN, cudaStream_t s, ph_mesh** out, BatchCounts* bc, bool dw) {
  if (!out) return PH_ERR_ARG;
  *out = nullptr;
  if (nE < 0 || nC < 0 || nN < 0) return PH_ERR_ARG;
  if (!bc && ((nE > 0 && (!coord || !tet)) || (nN > 0 && !neumann))) return PH_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(tet) & 15u) != 0) return PH_ERR_ARG;  // read as int4
  // Face arrays are sized by nFmax = 4 nE + nN >= nF and the CSR columns by
  // nFmax + 12 nE >= nnz, so the whole construction is enqueued at once and
  // synchronises once, at the end; int32 ids and CSR positions bound the size.
  const int64_t nFmax = 4 * nE + nN, nnzmax = nFmax + 12 * nE;
  if (nnzmax >= ((int64_t)1 << 31) - 1 || nC >= ((int64_t)1 << 31) - 1) return PH_ERR_OVERFLOW;
  ph_status st = PH_OK;  // everything runs in order on the caller's stream s
  // face-key buckets: 4 per largest vertex while the bucket ids stay below 2^31
  // (finer buckets shorten the match scans but cost more in the scattered
  // fill and the bucket scan than they save)
  const int sub = nC < ((int64_t)1 << 28) ? 2 : 0;
  const int64_t nb = (nC << sub) + 1;
  const int64_t nent = nFmax;
  const unsigned gF = grid_for(nFmax + 1);
  ph_mesh* m = new ph_mesh();
  memset(m, 0, sizeof *m);
  int64_t tot[3] = {0, 0, 0};
  unsigned bits = 0;
  // Two allocations: the mesh's arrays, and the scratch of the build (its
  // first part zeroed by one memset).  Few host calls keep the GPU fed.
  Carve mc, sc;
  const size_t o_status = mc.take<unsigned>(1), o_coord = mc.take<double>(3 * nC), o_tet = mc.take<int4>(nE);
  const size_t o_geo = mc.take<double>(PH_GEO_STRIDE * nE), o_tface = mc.take<int4>(nE);
  const size_t o_gexp = mc.take<int32_t>(nE), o_vol = mc.take<double2>(nE);
  const size_t o_tmult = mc.take<int4>(nE), o_tpos = mc.take<int4>(nE), o_trel = mc.take<ushort4>(nE);
  const size_t o_ftet = mc.take<int2>(nFmax), o_fvtx = mc.take<int32_t>(3 * nFmax);
  const size_t o_fkind = mc.take<int8_t>(nFmax), o_fmult = mc.take<int32_t>(nFmax + 1);
  const size_t o_farea = mc.take<double>(nFmax), o_rowptr = mc.take<int32_t>(nFmax + 1);
  const size_t o_colind = mc.take<int32_t>(nnzmax), o_rowptr_b = mc.take<int32_t>(bc ? nFmax + bc->n : 0);
  // scratch: zeroed part first
  const size_t o_tot = sc.take<int64_t>(3), o_cnt = sc.take<int32_t>(nb);
  const size_t o_s1 = sc.take<unsigned long long>(scan_state_words(nb));
  const size_t o_s2 = sc.take<unsigned long long>(scan_state_words(nE + 1));
  const size_t o_s3 = sc.take<unsigned long long>(scan_state_words(nFmax + 1));
  const size_t o_s4 = sc.take<unsigned long long>(scan_state_words(nFmax + 1));
  const size_t o_rowlen = sc.take<int32_t>(nN > 0 || nE == 0 ? nFmax + 1 : 0);  // else written by k_face_emit
  const size_t o_flag = sc.take<int32_t>(nN > 0 ? nFmax + 1 : 0);
  const size_t zero_bytes = sc.bytes;
  const size_t o_start = sc.take<int32_t>(nb), o_entries = sc.take<int4>(nent), o_mate = sc.take<int32_t>(4 * nE);
  const size_t o_newc = sc.take<int32_t>(nE + 1);
  const size_t o_rowlen2 = sc.take<int32_t>(nN > 0 || nE == 0 ? 0 : nFmax + 1);
  void* scratch = nullptr;
  PH_CU(cudaGetDevice(&m->device), "cudaGetDevice");
  m->nE = nE;
  m->nC = nC;
  PH_CU(alloc_bytes(&m->arena, mc.bytes, s), "alloc mesh");
  if (bc) PH_TRY(bc->inputs(&coord, &tet, &neumann));
  PH_CU(alloc_bytes(&scratch, sc.bytes, s), "alloc scratch");
  {
    void* A = m->arena;
    m->status = Carve::at<unsigned>(A, o_status);
    m->coord = Carve::at<double>(A, o_coord);
    m->tet = Carve::at<int4>(A, o_tet);
    m->geo = Carve::at<double>(A, o_geo);
    m->gexp = Carve::at<int32_t>(A, o_gexp);
    m->vol = Carve::at<double2>(A, o_vol);
    m->tface = Carve::at<int4>(A, o_tface);
    m->tmult = Carve::at<int4>(A, o_tmult);
    m->tpos = Carve::at<int4>(A, o_tpos);
    m->trel = Carve::at<ushort4>(A, o_trel);
    m->face_tet = Carve::at<int2>(A, o_ftet);
    m->face_vtx = Carve::at<int32_t>(A, o_fvtx);
    m->face_kind = Carve::at<int8_t>(A, o_fkind);
    m->face_mult = Carve::at<int32_t>(A, o_fmult);
    m->face_area = Carve::at<double>(A, o_farea);
    m->rowptr = Carve::at<int32_t>(A, o_rowptr);
    m->colind = Carve::at<int32_t>(A, o_colind);
    if (bc) bc->rowptr = Carve::at<int32_t>(A, o_rowptr_b);
  }
  {
  int64_t* d_tot = Carve::at<int64_t>(scratch, o_tot);  // [0] nF, [1] L, [2] nnz
  int32_t* cnt = Carve::at<int32_t>(scratch, o_cnt);
  int32_t* newc = Carve::at<int32_t>(scratch, o_newc);
  int32_t* start = Carve::at<int32_t>(scratch, o_start);
  int4* entries = Carve::at<int4>(scratch, o_entries);
  int32_t* mate = Carve::at<int32_t>(scratch, o_mate);
  int32_t* flag = nN > 0 ? Carve::at<int32_t>(scratch, o_flag) : nullptr;
  int32_t* rowlen = Carve::at<int32_t>(scratch, (nN > 0 || nE == 0) ? o_rowlen : o_rowlen2);
  unsigned long long* st1 = Carve::at<unsigned long long>(scratch, o_s1);
  unsigned long long* st2 = Carve::at<unsigned long long>(scratch, o_s2);
  unsigned long long* st3 = Carve::at<unsigned long long>(scratch, o_s3);
  unsigned long long* st4 = Carve::at<unsigned long long>(scratch, o_s4);
  if (!bc && nE > 0 && nE <= kSmallTets && nb <= kSmallBuckets && nN <= 4 * nE) {
    const SmallMesh sm{reinterpret_cast<const int4*>(tet), coord, neumann, nE, nC, nN, sub, nb, cnt, start, newc, flag,
                       rowlen, entries, mate, d_tot, m->coord, m->tet, m->tface, m->tmult, m->face_tet, m->face_vtx,
                       m->face_mult, m->rowptr, m->colind, reinterpret_cast<int32_t*>(m->tpos), m->face_kind,
                       reinterpret_cast<unsigned short*>(m->trel), m->geo, m->face_area, m->gexp, m->vol, m->status};
    {
      KernelTimer kt("k_small_connect", s, 2);
      k_small_connect<<<1, kSmallThreads, 0, s>>>(sm);
      PH_CU(launched(), "k_small_connect");
    }
    {
      KernelTimer kt("k_small_geom", s, 2);
      k_small_geom<<<grid_for(nE + nFmax, 128), 128, 0, s>>>(sm);
      PH_CU(launched(), "k_small_geom");
    }
    PH_TRY(read_counters(d_tot, 3, m->status, s, tot, &bits));
    goto built;
  }
  PH_CU(cudaMemsetAsync(scratch, 0, zero_bytes, s), "memset");
  PH_CU(cudaMemsetAsync(m->status, 0, sizeof(unsigned), s), "memset");
  if (nC > 0) PH_CU(cudaMemcpyAsync(m->coord, coord, sizeof(double) * 3 * nC, cudaMemcpyDeviceToDevice, s), "copy");

  // --- faces: bucket the keys, match them, number the faces ----------------
  if (nent > 0) {
    KernelTimer kt("k_face_count", s, 2);
    k_face_count<<<grid_for(nE + nN), kThreads, 0, s>>>(reinterpret_cast<const int4*>(tet), nE, nC, neumann, nN,
                                                        sub, cnt, m->tet, m->status);
    PH_CU(launched(), "k_face_count");
  }
  PH_TRY(exclusive_scan(cnt, start, nb, d_tot, s, m->status, nullptr, 0, st1));
  if (nent > 0) {
    {
      KernelTimer kt("k_face_fill", s, 2);
      k_face_fill<true><<<grid_for(nE + nN, kFillThreads), kFillThreads, 0, s>>>(m->tet, nE, nC, neumann, nN, sub, start, cnt, entries,
                                                         mate, m->coord, m->geo, m->gexp, m->vol, bc ? bc->d_toff : nullptr, bc ? bc->n : 0,
                                                                 m->status);
      PH_CU(launched(), "k_face_fill");
    }
    {
      KernelTimer kt("k_face_match", s, 2);
      k_face_match<<<grid_for((nent + 1) / 2), kThreads, 0, s>>>(entries, nent, start, sub, nE, mate, m->status);
      PH_CU(launched(), "k_face_match");
    }
  }
  // face bases: the scan counts each tet's first occurrences from the mates
  PH_TRY(exclusive_scan(nullptr, newc, nE + 1, d_tot, s, m->status, nullptr, 0, st2,
                        reinterpret_cast<const int4*>(mate), nE));  // nF -> d_tot[0]
  if (nE > 0) {
    KernelTimer kt("k_face_emit", s, 2);
    k_face_emit<<<grid_for(nE, kEmitThreads), kEmitThreads, 0, s>>>(
        m->tet, nE, reinterpret_cast<int4*>(mate), newc, m->tface, m->face_tet, m->face_vtx, m->face_kind, flag,
        nN > 0 ? nullptr : m->face_mult, m->tmult, rowlen, m->status);
    PH_CU(launched(), "k_face_emit");
  }

  // --- multipliers and CSR pattern (rows sized by nFmax >= L) ---------------
  if (nN > 0) {
    PH_TRY(exclusive_scan(flag, m->face_mult, nFmax + 1, d_tot + 1, s, m->status, d_tot, 1, st3));  // L -> d_tot[1]
    k_mult_fix<<<gF, kThreads, 0, s>>>(m->face_mult, m->face_kind, d_tot, nFmax, m->status);
    PH_CU(launched(), "k_mult_fix");
    if (nE > 0) {
      k_tet_mult<<<grid_for(nE), kThreads, 0, s>>>(m->tface, nE, m->face_mult, m->face_tet, m->tmult, rowlen,
                                                   m->status);
      PH_CU(launched(), "k_tet_mult");
    }
  } else {  // every face has a multiplier (k_face_emit wrote them, the slots' ids and the row lengths): L = nF
    PH_CU(cudaMemcpyAsync(d_tot + 1, d_tot, sizeof(int64_t), cudaMemcpyDeviceToDevice, s), "copy");
  }
  PH_TRY(exclusive_scan(rowlen, m->rowptr, nFmax + 1, d_tot + 2, s, m->status, d_tot + 1, 1, st4));  // nnz

  if (bc && bc->n > 0) {  // per-problem offsets of a batched build
    k_batch_offsets<<<grid_for(bc->n), kThreads, 0, s>>>(m->tface, m->face_mult, m->rowptr, d_tot, bc->d_toff, bc->n,
                                                         bc->d_counts, m->status);
    PH_CU(launched(), "k_batch_offsets");
  }

  // --- CSR columns and scatter positions (slots without a multiplier are never read)
  if (nFmax > 0) {
    KernelTimer kt("k_row_fill", s, 2);
    const auto fill = bc ? k_row_fill<true, true> : k_row_fill<false, true>;
    FillOffsets U{nullptr, nullptr, nullptr, 0, nullptr};
    if (bc) U = FillOffsets{bc->d_toff, bc->d_voff, bc->d_counts, bc->n, bc->rowptr};
    fill<<<gF, kThreads, 0, s>>>(m->face_tet, m->tface, m->tmult, m->face_mult, d_tot, nFmax, m->rowptr, m->colind,
                                 reinterpret_cast<int32_t*>(m->tpos), reinterpret_cast<unsigned short*>(m->trel),
                                 m->coord, m->face_vtx, m->face_area,
                                 U, m->status);
    PH_CU(launched(), "k_row_fill");
  }
  if (bc && nE > 0) {
    k_rebase_tets<<<grid_for(nE), kThreads, 0, s>>>(
        FillOffsets{bc->d_toff, bc->d_voff, bc->d_counts, bc->n, bc->rowptr}, nE, m->tet, m->tface, m->tmult, m->status);
    PH_CU(launched(), "k_rebase_tets");
  }
  if (bc && bc->n > 0)
    PH_CU(cudaMemcpyAsync(bc->h_counts, bc->d_counts, sizeof(long long) * 3 * bc->n, cudaMemcpyDeviceToHost, s),
          "copy");
  // the one synchronisation: counts and the first error of any kernel
  PH_TRY(read_counters(d_tot, 3, m->status, s, tot, &bits));
  }
built:
  free_async(scratch, s);
  scratch = nullptr;
  if (bits) {
    // a degenerate tet goes before a face that does not match, also where the
    // faces are matched first (k_small_connect)
    st = bits & (1u << PH_ERR_DEGENERATE) ? PH_ERR_DEGENERATE : status_from_bits(bits);
    goto fail;
  }
  m->nF = tot[0];
  m->L = tot[1];
  m->nnz = tot[2];
  // face kinds: every interior face has two slots and a boundary face one,
  // so 4 nE = 2 nFi + (nF - nFi); Neumann faces are the ones without multiplier
  m->nFi = 4 * nE - m->nF;
  m->nFn = m->nF - m->L;
  m->nFd = m->nF - m->nFi - m->nFn;
  m->geo_dw = dw;
  *out = m;
  return PH_OK;

fail:
  free_async(scratch, s);
  mesh_free(m, s);
  return st;
}

extern "C" ph_status ph_mesh_destroy(ph_mesh* mesh, void* stream) {
  if (!mesh) return PH_OK;
  mesh_free(mesh, (cudaStream_t)stream);
  return PH_OK;
}

extern "C" ph_status ph_mesh_info(const ph_mesh* m, ph_info* out) {
  if (!m || !out) return PH_ERR_ARG;
  out->nE = m->nE;
  out->nC = m->nC;
  out->nF = m->nF;
  out->nF_interior = m->nFi;
  out->nF_dirichlet = m->nFd;
  out->nF_neumann = m->nFn;
  out->L = m->L;
  out->nnz = m->nnz;
  return PH_OK;
}

extern "C" ph_status ph_mesh_faces(const ph_mesh* m, int32_t* tet_face, int32_t* face_tet, int32_t* face_vtx,
                                   int8_t* face_kind, int32_t* face_mult, double* face_centroid, double* face_area,
                                   void* stream) {
  if (!m) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  const int64_t nE = m->nE, nF = m->nF;
  if (tet_face && nE) e = cudaMemcpyAsync(tet_face, m->tface, sizeof(int4) * nE, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_tet && nF)
    e = cudaMemcpyAsync(face_tet, m->face_tet, sizeof(int2) * nF, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_vtx && nF)
    e = cudaMemcpyAsync(face_vtx, m->face_vtx, sizeof(int32_t) * 3 * nF, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_kind && nF)
    e = cudaMemcpyAsync(face_kind, m->face_kind, nF, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_mult && nF)
    e = cudaMemcpyAsync(face_mult, m->face_mult, sizeof(int32_t) * nF, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_area && nF)
    e = cudaMemcpyAsync(face_area, m->face_area, sizeof(double) * nF, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && face_centroid && nF) {
    k_face_centroid<<<grid_for(nF), kThreads, 0, s>>>(m->coord, m->face_vtx, nF, face_centroid);
    e = launched();
  }
  return cuda_status(e, "ph_mesh_faces");
}

extern "C" ph_status ph_csr_pattern(const ph_mesh* m, int32_t* rowptr, int32_t* colind, void* stream) {
  if (!m || !rowptr || (m->nnz > 0 && !colind)) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(rowptr, m->rowptr, sizeof(int32_t) * (m->L + 1), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && m->nnz)
    e = cudaMemcpyAsync(colind, m->colind, sizeof(int32_t) * m->nnz, cudaMemcpyDeviceToDevice, s);
  return cuda_status(e, "ph_csr_pattern");
}

extern "C" ph_status ph_mesh_check(ph_mesh* m, void* stream) {
  if (!m) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned bits = 0;
  cudaError_t e = cudaMemcpyAsync(&bits, m->status, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->status, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_status(e, "ph_mesh_check");
  return status_from_bits(bits);
}

// ---------------------------------------------------------------------------
// Batched build: n meshes at once.  Their disjoint union (vertex ids of
// problem p shifted by the vertices of the problems before it) is built as one
// mesh: faces of different problems never match, and the first-occurrence
// numbering of the union, restricted to problem p, is p's own numbering
// shifted by the faces of the problems before it (p's tets are consecutive);
// the same holds for multipliers, CSR rows and CSR entries.  So one build
// gives every problem's connectivity; a rebase pass then subtracts each
// problem's offsets, and the per-problem meshes are views into the union's
// memory with local ids, bit-identical to building each alone.
// ---------------------------------------------------------------------------
namespace {

struct UnionSources {
  const int32_t* tet;  // problem's tets (nE_p x 4)
  const int32_t* nb;   // problem's Neumann triples or null
};

// union tets and Neumann triples: problem p's ids shifted by voff[p].  An id
// outside [0, nC_p) would land on another problem's vertex, so it becomes -1,
// which the union build rejects (PH_ERR_ARG).
__device__ __forceinline__ int shift_vertex(int x, int v, int nv) { return (x >= 0 && x < nv) ? x + v : -1; }

__global__ void k_union_inputs(const UnionSources* __restrict__ src, const int64_t* __restrict__ toff,
                               const int64_t* __restrict__ noff, const int64_t* __restrict__ voff, int32_t n,
                               int64_t nE, int64_t nN, int4* __restrict__ tet_u, int32_t* __restrict__ nb_u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < nE) {
    const int p = problem_of(toff, n, i);
    const int v = (int)voff[p], nv = (int)(voff[p + 1] - voff[p]);
    const int4 t = reinterpret_cast<const int4*>(src[p].tet)[i - toff[p]];
    tet_u[i] = make_int4(shift_vertex(t.x, v, nv), shift_vertex(t.y, v, nv), shift_vertex(t.z, v, nv),
                         shift_vertex(t.w, v, nv));
  } else if (i < nE + nN) {
    const int64_t j = i - nE;
    const int p = problem_of(noff, n, j);
    const int v = (int)voff[p], nv = (int)(voff[p + 1] - voff[p]);
    const int64_t k = j - noff[p];
    nb_u[3 * j] = shift_vertex(src[p].nb[3 * k], v, nv);
    nb_u[3 * j + 1] = shift_vertex(src[p].nb[3 * k + 1], v, nv);
    nb_u[3 * j + 2] = shift_vertex(src[p].nb[3 * k + 2], v, nv);
  }
}


}  // namespace

extern "C" ph_status ph_mesh_create_batch(int32_t n, const double* const* coord, const int64_t* nC,
                                          const int32_t* const* tet, const int64_t* nE,
                                          const int32_t* const* neumann, const int64_t* nN, void* stream,
                                          ph_mesh** out) {
  if (n < 0 || !out || (n > 0 && (!coord || !nC || !tet || !nE))) return PH_ERR_ARG;
  for (int32_t p = 0; p < n; ++p) out[p] = nullptr;
  if (n == 0) return PH_OK;
  cudaStream_t s = (cudaStream_t)stream;
  // host offsets: tets, Neumann triples, vertices
  std::vector<int64_t> toff(n + 1, 0), noff(n + 1, 0), voff(n + 1, 0);
  std::vector<UnionSources> src(n);
  for (int32_t p = 0; p < n; ++p) {
    const int64_t np = nN ? nN[p] : 0;
    if (nE[p] < 0 || nC[p] < 0 || np < 0 || (nE[p] > 0 && (!coord[p] || !tet[p])) ||
        (np > 0 && (!neumann || !neumann[p])) || (reinterpret_cast<uintptr_t>(tet[p]) & 15u) != 0)
      return PH_ERR_ARG;
    toff[p + 1] = toff[p] + nE[p];
    noff[p + 1] = noff[p] + np;
    voff[p + 1] = voff[p] + nC[p];
    src[p] = UnionSources{tet[p], np > 0 ? neumann[p] : nullptr};
  }
  const int64_t nEu = toff[n], nNu = noff[n], nCu = voff[n];
  if (16 * nEu + nNu >= ((int64_t)1 << 31) - 1 || nCu >= ((int64_t)1 << 31) - 1) return PH_ERR_OVERFLOW;
  void* in = nullptr;
  std::vector<long long> cnt(3 * (size_t)n, -1);
  BatchCounts bc;
  bc.n = n;
  bc.h_counts = cnt.data();
  bc.rowptr = nullptr;
  std::vector<int64_t> offs;
  bc.inputs = [&](const double** coord_out, const int32_t** tet_out, const int32_t** nb_out) {
    // union inputs and the offset tables in one allocation
    Carve ic;
    const size_t o_coord = ic.take<double>(3 * nCu), o_tet = ic.take<int4>(nEu), o_nb = ic.take<int32_t>(3 * nNu);
    const size_t o_src = ic.take<UnionSources>(n), o_off = ic.take<int64_t>(3 * (n + 1));
    const size_t o_cnt = ic.take<long long>(3 * n);
    cudaError_t e = alloc_bytes(&in, ic.bytes, s);
    if (e != cudaSuccess) return cuda_status(e, "alloc batch inputs");
    double* coord_u = Carve::at<double>(in, o_coord);
    int4* tet_u = Carve::at<int4>(in, o_tet);
    int32_t* nb_u = Carve::at<int32_t>(in, o_nb);
    UnionSources* d_src = Carve::at<UnionSources>(in, o_src);
    int64_t* d_off = Carve::at<int64_t>(in, o_off);  // toff, noff, voff
    offs.insert(offs.end(), toff.begin(), toff.end());
    offs.insert(offs.end(), noff.begin(), noff.end());
    offs.insert(offs.end(), voff.begin(), voff.end());
    for (int32_t p = 0; p < n && e == cudaSuccess; ++p)
      if (nC[p] > 0)
        e = cudaMemcpyAsync(coord_u + 3 * voff[p], coord[p], sizeof(double) * 3 * nC[p], cudaMemcpyDeviceToDevice, s);
    // pageable sources: the copies return once the data is staged
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_src, src.data(), sizeof(UnionSources) * n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(d_off, offs.data(), sizeof(int64_t) * offs.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && nEu + nNu > 0) {
      k_union_inputs<<<grid_for(nEu + nNu), kThreads, 0, s>>>(d_src, d_off, d_off + (n + 1), d_off + 2 * (n + 1), n, nEu,
                                                            nNu, tet_u, nb_u);
      e = launched();
    }
    bc.d_toff = d_off;
    bc.d_voff = d_off + 2 * (n + 1);
    bc.d_counts = Carve::at<long long>(in, o_cnt);
    *coord_out = coord_u;
    *tet_out = reinterpret_cast<const int32_t*>(tet_u);
    *nb_out = nNu > 0 ? nb_u : nullptr;
    return cuda_status(e, "ph_mesh_create_batch inputs");
  };
  ph_mesh* u = nullptr;
  ph_status st = mesh_build(nullptr, nCu, nullptr, nEu, nullptr, nNu, s, &u, &bc);
  free_async(in, s);
  if (st != PH_OK) return st;
  cudaError_t e = cudaSuccess;
  // per-problem face, multiplier and CSR offsets; an empty problem starts
  // where the next one does
  std::vector<int64_t> foff(n + 1, 0), moff(n + 1, 0), zoff(n + 1, 0);
  foff[n] = u->nF;
  moff[n] = u->L;
  zoff[n] = u->nnz;
  bool ordered = true;
  for (int32_t p = n - 1; p >= 0; --p) {
    const bool empty = cnt[3 * p] < 0;
    foff[p] = empty ? foff[p + 1] : cnt[3 * p];
    moff[p] = empty ? moff[p + 1] : cnt[3 * p + 1];
    zoff[p] = empty ? zoff[p + 1] : cnt[3 * p + 2];
    ordered = ordered && foff[p] <= foff[p + 1] && moff[p] <= moff[p + 1] && zoff[p] <= zoff[p + 1];
  }
  if (!ordered || foff[0] != 0 || moff[0] != 0 || zoff[0] != 0) {
    mesh_free(u, s);
    return PH_ERR_ARG;
  }
  for (int32_t p = 0; p < n && e == cudaSuccess; ++p)  // no row wrote the one row pointer of an empty system
    if (moff[p + 1] == moff[p]) e = cudaMemsetAsync(bc.rowptr + moff[p] + p, 0, sizeof(int32_t), s);
  if (e != cudaSuccess) {
    mesh_free(u, s);
    return cuda_status(e, "ph_mesh_create_batch rows");
  }
  // the views: each problem's slices of the union arrays, local ids
  ph_mesh_shared* sh = new ph_mesh_shared();
  sh->refs.store(n);
  sh->arena = u->arena;
  for (int32_t p = 0; p < n; ++p) {
    ph_mesh* m = new ph_mesh();
    memset(m, 0, sizeof *m);
    const int64_t t0 = toff[p], v0 = voff[p], f0 = foff[p], m0 = moff[p], z0 = zoff[p];
    m->device = u->device;
    m->shared = sh;
    m->nE = nE[p];
    m->nC = nC[p];
    m->nF = foff[p + 1] - f0;
    m->L = moff[p + 1] - m0;
    m->nnz = zoff[p + 1] - z0;
    m->nFi = 4 * m->nE - m->nF;
    m->nFn = m->nF - m->L;
    m->nFd = m->nF - m->nFi - m->nFn;
    m->coord = u->coord + 3 * v0;
    m->tet = u->tet + t0;
    m->tface = u->tface + t0;
    m->tmult = u->tmult + t0;
    m->tpos = u->tpos + t0;
    m->trel = u->trel + t0;
    m->geo = u->geo + PH_GEO_STRIDE * t0;
    m->gexp = u->gexp + t0;
    m->vol = u->vol + t0;
    m->face_tet = u->face_tet + f0;
    m->face_vtx = u->face_vtx + 3 * f0;
    m->face_kind = u->face_kind + f0;
    m->face_mult = u->face_mult + f0;
    m->face_area = u->face_area + f0;
    m->rowptr = bc.rowptr + m0 + p;
    m->colind = u->colind + z0;
    m->status = u->status;
    out[p] = m;
  }
  delete u;  // its arena now belongs to the views
  return PH_OK;
}
