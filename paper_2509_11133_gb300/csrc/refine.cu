// Uniform 1 -> 12 refinement on the device (Section 3.4, Listing RedRefine)
// with the edge numbering of Listing NumEdges.
//
// Edges are numbered as in edges.cuh.  New nodes are numbered as the listing's
// stable unique of [centroid, M1..M6] per tet gives them: walking the tets in
// order, each tet adds its centroid and then the midpoints of its not-yet-seen
// edges, i.e.
//     centroid(t)        = nC + t + (first occurrences in tets < t),
//     midpoint(edge, f)  = nC + t_f + 1 + (first occurrences before slot f),
// f the edge's first slot.  Coordinates: ((P0 + P1) + P2 + P3) / 4 and
// (P_a + P_b) / 2 with the endpoints of the first occurrence.  Child 1 of
// parent t replaces it; children 2..12 sit at nE + 11 t + (0..10).  Boundary
// triples [n1 n2 n3] (the paper's Db, Nb) become [n1 m12 m13] in place and
// [n2 m23 m12], [n3 m13 m23], [m12 m23 m13] at nF + 3 i + (0..2) (refineFaces).
#include <math.h>
#include <string.h>

#include "edges.cuh"
#include "ph_internal.cuh"

namespace {

// id of the midpoint whose edge first occurs in slot f
__device__ __forceinline__ int midpoint(int64_t nC, const int32_t* __restrict__ ebase,
                                        const uint8_t* __restrict__ mask, int f) {
  return (int)(nC + f / 6 + 1) + edge_of_first(ebase, mask, f);
}

// per tet: centroid and midpoint ids, coordinates and the 12 children.  The
// children of a block's tets are staged in shared memory and written as one
// contiguous run (a thread's own 11 are 176 bytes from its neighbour's: a warp's
// store touched 32 half-filled sectors, 11 times).  Bound by its writes, 16
// bytes per child and 24 per new node: 130 -> 90 us at 1M tets (250 MB).
constexpr int kRefineThreads = 128;

__global__ void __launch_bounds__(kRefineThreads) k_refine_tets(
    const double* __restrict__ coord, const int4* __restrict__ tet, int64_t nE, int64_t nC,
    const int32_t* __restrict__ first, const int32_t* __restrict__ ebase, const uint8_t* __restrict__ mask,
    double* __restrict__ coord_out, int4* __restrict__ tet_out) {
  __shared__ int4 kids[11 * kRefineThreads];
  const int64_t t0 = blockIdx.x * (int64_t)kRefineThreads, t = t0 + threadIdx.x;
  if (t < nE) {
    const int4 v = tet[t];
    const int2* fp = reinterpret_cast<const int2*>(first + 6 * t);
    const int2 fa = fp[0], fb = fp[1], fc = fp[2];
    const int f[6] = {fa.x, fa.y, fb.x, fb.y, fc.x, fc.y};
    const int cent = (int)(nC + t + ebase[t]);
    int mid[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) mid[j] = midpoint(nC, ebase, mask, f[j]);
    double P[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int d = 0; d < 3; ++d) P[i][d] = coord[3 * (int64_t)vget(v, i) + d];
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (f[j] == (int)(6 * t + j)) {
        int p, q;
        local_edge(j, p, q);
#pragma unroll
        for (int d = 0; d < 3; ++d) coord_out[3 * (int64_t)mid[j] + d] = (P[p][d] + P[q][d]) / 2.0;
      }
#pragma unroll
    for (int d = 0; d < 3; ++d)
      coord_out[3 * (int64_t)cent + d] = (((P[0][d] + P[1][d]) + P[2][d]) + P[3][d]) / 4.0;
    const int I = v.x, J = v.y, K = v.z, L = v.w;
    const int IJ = mid[0], IK = mid[1], IL = mid[2], JK = mid[3], JL = mid[4], KL = mid[5], C = cent;
    tet_out[t] = make_int4(I, IJ, IK, IL);
    int4* o = kids + 11 * threadIdx.x;
    o[0] = make_int4(J, JK, IJ, JL);
    o[1] = make_int4(K, IK, JK, KL);
    o[2] = make_int4(L, KL, JL, IL);
    o[3] = make_int4(IJ, IK, IL, C);
    o[4] = make_int4(JK, IJ, JL, C);
    o[5] = make_int4(IK, JK, KL, C);
    o[6] = make_int4(KL, JL, IL, C);
    o[7] = make_int4(IJ, JK, IK, C);
    o[8] = make_int4(IK, KL, IL, C);
    o[9] = make_int4(IJ, IL, JL, C);
    o[10] = make_int4(KL, JK, JL, C);
  }
  __syncthreads();
  const int have = (int)(nE - t0 < kRefineThreads ? nE - t0 : kRefineThreads);
  for (int i = threadIdx.x; i < 11 * have; i += kRefineThreads) tet_out[nE + 11 * t0 + i] = kids[i];
}

__device__ __forceinline__ int find_mid(const int2* __restrict__ entries, const int32_t* __restrict__ start, int sub,
                                        const int32_t* __restrict__ first, const int32_t* __restrict__ ebase,
                                        const uint8_t* __restrict__ mask, int x, int y, int64_t nC) {
  if (x < 0 || y < 0 || x >= nC || y >= nC || x == y) return -1;
  const int hi = max(x, y), lo = min(x, y);
  const int64_t b = edge_bucket(lo, hi, sub);
  for (int k = start[b]; k < start[b + 1]; ++k)
    if (entries[k].x == lo) return midpoint(nC, ebase, mask, first[entries[k].y]);
  return -1;
}

// Returns at once when an invalid tet was flagged: the entries are incomplete.
__global__ void k_refine_lists(const int32_t* __restrict__ in, int64_t nl, const int2* __restrict__ entries,
                               const int32_t* __restrict__ start, int sub, const int32_t* __restrict__ first,
                               const int32_t* __restrict__ ebase, const uint8_t* __restrict__ mask, int64_t nC,
                               int32_t* __restrict__ out, unsigned* status, const unsigned* invalid) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nl || *invalid) return;
  const int n1 = in[3 * i], n2 = in[3 * i + 1], n3 = in[3 * i + 2];
  const int m12 = find_mid(entries, start, sub, first, ebase, mask, n1, n2, nC);
  const int m13 = find_mid(entries, start, sub, first, ebase, mask, n1, n3, nC);
  const int m23 = find_mid(entries, start, sub, first, ebase, mask, n2, n3, nC);
  if (m12 < 0 || m13 < 0 || m23 < 0) { ph_flag(status, PH_ERR_ARG); return; }
  int32_t* a = out + 3 * i;
  a[0] = n1; a[1] = m12; a[2] = m13;
  int32_t* b = out + 3 * (nl + 3 * i);
  b[0] = n2; b[1] = m23; b[2] = m12;
  b[3] = n3; b[4] = m13; b[5] = m23;
  b[6] = m12; b[7] = m23; b[8] = m13;
}

}  // namespace

using namespace ph;

struct ph_refined {
  int64_t nC, nE, nEd, nl;  // refined counts (nEd: edges of the parent mesh)
  void* arena;              // coord and tet
  double* coord;
  int4* tet;
  int32_t* lists;
};

static void refined_free(ph_refined* r, cudaStream_t s) {
  free_async(r->arena, s);
  free_async(r->lists, s);
  delete r;
}

extern "C" ph_status ph_refine(const double* coord, int64_t nC, const int32_t* tet, int64_t nE,
                               const int32_t* lists, int64_t nl, void* stream, ph_refined** out) {
  if (!out) return PH_ERR_ARG;
  *out = nullptr;
  if (nC < 0 || nE < 0 || nl < 0 || (nE > 0 && (!coord || !tet)) || (nl > 0 && !lists)) return PH_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(tet) & 15u) != 0) return PH_ERR_ARG;  // read as int4
  if (6 * nE >= ((int64_t)1 << 31) - 1 || 12 * nE >= ((int64_t)1 << 31) - 1 || 4 * nl >= ((int64_t)1 << 31) / 3)
    return PH_ERR_OVERFLOW;
  cudaStream_t s = (cudaStream_t)stream;
  EdgeNumbering E;
  struct Head {
    int64_t nEd;
    unsigned status, lists;  // errors of the tets, of the lists
  };
  Head* d_head = nullptr;
  Head h{0, 0, 0};
  ph_refined* r = new ph_refined();
  memset(r, 0, sizeof *r);
  cudaError_t e = cudaSuccess;
  ph_status st = PH_OK;
#define RF_CU(expr)                      \
  do {                                   \
    e = (expr);                          \
    if (e != cudaSuccess) goto cuda_fail; \
  } while (0)
  RF_CU(alloc(&d_head, 1, s));
  RF_CU(cudaMemsetAsync(d_head, 0, sizeof(Head), s));
  st = enqueue_edges(reinterpret_cast<const int4*>(tet), nE, nC, &d_head->status, &d_head->nEd, s, &E);
  if (st != PH_OK) goto fail;
  r->nl = 4 * nl;
  if (nl > 0) {  // before the synchronisation, which then reports a bad triple too
    RF_CU(alloc(&r->lists, (size_t)(3 * r->nl), s));
    k_refine_lists<<<grid_for(nl), kThreads, 0, s>>>(lists, nl, E.entries, E.start, E.sub, E.first, E.ebase, E.mask, nC,
                                                     r->lists, &d_head->lists, &d_head->status);
    RF_CU(launched());
  }
  RF_CU(cudaMemcpyAsync(&h, d_head, sizeof h, cudaMemcpyDeviceToHost, s));
  RF_CU(cudaStreamSynchronize(s));
  if (h.status | h.lists) { st = status_from_bits(h.status ? h.status : h.lists); goto fail; }
  r->nEd = h.nEd;
  r->nC = nC + nE + h.nEd;
  r->nE = 12 * nE;
  if (r->nC >= ((int64_t)1 << 31) - 1) { st = PH_ERR_OVERFLOW; goto fail; }
  {
    Carve c;
    const size_t o_tet = c.take<int4>(r->nE), o_coord = c.take<double>(3 * r->nC);
    RF_CU(alloc_bytes(&r->arena, c.bytes + 16, s));
    r->tet = Carve::at<int4>(r->arena, o_tet);
    r->coord = Carve::at<double>(r->arena, o_coord);
  }
  if (nC > 0) RF_CU(cudaMemcpyAsync(r->coord, coord, sizeof(double) * 3 * nC, cudaMemcpyDeviceToDevice, s));
  if (nE > 0) {
    k_refine_tets<<<grid_for(nE, kRefineThreads), kRefineThreads, 0, s>>>(
        coord, reinterpret_cast<const int4*>(tet), nE, nC, E.first, E.ebase, E.mask, r->coord, r->tet);
    RF_CU(launched());
  }
  RF_CU(cudaStreamSynchronize(s));  // the caller's arrays have been read
  release_edges(E, s);
  free_async(d_head, s);
  *out = r;
  return PH_OK;
cuda_fail:
  st = cuda_status(e, "ph_refine");
fail:
  release_edges(E, s);
  free_async(d_head, s);
  refined_free(r, s);
  return st;
#undef RF_CU
}

extern "C" ph_status ph_refined_info(const ph_refined* r, int64_t* nC, int64_t* nE, int64_t* nEd_parent,
                                     int64_t* nl) {
  if (!r) return PH_ERR_ARG;
  if (nC) *nC = r->nC;
  if (nE) *nE = r->nE;
  if (nEd_parent) *nEd_parent = r->nEd;
  if (nl) *nl = r->nl;
  return PH_OK;
}

extern "C" ph_status ph_refined_copy(const ph_refined* r, double* coord, int32_t* tet, int32_t* lists, void* stream) {
  if (!r) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  if (coord && r->nC) e = cudaMemcpyAsync(coord, r->coord, sizeof(double) * 3 * r->nC, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && tet && r->nE)
    e = cudaMemcpyAsync(tet, r->tet, sizeof(int4) * r->nE, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && lists && r->nl)
    e = cudaMemcpyAsync(lists, r->lists, sizeof(int32_t) * 3 * r->nl, cudaMemcpyDeviceToDevice, s);
  return cuda_status(e, "ph_refined_copy");
}

extern "C" ph_status ph_refined_destroy(ph_refined* r, void* stream) {
  if (!r) return PH_OK;
  refined_free(r, (cudaStream_t)stream);
  return PH_OK;
}
