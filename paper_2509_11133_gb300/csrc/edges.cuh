// Edge numbering of Listing NumEdges on the device, shared by the refinement
// (ph_refine) and the edge-patch Schwarz preconditioner (ph_schwarz_*).
//
// Every local edge of every tet (local order IJ, IK, IL, JK, JL, KL; slot
// 6t+j) is a key (lo, hi) counting-sorted into buckets by hi and two bits of lo;
// within a bucket each occurrence finds the smallest slot with the same key (its
// edge's first occurrence).  Edge ids are first-occurrence ranks, as the
// listing's stable unique gives them: edge_id(slot) = ebase[t_f] + (first
// occurrences before slot f inside tet t_f), f = first[slot]; the first
// occurrences of a tet are the bits of its mask.
//
// Buckets by hi alone hold ~35 entries on refined meshes, and every entry reads
// its whole bucket: four buckets per vertex take k_edge_first from 82 to 61 us
// at 1M tets.
#pragma once

#include "ph_internal.cuh"

namespace {  // device code: a private copy per translation unit

__device__ __forceinline__ int vget(int4 v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// local edge j: IJ, IK, IL, JK, JL, KL
__device__ __forceinline__ void local_edge(int j, int& p, int& q) {
  const int P[6] = {0, 0, 0, 1, 1, 2};
  const int Q[6] = {1, 2, 3, 2, 3, 3};
  p = P[j];
  q = Q[j];
}

__device__ __forceinline__ bool valid_tet(int4 v, int64_t nC) {
  bool in = v.x >= 0 && v.y >= 0 && v.z >= 0 && v.w >= 0 && v.x < nC && v.y < nC && v.z < nC && v.w < nC;
  bool distinct = v.x != v.y && v.x != v.z && v.x != v.w && v.y != v.z && v.y != v.w && v.z != v.w;
  return in && distinct;
}

// bucket of edge (lo, hi): `sub` bits of lo below hi
__device__ __forceinline__ int64_t edge_bucket(int lo, int hi, int sub) {
  return ((int64_t)hi << sub) | (lo & ((1 << sub) - 1));
}

__global__ void k_edge_count(const int4* __restrict__ tet, int64_t nE, int64_t nC, int sub, int32_t* __restrict__ cnt,
                             unsigned* status) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nE) return;
  const int4 v = tet[t];
  if (!valid_tet(v, nC)) { ph_flag(status, PH_ERR_ARG); return; }
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    int p, q;
    local_edge(j, p, q);
    const int x = vget(v, p), y = vget(v, q);
    atomicAdd(&cnt[edge_bucket(min(x, y), max(x, y), sub)], 1);
  }
}

// entry = (lo, slot)
// Both kernels below return at once once an invalid tet was flagged: the
// entries of such a mesh are incomplete and must not be dereferenced.
__global__ void k_edge_fill(const int4* __restrict__ tet, int64_t nE, int sub, const int32_t* __restrict__ start,
                            int32_t* __restrict__ cnt, int2* __restrict__ entries, const unsigned* status) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nE || *status) return;
  const int4 v = tet[t];
  int pos[6];  // six atomics in flight, then their stores
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    int p, q;
    local_edge(j, p, q);
    const int a = vget(v, p), b = vget(v, q);
    const int64_t k = edge_bucket(min(a, b), max(a, b), sub);
    pos[j] = start[k] + atomicSub(&cnt[k], 1) - 1;
  }
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    int p, q;
    local_edge(j, p, q);
    entries[pos[j]] = make_int2(min(vget(v, p), vget(v, q)), (int)(6 * t + j));
  }
}

// first[slot] = smallest slot with the same (lo, hi); the bucket of entry i is
// found from its slot's tet (hi = max of the slot's endpoints).
__global__ void k_edge_first(const int4* __restrict__ tet, const int2* __restrict__ entries, int64_t nent, int sub,
                             const int32_t* __restrict__ start, int32_t* __restrict__ first, const unsigned* status) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nent || *status) return;
  const int2 e = entries[i];
  const int t = e.y / 6, j = e.y % 6;
  int p, q;
  local_edge(j, p, q);
  const int4 v = tet[t];
  const int64_t bucket = edge_bucket(e.x, max(vget(v, p), vget(v, q)), sub);
  const int begin = start[bucket], end = start[bucket + 1];
  int m = e.y;
  for (int k = begin; k < end; ++k) {
    const int2 f = entries[k];
    if (f.x == e.x && f.y < m) m = f.y;
  }
  first[e.y] = m;
}

// The tet's mask of first occurrences and their number.
__global__ void k_edge_newcount(const int32_t* __restrict__ first, int64_t nE, uint8_t* __restrict__ mask,
                                int32_t* __restrict__ ecount) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nE) return;
  const int2* f = reinterpret_cast<const int2*>(first + 6 * t);
  const int2 a = f[0], b = f[1], c = f[2];
  const int s = (int)(6 * t);
  const unsigned m = (a.x == s) | (a.y == s + 1) << 1 | (b.x == s + 2) << 2 | (b.y == s + 3) << 3 |
                     (c.x == s + 4) << 4 | (c.y == s + 5) << 5;
  mask[t] = (uint8_t)m;
  ecount[t] = __popc(m);
}

// Edge id of the first occurrence in slot f.
__device__ __forceinline__ int edge_of_first(const int32_t* __restrict__ ebase, const uint8_t* __restrict__ mask,
                                             int f) {
  const int t = f / 6, j = f - 6 * t;
  return ebase[t] + __popc(mask[t] & ((1u << j) - 1u));
}

// Edge id of a slot from the numbering (first occurrence slot f = first[slot]).
__device__ __forceinline__ int edge_id(const int32_t* __restrict__ first, const int32_t* __restrict__ ebase,
                                       const uint8_t* __restrict__ mask, int64_t slot) {
  return edge_of_first(ebase, mask, first[slot]);
}

// Buffers of one numbering (one stream-ordered allocation of pool memory).
struct EdgeNumbering {
  void* arena = nullptr;
  int sub = 0;  // buckets per vertex: 2^sub
  int32_t *start = nullptr, *first = nullptr, *ebase = nullptr;
  int2* entries = nullptr;
  uint8_t* mask = nullptr;
};

void release_edges(EdgeNumbering& E, cudaStream_t s) {
  ph::free_async(E.arena, s);
  E = EdgeNumbering();
}

// Enqueue the numbering of the edges of tet[nE] (vertex ids checked against
// nC; errors go to *status); the edge count lands in *d_nEd.  No
// synchronisation.
ph_status enqueue_edges(const int4* tet, int64_t nE, int64_t nC, unsigned* status, int64_t* d_nEd, cudaStream_t s,
                        EdgeNumbering* E) {
  const int64_t nent = 6 * nE;
  E->sub = nC < ((int64_t)1 << 28) ? 2 : 0;
  const int64_t nb = (nC << E->sub) + 1;
  ph::Carve c;  // the part to clear first
  const size_t o_cnt = c.take<int32_t>(nb), o_ebase = c.take<int32_t>(nE + 1);
  const size_t o_s1 = c.take<unsigned long long>(ph::scan_state_words(nb));
  const size_t o_s2 = c.take<unsigned long long>(ph::scan_state_words(nE + 1));
  const size_t clear = c.bytes;
  const size_t o_start = c.take<int32_t>(nb), o_entries = c.take<int2>(nent), o_first = c.take<int32_t>(nent);
  const size_t o_mask = c.take<uint8_t>(nE);
  cudaError_t e = ph::alloc_bytes(&E->arena, c.bytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(E->arena, 0, clear, s);
  if (e != cudaSuccess) return ph::cuda_status(e, "edge numbering");
  int32_t* cnt = ph::Carve::at<int32_t>(E->arena, o_cnt);
  E->ebase = ph::Carve::at<int32_t>(E->arena, o_ebase);
  E->start = ph::Carve::at<int32_t>(E->arena, o_start);
  E->entries = ph::Carve::at<int2>(E->arena, o_entries);
  E->first = ph::Carve::at<int32_t>(E->arena, o_first);
  E->mask = ph::Carve::at<uint8_t>(E->arena, o_mask);
  if (nE > 0) {
    k_edge_count<<<ph::grid_for(nE), ph::kThreads, 0, s>>>(tet, nE, nC, E->sub, cnt, status);
    e = ph::launched();
    if (e != cudaSuccess) return ph::cuda_status(e, "edge numbering");
  }
  ph_status st = ph::exclusive_scan(cnt, E->start, nb, d_nEd, s, status, nullptr, 0,
                                    ph::Carve::at<unsigned long long>(E->arena, o_s1));
  if (st != PH_OK) return st;
  if (nE > 0) {
    k_edge_fill<<<ph::grid_for(nE), ph::kThreads, 0, s>>>(tet, nE, E->sub, E->start, cnt, E->entries, status);
    k_edge_first<<<ph::grid_for(nent), ph::kThreads, 0, s>>>(tet, E->entries, nent, E->sub, E->start, E->first,
                                                             status);
    k_edge_newcount<<<ph::grid_for(nE), ph::kThreads, 0, s>>>(E->first, nE, E->mask, E->ebase);
    e = ph::launched(3);
    if (e != cudaSuccess) return ph::cuda_status(e, "edge numbering");
  }
  return ph::exclusive_scan(E->ebase, E->ebase, nE + 1, d_nEd, s, status, nullptr, 0,
                            ph::Carve::at<unsigned long long>(E->arena, o_s2));
}

}  // namespace
