// Internals of the conjugate-gradient solver shared by the Jacobi and the
// Schwarz-preconditioned solves: launch shape, device scalars, deterministic
// block and grid reductions, and the Schwarz preconditioner's data.
#pragma once

#include "ph_internal.cuh"

namespace ph_pcg {

constexpr int RT = 256;   // threads per block
constexpr int RB = 1216;  // blocks (8 x 152 SMs) for vector kernels and partial sums

struct Scalars {
  double rz, pq, alpha, beta, rr, bb;
  unsigned done;  // blocks finished in the current reducing kernel (last-block detection)
  unsigned bad;   // a non-positive diagonal entry was seen
  double qtail;   // q of the last row of an odd system (k_pcg_loop)
  int it;         // iterations done (k_pcg_loop)
  unsigned late;  // a wait of k_pcg_loop ran out
  double pad[16];
  unsigned bar;   // k_pcg_loop: blocks that have arrived (a cache line of its own)
};

// Partial sums: part[0, RB) = p.q, part[RB, 2RB) = r.z, part[2RB, 3RB) = r.r.
// k_pcg_loop (systems of at most kLoopMaxN rows) publishes its sums there: RB
// sums of p.q, RB of r.z in row order, then RB / 2 of r.z and RB / 2 of r.r in
// pair order (one per 256 rows or pairs, or in systems of at most kLoopWarpN
// rows one per warp).
constexpr int64_t kLoopMaxN = (int64_t)RB * RT;  // one row per thread of the vector kernels
constexpr int64_t kLoopWarpN = 32 * (int64_t)RB;
constexpr size_t kPart = 3 * (size_t)RB;

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sm[RT / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = threadIdx.x < RT / 32 ? sm[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;  // valid in thread 0
}

// Sum of part[off, off + RB) in a fixed order (every caller gets the same
// value); the partials come from other blocks, so they bypass L1.
__device__ __forceinline__ double sum_partials(const double* __restrict__ part, int off) {
  double v = 0.0;
  for (int i = threadIdx.x; i < RB; i += RT) v += __ldcg(part + off + i);
  return block_sum(v);
}

// True in the block that finishes last (it then owns the final reduction).
// The caller's thread 0 wrote its partial before; the fence orders it before
// the count.
__device__ __forceinline__ bool last_block(unsigned* done) {
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  return s_last;
}

// Index of (i, j), i <= j, in a packed row-major upper triangle of order k.
__host__ __device__ __forceinline__ int upper(int i, int j, int k) { return i * k - i * (i - 1) / 2 + (j - i); }

// z = M r for the edge-patch Schwarz preconditioner P (y: scratch of
// P->nmem doubles), with the sum r.z: init sets rz, otherwise the last block
// sets beta = r.z / rz_old and rz.  Two launches.
cudaError_t schwarz_apply(const ph_schwarz* P, const double* r, double* z, double* y, double* part, Scalars* sc,
                          bool init, cudaStream_t s);

}  // namespace ph_pcg

// Additive Schwarz preconditioner over edge patches: patch e holds the
// multipliers of the faces around edge e; M = sum_e R_e' (R_e H R_e')^-1 R_e.
// Patches are grouped by their number of members k (a patch wider than
// kSchwarzDense becomes k patches of one member: its diagonal), and within a
// group every array is slot-major (entry q of patch s at base + q count + s),
// so the threads of a warp -- consecutive patches of one group -- make
// contiguous accesses.
constexpr int kSchwarzDense = 16;  // widest patch inverted densely

struct SchwarzGroups {
  int64_t count[kSchwarzDense + 1];  // patches with k members
  int64_t first[kSchwarzDense + 2];  // index of the first patch of group k (patches ordered by k)
  int64_t mbase[kSchwarzDense + 1];  // group k in mem and y: k slots per patch
  int64_t bbase[kSchwarzDense + 1];  // group k in blk: k(k+1)/2 entries per patch
};

struct ph_schwarz {
  int device;
  int64_t L, nEd, nmem, npatch, nblk;
  SchwarzGroups g;
  int32_t* mem;    // multiplier ids, ascending within a patch
  double* blk;     // patch inverses: packed upper triangle, row-major
  int32_t* fslot;  // 3L: positions in mem (and y) of each multiplier in the patches of its face's three edges
};

namespace ph_pcg {

// Group of patch index t (patches ordered by group).
__device__ __forceinline__ int group_of(const SchwarzGroups& g, int64_t t) {
  int k = 1;
  while (k < kSchwarzDense && t >= g.first[k + 1]) ++k;
  return k;
}

// y = block^-1 r_patch for one patch of K members (slot-major group arrays,
// stride n): the packed inverse in registers, sums in member order.  rval(m)
// is the residual of multiplier m; STREAM reads the block past the caches
// (it is read once per application).
template <int K, bool STREAM, class R>
__device__ __forceinline__ void patch_solve(int64_t s, int64_t n, const int32_t* __restrict__ mem,
                                            const double* __restrict__ blk, const R& rval, double* __restrict__ y) {
  constexpr int NQ = K * (K + 1) / 2;
  double rv[K];
  if (!STREAM && K > 6) {  // the block would not fit the caller's registers; its second use hits L1
#pragma unroll
    for (int j = 0; j < K; ++j) rv[j] = rval(__ldg(mem + j * n + s));
#pragma unroll 1
    for (int i = 0; i < K; ++i) {
      double v = 0.0;
#pragma unroll
      for (int j = 0; j < K; ++j) v = fma(__ldg(blk + (i <= j ? upper(i, j, K) : upper(j, i, K)) * n + s), rv[j], v);
      y[i * n + s] = v;
    }
    return;
  }
  double m[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) m[q] = STREAM ? __ldcs(blk + q * n + s) : __ldg(blk + q * n + s);
#pragma unroll
  for (int j = 0; j < K; ++j) rv[j] = rval(__ldg(mem + j * n + s));
#pragma unroll
  for (int i = 0; i < K; ++i) {
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < K; ++j) v = fma(m[i <= j ? upper(i, j, K) : upper(j, i, K)], rv[j], v);
    y[i * n + s] = v;
  }
}

// The same for patch t of group k.
template <bool STREAM, class R>
__device__ __forceinline__ void patch_apply(const SchwarzGroups& g, int64_t t, int k, const int32_t* __restrict__ mem,
                                            const double* __restrict__ blk, const R& rval, double* __restrict__ y) {
  const int64_t s = t - g.first[k], n = g.count[k];
  const int32_t* mm = mem + g.mbase[k];
  const double* bb = blk + g.bbase[k];
  double* yy = y + g.mbase[k];
  switch (k) {  // uniform across a warp except at the group boundaries
    case 1: patch_solve<1, STREAM>(s, n, mm, bb, rval, yy); break;
    case 2: patch_solve<2, STREAM>(s, n, mm, bb, rval, yy); break;
    case 3: patch_solve<3, STREAM>(s, n, mm, bb, rval, yy); break;
    case 4: patch_solve<4, STREAM>(s, n, mm, bb, rval, yy); break;
    case 5: patch_solve<5, STREAM>(s, n, mm, bb, rval, yy); break;
    case 6: patch_solve<6, STREAM>(s, n, mm, bb, rval, yy); break;
    case 7: patch_solve<7, STREAM>(s, n, mm, bb, rval, yy); break;
    case 8: patch_solve<8, STREAM>(s, n, mm, bb, rval, yy); break;
    default: {  // 9..kSchwarzDense members: rare; the block read entry by entry
      double rv[kSchwarzDense];
      for (int j = 0; j < k; ++j) rv[j] = rval(__ldg(mm + j * n + s));
      for (int i = 0; i < k; ++i) {
        double v = 0.0;
        for (int j = 0; j < k; ++j) v = fma(__ldg(bb + (int64_t)(i <= j ? upper(i, j, k) : upper(j, i, k)) * n + s),
                                            rv[j], v);
        yy[i * n + s] = v;
      }
    }
  }
}

}  // namespace ph_pcg
