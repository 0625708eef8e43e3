// Jacobi-preconditioned conjugate gradients for the condensed face system
// H Lambda = rhs (Eq. schur; the paper solves it with MATLAB's backslash).
// All reductions use a fixed grid and a fixed summation order, so repeated
// solves are bitwise reproducible.
#include <math.h>

#include "pcg.cuh"
#include "ph_internal.cuh"

namespace {

using namespace ph_pcg;

// Workspace of one solve (doubles): r, p, q, dinv (4 vectors of vec_stride(n)
// doubles, so each starts 256-byte aligned), then the partial sums, then
// Scalars.
inline size_t vec_stride(int64_t n) { return ((size_t)n + 31) & ~(size_t)31; }
// Second buffers of r and p for k_pcg_loop with a preconditioner (they follow
// the preconditioner's scratch, on an even offset).
inline size_t loop_extra(int64_t n) { return n <= kLoopMaxN ? 2 * vec_stride(n) + 1 : 0; }
inline size_t workspace_doubles(int64_t n) { return vec_stride(4 * (int64_t)vec_stride(n) + kPart + (sizeof(Scalars) + 7) / 8); }

__global__ void __launch_bounds__(RT) k_pcg_init(int64_t n, const int32_t* __restrict__ rowptr,
                                                 const int32_t* __restrict__ colind, const double* __restrict__ val,
                                                 const double* __restrict__ b, double* __restrict__ x,
                                                 double* __restrict__ r, double* __restrict__ p,
                                                 double* __restrict__ dinv, double* __restrict__ part,
                                                 Scalars* __restrict__ sc) {
  double rz = 0.0, bb = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    double d = 0.0;
    for (int j = rowptr[i]; j < rowptr[i + 1]; ++j)
      if (colind[j] == i) d = val[j];
    if (!(d > 0.0)) atomicOr(&sc->bad, 1u);
    const double di = d > 0.0 ? 1.0 / d : 0.0;
    const double bi = b[i];
    dinv[i] = di;
    x[i] = 0.0;
    r[i] = bi;
    p[i] = di * bi;
    rz = fma(bi, di * bi, rz);
    bb = fma(bi, bi, bb);
  }
  rz = block_sum(rz);
  bb = block_sum(bb);
  if (threadIdx.x == 0) {
    part[RB + blockIdx.x] = rz;
    part[2 * RB + blockIdx.x] = bb;
  }
  if (last_block(&sc->done)) {
    const double rz_t = sum_partials(part, RB);
    const double bb_t = sum_partials(part, 2 * RB);
    if (threadIdx.x == 0) {
      sc->rz = rz_t;
      sc->bb = bb_t;
      sc->rr = bb_t;
      sc->done = 0;
    }
  }
}

// The solver keeps H in a slot-major ELL copy made once per solve: slot u of
// row i at u n + i (column -1 past the row's end), W = the longest row.  A
// warp's loads of slot u are then contiguous.  Rows of the condensed system
// hold 4 or 7 entries, so the copy costs ~W/7 of the CSR bytes.
constexpr int kEllMaxWidth = 16;  // wider rows keep the CSR kernel

__global__ void k_row_width(int64_t n, const int32_t* __restrict__ rowptr, unsigned* __restrict__ wmax) {
  unsigned w = 0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT)
    w = max(w, (unsigned)(rowptr[i + 1] - rowptr[i]));
  for (int o = 16; o > 0; o >>= 1) w = max(w, __shfl_down_sync(0xffffffffu, w, o));
  if ((threadIdx.x & 31) == 0) atomicMax(wmax, w);
}

__global__ void k_to_ell(int64_t n, int W, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                         const double* __restrict__ val, int32_t* __restrict__ ecol, double* __restrict__ eval) {
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    const int j0 = rowptr[i], len = rowptr[i + 1] - j0;
    for (int u = 0; u < W; ++u) {
      ecol[u * n + i] = u < len ? colind[j0 + u] : -1;
      eval[u * n + i] = u < len ? val[j0 + u] : 0.0;
    }
  }
}

// q = H p and p.q (ELL copy, one thread per row; the row sum is the fma chain
// in column order); the last block sets alpha = r.z / p.q.
template <int W>
__global__ void __launch_bounds__(RT) k_spmv_dot_ell(int64_t n, int w, const int32_t* __restrict__ ecol,
                                                     const double* __restrict__ eval, const double* __restrict__ p,
                                                     double* __restrict__ q, double* __restrict__ part,
                                                     Scalars* __restrict__ sc) {
  double pq = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    int c[W];
    double v[W];
#pragma unroll
    for (int u = 0; u < W; ++u) {
      c[u] = u < w ? __ldcs(ecol + u * n + i) : -1;
      v[u] = u < w ? __ldcs(eval + u * n + i) : 0.0;
    }
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (c[u] >= 0) s = fma(v[u], __ldg(p + c[u]), s);
    q[i] = s;
    pq = fma(__ldg(p + i), s, pq);
  }
  pq = block_sum(pq);
  if (threadIdx.x == 0) part[blockIdx.x] = pq;
  if (last_block(&sc->done)) {
    const double pq_t = sum_partials(part, 0);
    if (threadIdx.x == 0) {
      sc->pq = pq_t;
      sc->alpha = pq_t > 0.0 ? sc->rz / pq_t : 0.0;
      sc->done = 0;
    }
  }
}

// The same on the CSR arrays, for rows wider than kEllMaxWidth: one thread per
// row, the first 8 values and columns loaded at once (predicated) before the
// gathers, longer rows finished in a loop.
__global__ void __launch_bounds__(RT) k_spmv_dot(int64_t n, const int32_t* __restrict__ rowptr,
                                                 const int32_t* __restrict__ colind, const double* __restrict__ val,
                                                 const double* __restrict__ p, double* __restrict__ q,
                                                 double* __restrict__ part, Scalars* __restrict__ sc) {
  double pq = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    const int j0 = __ldg(rowptr + i), j1 = __ldg(rowptr + i + 1);
    const int len = j1 - j0;
    int c[8];
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      c[u] = u < len ? __ldg(colind + j0 + u) : 0;
      v[u] = u < len ? __ldg(val + j0 + u) : 0.0;
    }
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (u < len) s = fma(v[u], __ldg(p + c[u]), s);
    for (int j = j0 + 8; j < j1; ++j) s = fma(__ldg(val + j), __ldg(p + __ldg(colind + j)), s);
    q[i] = s;
    pq = fma(__ldg(p + i), s, pq);
  }
  pq = block_sum(pq);
  if (threadIdx.x == 0) part[blockIdx.x] = pq;
  if (last_block(&sc->done)) {
    const double pq_t = sum_partials(part, 0);
    if (threadIdx.x == 0) {
      sc->pq = pq_t;
      sc->alpha = pq_t > 0.0 ? sc->rz / pq_t : 0.0;
      sc->done = 0;
    }
  }
}

// x += alpha p, r -= alpha q (pairs of entries per 16-byte access), and the
// sums r.r and (Jacobi, JAC) r.z with z = dinv r; the last block sets rr and
// (JAC) beta = r.z_new / r.z.  With another preconditioner z and beta come
// from its application.
template <bool VEC, bool JAC>
__global__ void __launch_bounds__(RT) k_update(int64_t n, double* __restrict__ x, double* __restrict__ r,
                                               const double* __restrict__ p, const double* __restrict__ q,
                                               const double* __restrict__ dinv, Scalars* __restrict__ sc,
                                               double* __restrict__ part) {
  const double alpha = sc->alpha;
  double rz = 0.0, rr = 0.0;
  const int64_t stride = (int64_t)RB * RT;
  if (VEC) {  // x 16-byte aligned; r, p, q, dinv always are
    const int64_t n2 = n / 2;
    for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n2; i += stride) {
      const double2 xi = reinterpret_cast<const double2*>(x)[i], pi = reinterpret_cast<const double2*>(p)[i];
      const double2 qi = reinterpret_cast<const double2*>(q)[i], ri = reinterpret_cast<const double2*>(r)[i];
      const double2 di = JAC ? reinterpret_cast<const double2*>(dinv)[i] : make_double2(0.0, 0.0);
      const double2 xo = make_double2(fma(alpha, pi.x, xi.x), fma(alpha, pi.y, xi.y));
      const double2 ro = make_double2(fma(-alpha, qi.x, ri.x), fma(-alpha, qi.y, ri.y));
      __stcs(reinterpret_cast<double2*>(x) + i, xo);
      reinterpret_cast<double2*>(r)[i] = ro;
      if (JAC) {
        rz = fma(ro.x, di.x * ro.x, rz);
        rz = fma(ro.y, di.y * ro.y, rz);
      }
      rr = fma(ro.x, ro.x, rr);
      rr = fma(ro.y, ro.y, rr);
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
      const int64_t i = n - 1;
      x[i] = fma(alpha, p[i], x[i]);
      const double ri = fma(-alpha, q[i], r[i]);
      r[i] = ri;
      if (JAC) rz = fma(ri, dinv[i] * ri, rz);
      rr = fma(ri, ri, rr);
    }
  } else {
    for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += stride) {
      x[i] = fma(alpha, p[i], x[i]);
      const double ri = fma(-alpha, q[i], r[i]);
      r[i] = ri;
      if (JAC) rz = fma(ri, dinv[i] * ri, rz);
      rr = fma(ri, ri, rr);
    }
  }
  rz = block_sum(rz);
  rr = block_sum(rr);
  if (threadIdx.x == 0) {
    part[RB + blockIdx.x] = rz;
    part[2 * RB + blockIdx.x] = rr;
  }
  if (last_block(&sc->done)) {
    const double rz_t = JAC ? sum_partials(part, RB) : 0.0;
    const double rr_t = sum_partials(part, 2 * RB);
    if (threadIdx.x == 0) {
      if (JAC) {
        const double rz_old = sc->rz;
        sc->beta = rz_old > 0.0 ? rz_t / rz_old : 0.0;
        sc->rz = rz_t;
      }
      sc->rr = rr_t;
      sc->done = 0;
    }
  }
}

// p = z + beta p for a preconditioned residual z held in memory.
__global__ void __launch_bounds__(RT) k_direction_z(int64_t n, double* __restrict__ p, const double* __restrict__ z,
                                                    const Scalars* __restrict__ sc) {
  const double beta = sc->beta;
  const int64_t n2 = (n + 1) / 2;  // vectors are padded to an even length
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n2; i += (int64_t)RB * RT) {
    const double2 pi = reinterpret_cast<const double2*>(p)[i], zi = reinterpret_cast<const double2*>(z)[i];
    reinterpret_cast<double2*>(p)[i] = make_double2(fma(beta, pi.x, zi.x), fma(beta, pi.y, zi.y));
  }
}

// p = dinv r + beta p (all workspace vectors: 16-byte pairs).
__global__ void __launch_bounds__(RT) k_direction(int64_t n, double* __restrict__ p, const double* __restrict__ r,
                                                  const double* __restrict__ dinv, const Scalars* __restrict__ sc) {
  const double beta = sc->beta;
  const int64_t n2 = (n + 1) / 2;  // vectors are padded to an even length
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n2; i += (int64_t)RB * RT) {
    const double2 pi = reinterpret_cast<const double2*>(p)[i], ri = reinterpret_cast<const double2*>(r)[i];
    const double2 di = reinterpret_cast<const double2*>(dinv)[i];
    reinterpret_cast<double2*>(p)[i] = make_double2(fma(beta, pi.x, di.x * ri.x), fma(beta, pi.y, di.y * ri.y));
  }
}

// H in the solver: the ELL copy when its rows are at most kEllMaxWidth wide.
struct Matrix {
  const int32_t *rowptr, *colind;
  const double* values;
  int w;  // ELL width, 0 = use the CSR arrays
  const int32_t* ecol;
  const double* eval;
};

inline void launch_spmv_dot(int64_t n, const Matrix& A, const double* p, double* q, double* part, Scalars* sc,
                            cudaStream_t s) {
  if (A.w == 0) k_spmv_dot<<<RB, RT, 0, s>>>(n, A.rowptr, A.colind, A.values, p, q, part, sc);
  else if (A.w <= 4) k_spmv_dot_ell<4><<<RB, RT, 0, s>>>(n, A.w, A.ecol, A.eval, p, q, part, sc);
  else if (A.w <= 7) k_spmv_dot_ell<7><<<RB, RT, 0, s>>>(n, A.w, A.ecol, A.eval, p, q, part, sc);
  else k_spmv_dot_ell<kEllMaxWidth><<<RB, RT, 0, s>>>(n, A.w, A.ecol, A.eval, p, q, part, sc);
}

// one PCG iteration: 3 launches (Jacobi, z = dinv r fused), or 5 with the
// Schwarz preconditioner P (z kept in the dinv vector, y its scratch)
inline cudaError_t pcg_iteration(int64_t n, const Matrix& A, double* x, double* r, double* p, double* q,
                                 double* dinv, double* part, Scalars* sc, const ph_schwarz* P, double* y,
                                 cudaStream_t s) {
  launch_spmv_dot(n, A, p, q, part, sc, s);
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  if (!P) {
    if (vec) k_update<true, true><<<RB, RT, 0, s>>>(n, x, r, p, q, dinv, sc, part);
    else k_update<false, true><<<RB, RT, 0, s>>>(n, x, r, p, q, dinv, sc, part);
    k_direction<<<RB, RT, 0, s>>>(n, p, r, dinv, sc);
    return ph::launched(3);
  }
  if (vec) k_update<true, false><<<RB, RT, 0, s>>>(n, x, r, p, q, dinv, sc, part);
  else k_update<false, false><<<RB, RT, 0, s>>>(n, x, r, p, q, dinv, sc, part);
  cudaError_t e = ph::launched(2);
  if (e == cudaSuccess) e = schwarz_apply(P, r, dinv, y, part, sc, false, s);
  if (e == cudaSuccess) {
    k_direction_z<<<RB, RT, 0, s>>>(n, p, dinv, sc);
    e = ph::launched();
  }
  return e;
}

// ---------------------------------------------------------------------------
// Small and middle systems (n <= kLoopMaxN): the whole iteration in one
// cooperative launch.  The kernels above launch 1216 blocks whatever n is and
// spend ~10 us each on starting and counting them: a 1376-row Schwarz
// iteration took 43 us, a 47,520-row Jacobi iteration 36 us, while their
// arithmetic and data (in L1 and L2) take a fraction of a microsecond.  Here a
// grid of at most the co-resident blocks owns the rows for the whole solve;
// the blocks meet once per dependent reduction, twice in a Jacobi iteration
// and three times in a Schwarz iteration.  What bounds it is the chain of
// those phases (L2 round trips of the gathers and of the sums, FP64 latency)
// and, above ~100 rows per SM, the FP64 pipe (a warp's FP64 instruction takes
// 18 cycles of it).
//
//   A  q = H p with p = z + beta p_old formed at every gather (p_old and p in
//      two buffers): saves the direction pass and its meeting for 7 more FMA
//      a row;                                              sums p.q
//   B  x += alpha p, r -= alpha q (Jacobi: z = dinv r too); sums r.z or, when
//      convergence is tested, r.r.  Schwarz: the patch solves in the same
//      phase, on r - alpha q formed at every gather (r in two buffers);
//   C  (Schwarz) z = the sums of the patch values;          sums r.z
//
// Every sum is formed in the order of the kernels above (thread, warp, block,
// grid, which for n <= kLoopMaxN means one row, or one pair of rows, per
// thread), so the iterates, the iteration count and x are theirs bit for bit:
// blocks publish the sums of single warps, or of virtual 256-thread blocks,
// and every block finishes the same tree on them.  Us per iteration, the
// kernels above and this loop, on jittered meshes:
//     rows        1,650   9,234  21,600  50,688  98,400  169,344  297,714
//     Jacobi     34  8   36 10   36 10   37 11   37 16    41 20    43 30
//     Schwarz    47 12   47 14   47 15   47 17   51 24    57 33    64 41
// so the loop takes every size that one row per thread allows.  Of a small
// system's 20,000 to 24,000 cycles, about 4,600 a phase are the meeting (2,600),
// reading the sums (900, an L2 trip across the dies), their tree and the division
// (69 cycles per dependent FP64 operation).
//
// The meeting is a counter: each block adds one with release semantics after a
// block barrier and polls it with acquire semantics before the next one, so that
// what any thread wrote before a meeting happens before what any thread reads
// after it.  (Polling tagged sums instead of a counter saves the trip that then
// reads the sums, but 152 blocks polling 152 sums take 7,100 cycles to see them
// all against 1,400.)  The acquire empties L1 of the matrix and the patch inverses,
// which costs a 47,520-row Jacobi solve 6 to 12% and the Schwarz solves 2%; without
// it nothing orders the reads.  A relaxed poll and an acquire at its end take the
// same time, a relaxed poll and a fence 5 to 7% more.
// ---------------------------------------------------------------------------
struct LoopArgs {
  int64_t n;
  int w;                     // ELL width (0: the CSR arrays)
  const int32_t *rowptr, *col;
  const double* val;
  double *x, *r, *r2, *p, *p2, *q, *z;  // Jacobi: r holds z = dinv r while the kernel runs; r2, q, z unused
  const double* dinv;
  double* part;              // published sums
  unsigned* bar;             // arrivals (zero at the launch)
  Scalars* sc;
  double tol, res;           // rtol ||b||, the residual norm so far
  int it, it_stop, maxit, spin_limit;
  int withhold;              // block that never arrives (test hook), or -1
  int rows, slots;           // rows of a slot, slots per block
  SchwarzGroups g;
  int wfirst[kSchwarzDense + 2];  // group k's patches take the warps [wfirst[k], wfirst[k + 1]) of 32
  const int32_t *mem, *fslot;
  const double* blk;
  double* y;
};

// All blocks of the grid meet (they are co-resident: a cooperative launch).
// Bounded: *late is set, and the call returns, when the wait runs out.
__device__ __forceinline__ void loop_meet(unsigned* bar, unsigned& target, int spin_limit, int withhold, int* late) {
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    if ((int)blockIdx.x != withhold)
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned seen;
    for (int spins = 0;; ++spins) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      if ((int)(seen - target) >= 0) break;
      if (spins > spin_limit) {
        *late = 1;
        break;
      }
    }
  }
  __syncthreads();
}

// The sums of eight vectors of 32 (vector w at sm[32 w ..]), each in the order
// of block_sum's shuffle tree, and their total as block_sum forms it, by one
// warp (every lane gets it): the steps of several vectors share an instruction
// (lanes that the tree of one vector leaves idle take the next vector's), 12
// additions instead of 43.
__device__ __forceinline__ double packed_block_sum(const double* sm) {
  const int lane = threadIdx.x & 31;
  double v[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) v[w] = sm[32 * w + lane];
#pragma unroll
  for (int m = 4, o = 16; m >= 1; m >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int j = 0; j < m; ++j) {
      const double keep = up ? v[2 * j + 1] : v[2 * j], send = up ? v[2 * j] : v[2 * j + 1];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  // vector w now sits in the lanes with bits 4, 3, 2 = bits 0, 1, 2 of w
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 4);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 8);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
  return v[0];
}

// The total of cnt published sums in sum_partials' order, in every thread: sums
// of warps (WARPS: eight make a virtual block) or of virtual blocks.  Steps
// that would add zeros are left out.  `ratio` of the total comes with it: one
// thread divides (a division in every thread would take the block 2,000
// cycles of the FP64 pipe).
template <bool WARPS, class F>
__device__ __forceinline__ double2 loop_total(const double* part, int cnt, const F& ratio) {
  __shared__ double sm[8];
  __shared__ double2 out;
  const int nvb = WARPS ? (cnt + 7) >> 3 : cnt;
  const int nw = min(8, (nvb + 31) >> 5);  // warps with a share; the others' sums are zero
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid < nw) {
    double v = 0.0;
    if (WARPS) {
      for (int b = threadIdx.x; b < nvb; b += RT) {
        double w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = 8 * b + i < cnt ? __ldcg(part + 8 * b + i) : 0.0;
        v += ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
      }
    } else {
      constexpr int M = (RB + RT - 1) / RT;
      double w[M];
#pragma unroll
      for (int k = 0; k < M; ++k) w[k] = threadIdx.x + k * RT < nvb ? __ldcg(part + threadIdx.x + k * RT) : 0.0;
      v = w[0];
#pragma unroll
      for (int k = 1; k < M; ++k)
        if (k * RT < nvb) v += w[k];
    }
    for (int o = nvb > 16 ? 16 : nvb > 8 ? 8 : 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) {
      if (nw == 1) out = make_double2(v, ratio(v));
      else sm[wid] = v;
    }
  }
  __syncthreads();
  if (nw > 1) {
    if (wid == 0) {
      double v = lane < nw ? sm[lane] : 0.0;
      if (nw > 4) v += __shfl_down_sync(0xffffffffu, v, 4);
      if (nw > 2) v += __shfl_down_sync(0xffffffffu, v, 2);
      v += __shfl_down_sync(0xffffffffu, v, 1);
      if (lane == 0) out = make_double2(v, ratio(v));
    }
    __syncthreads();
  }
  return out;
}

// One row of H p, p = z + beta p_old: the fma chain in column order of
// k_spmv_dot and k_spmv_dot_ell.
template <class G>
__device__ __forceinline__ double loop_row(const LoopArgs& A, int64_t i, const G& pnew) {
  double s = 0.0;
  if (A.w > 0 && A.w <= 7) {
    int c[7];
    double v[7], g[7];
#pragma unroll
    for (int u = 0; u < 7; ++u) {
      c[u] = u < A.w ? __ldg(A.col + u * A.n + i) : -1;
      v[u] = u < A.w ? __ldg(A.val + u * A.n + i) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 7; ++u) g[u] = c[u] >= 0 ? pnew(c[u]) : 0.0;
#pragma unroll
    for (int u = 0; u < 7; ++u)
      if (c[u] >= 0) s = fma(v[u], g[u], s);
  } else if (A.w > 0) {
    for (int u = 0; u < A.w; ++u) {
      const int c = __ldg(A.col + u * A.n + i);
      if (c >= 0) s = fma(__ldg(A.val + u * A.n + i), pnew(c), s);
    }
  } else {
    const int j0 = __ldg(A.rowptr + i), j1 = __ldg(A.rowptr + i + 1);
    int c[8];
    double v[8], g[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      c[u] = j0 + u < j1 ? __ldg(A.col + j0 + u) : -1;
      v[u] = j0 + u < j1 ? __ldg(A.val + j0 + u) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) g[u] = c[u] >= 0 ? pnew(c[u]) : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c[u] >= 0) s = fma(v[u], g[u], s);
    for (int j = j0 + 8; j < j1; ++j) s = fma(__ldg(A.val + j), pnew(__ldg(A.col + j)), s);
  }
  return s;
}

constexpr int kLoopRows = 512;  // rows of a slot in larger systems: two virtual blocks of rows, one of pairs

// SCHW: Schwarz, else Jacobi.  WARPS: sums published per warp, one slot of
// A.rows = 64..256 rows per block; else per virtual block, slots of 512.
template <bool SCHW, bool WARPS>
__global__ void __launch_bounds__(RT, SCHW ? 2 : 3) k_pcg_loop(const __grid_constant__ LoopArgs A) {
  extern __shared__ __align__(16) double s_rows[];  // Jacobi: r, then q, of the block's rows
  __shared__ double s_sum[WARPS ? 1 : kLoopRows];
  __shared__ int s_late;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  const int rows = WARPS ? A.rows : kLoopRows;
  constexpr int PER = WARPS ? 1 : 2;  // rows per thread: tid and tid + RT
  const int64_t n = A.n, n2 = n / 2;
  const int nslot = (int)((n + rows - 1) / rows);
  const int nscal = nslot * (WARPS ? rows / 32 : 2), npair = WARPS ? nslot * (rows / 64) : nslot;
  const bool tail = (n & 1) && blockIdx.x == 0 && tid == 0;  // the last row of an odd n, as in k_update
  double* s_r = s_rows;
  double* s_q = s_rows + (size_t)A.slots * rows;
  double *part_pq = A.part, *part_rz = part_pq + RB, *pair_rz = part_rz + RB, *pair_rr = pair_rz + RB / 2;
  Scalars* sc = A.sc;
  double rz = __ldcg(&sc->rz), beta = __ldcg(&sc->beta), alpha = 0.0, pq = 0.0, rr = 0.0, r_tail = 0.0;
  unsigned target = 0;
  double *pold = A.p, *pnew = A.p2, *r = A.r, *rnew = SCHW ? A.r2 : A.r;
  double* z = SCHW ? A.z : A.r;
  int it = A.it;
  double res = A.res;
  if (tid == 0) s_late = 0;

  // scalar-order sums of the slot's rows (v[0], v[1]: rows tid, tid + RT)
  const auto publish_rows = [&](double* part, int b, const double v[PER]) {
    if (WARPS) {
      double t = v[0];
      if (tid < rows)
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (tid < rows && lane == 0) __stcg(part + b * (rows / 32) + wid, t);
    } else {
      __syncthreads();  // s_sum is free
      s_sum[tid] = v[0];
      s_sum[tid + RT] = v[PER - 1];
      __syncthreads();
      if (wid < 2) {
        const double t = packed_block_sum(s_sum + RT * wid);
        if (lane == 0) __stcg(part + 2 * b + wid, t);
      }
    }
  };
  // pair-order sums: vz (if `first`) and vr (if `second`) of pair tid
  const auto publish_pairs = [&](int b, double vz, bool first, double vr, bool second) {
    if (WARPS) {
      if (tid < rows / 2) {
        if (first)
          for (int o = 16; o > 0; o >>= 1) vz += __shfl_down_sync(0xffffffffu, vz, o);
        if (second)
          for (int o = 16; o > 0; o >>= 1) vr += __shfl_down_sync(0xffffffffu, vr, o);
        if (lane == 0) {
          const int at = b * (rows / 64) + wid;
          if (first) __stcg(pair_rz + at, vz);
          if (second) __stcg(pair_rr + at, vr);
        }
      }
    } else if (first || second) {
      __syncthreads();
      s_sum[tid] = vz;
      s_sum[tid + RT] = vr;
      __syncthreads();
      if (wid == 0 && first) {
        const double t = packed_block_sum(s_sum);
        if (lane == 0) __stcg(pair_rz + b, t);
      }
      if (wid == 1 && second) {
        const double t = packed_block_sum(s_sum + RT);
        if (lane == 0) __stcg(pair_rr + b, t);
      }
    }
  };

  const auto total_only = [](double) { return 0.0; };
  const auto beta_of = [&](double v) { return rz > 0.0 ? v / rz : 0.0; };
  if (!SCHW) {  // r to shared memory; z = dinv r takes its place
    for (int k = 0, b = blockIdx.x; b < nslot; ++k, b += gridDim.x) {
      for (int j = tid; j < rows; j += RT) {
        const int64_t i = (int64_t)b * rows + j;
        if (i < n) {
          s_r[k * rows + j] = A.r[i];
          if (!((n & 1) && i == n - 1)) z[i] = __ldg(A.dinv + i) * s_r[k * rows + j];
        }
      }
      if (tail && k == 0) {
        r_tail = A.r[n - 1];
        z[n - 1] = __ldg(A.dinv + n - 1) * r_tail;
      }
    }
  }
  loop_meet(A.bar, target, A.spin_limit, A.withhold, &s_late);

  while (!s_late && res > A.tol && it < A.maxit && it < A.it_stop) {
    const int batch = min(8, A.maxit - it);
    for (int step = 0; step < batch; ++step) {
      const bool test = step == batch - 1;
      // A: q = H p, p.q
      const auto dir = [&](int64_t c) { return fma(beta, __ldcg(pold + c), __ldcg(z + c)); };
      for (int k = 0, b = blockIdx.x; b < nslot; ++k, b += gridDim.x) {
        double v[PER];
#pragma unroll
        for (int h = 0; h < PER; ++h) {
          const int j = tid + h * RT;
          const int64_t i = (int64_t)b * rows + j;
          v[h] = 0.0;
          if (j < rows && i < n) {
            const double q = loop_row(A, i, dir), pi = dir(i);
            pnew[i] = pi;
            if (SCHW) A.q[i] = q;
            else s_q[k * rows + j] = q;
            if (!SCHW && (n & 1) && i == n - 1) sc->qtail = q;
            v[h] = fma(pi, q, 0.0);
          }
        }
        publish_rows(part_pq, b, v);
      }
      loop_meet(A.bar, target, A.spin_limit, A.withhold, &s_late);
      if (s_late) break;
      const double2 pa = loop_total<WARPS>(part_pq, nscal, [&](double v) { return v > 0.0 ? rz / v : 0.0; });
      pq = pa.x;
      alpha = pa.y;

      // B: x, r (pairs of rows), their sums; the patch solves
      if (SCHW) {
        const auto res_of = [&](int m) { return fma(-alpha, __ldcg(A.q + m), __ldcg(r + m)); };
        // 32 patches of one size per warp (a warp of several sizes would take
        // them one after the other), the last warps first: the first ones
        // have the rows
        int k = 1;
        for (int wp = (RT / 32 - 1 - wid) * gridDim.x + blockIdx.x; wp < A.wfirst[kSchwarzDense + 1];
             wp += gridDim.x * (RT / 32)) {
          while (wp >= A.wfirst[k + 1]) ++k;
          const int64_t t = A.g.first[k] + (int64_t)(wp - A.wfirst[k]) * 32 + lane;
          if (t < A.g.first[k + 1]) patch_apply<false>(A.g, t, k, A.mem, A.blk, res_of, A.y);
        }
      }
      for (int k = 0, b = blockIdx.x; b < nslot; ++k, b += gridDim.x) {
        double vz = 0.0, vr = 0.0;
        const int64_t i2 = (int64_t)b * (rows / 2) + tid;
        if (tid < rows / 2 && i2 < n2) {
          double2* xp = reinterpret_cast<double2*>(A.x) + i2;
          const double2 xi = *xp, pi = __ldcg(reinterpret_cast<const double2*>(pnew) + i2);
          *xp = make_double2(fma(alpha, pi.x, xi.x), fma(alpha, pi.y, xi.y));
          double2 qi, ri;
          if (SCHW) {
            qi = __ldcg(reinterpret_cast<const double2*>(A.q) + i2);
            ri = __ldcg(reinterpret_cast<const double2*>(r) + i2);
          } else {
            qi = reinterpret_cast<const double2*>(s_q + k * rows)[tid];
            ri = reinterpret_cast<const double2*>(s_r + k * rows)[tid];
          }
          const double2 ro = make_double2(fma(-alpha, qi.x, ri.x), fma(-alpha, qi.y, ri.y));
          if (SCHW) {
            reinterpret_cast<double2*>(rnew)[i2] = ro;
          } else {
            reinterpret_cast<double2*>(s_r + k * rows)[tid] = ro;
            const double2 di = __ldg(reinterpret_cast<const double2*>(A.dinv) + i2);
            const double2 zo = make_double2(di.x * ro.x, di.y * ro.y);
            reinterpret_cast<double2*>(z)[i2] = zo;
            vz = fma(ro.y, zo.y, fma(ro.x, zo.x, 0.0));
          }
          if (test) vr = fma(ro.y, ro.y, fma(ro.x, ro.x, 0.0));
        }
        if (tail && k == 0) {
          const int64_t i = n - 1;
          A.x[i] = fma(alpha, __ldcg(pnew + i), A.x[i]);
          const double ri = fma(-alpha, __ldcg(SCHW ? A.q + i : &sc->qtail), SCHW ? __ldcg(r + i) : r_tail);
          if (SCHW) {
            rnew[i] = ri;
          } else {
            r_tail = ri;
            const double zi = __ldg(A.dinv + i) * ri;
            z[i] = zi;
            vz = fma(ri, zi, vz);
          }
          if (test) vr = fma(ri, ri, vr);
        }
        publish_pairs(b, vz, !SCHW, vr, test);
      }
      double2 zb;  // r.z and beta
      loop_meet(A.bar, target, A.spin_limit, A.withhold, &s_late);
      if (s_late) break;
      if (test) {
        rr = loop_total<WARPS>(pair_rr, npair, total_only).x;
        __syncthreads();  // every thread has it: the next total may be formed
      }
      if (SCHW) {
        // C: z from the patch values, r.z
          for (int b = blockIdx.x; b < nslot; b += gridDim.x) {
          double v[PER];
#pragma unroll
          for (int h = 0; h < PER; ++h) {
            const int j = tid + h * RT;
            const int64_t i = (int64_t)b * rows + j;
            v[h] = 0.0;
            if (j < rows && i < n) {
              const int s0 = __ldg(A.fslot + 3 * i), s1 = __ldg(A.fslot + 3 * i + 1), s2 = __ldg(A.fslot + 3 * i + 2);
              const double zi = (__ldcg(A.y + s0) + __ldcg(A.y + s1)) + __ldcg(A.y + s2);
              z[i] = zi;
              v[h] = fma(__ldcg(rnew + i), zi, 0.0);
            }
          }
          publish_rows(part_rz, b, v);
        }
        loop_meet(A.bar, target, A.spin_limit, A.withhold, &s_late);
        if (s_late) break;
        zb = loop_total<WARPS>(part_rz, nscal, beta_of);
      } else {
        zb = loop_total<WARPS>(pair_rz, npair, beta_of);
      }
      beta = zb.y;
      rz = zb.x;
      double* t = pold;
      pold = pnew;
      pnew = t;
      if (SCHW) {
        t = r;
        r = rnew;
        rnew = t;
      }
    }
    if (s_late) break;
    it += batch;
    res = sqrt(rr);
    if (pq <= 0.0 && res > A.tol) break;  // breakdown (H not SPD)
  }
  if (!SCHW && !s_late) {  // r back in its place (a further launch reads it)
    for (int k = 0, b = blockIdx.x; b < nslot; ++k, b += gridDim.x)
      for (int j = tid; j < rows; j += RT) {
        const int64_t i = (int64_t)b * rows + j;
        if (i < n && !((n & 1) && i == n - 1)) A.r[i] = s_r[k * rows + j];
      }
    if (tail) A.r[n - 1] = r_tail;
  }
  if (tid == 0 && s_late) atomicOr(&sc->late, 1u);
  if (blockIdx.x == 0 && tid == 0) {
    sc->rz = rz;
    sc->beta = beta;
    sc->alpha = alpha;
    sc->pq = pq;
    sc->rr = rr;
    sc->it = it;
  }
}

constexpr int kLoopSpinLimit = 1 << 21;  // polls (about a microsecond each)
// Test hook (ph_test_pcg_loop): 1 keeps the solver from k_pcg_loop; 2 lets its first
// block never arrive, and the polls of all run out after kLoopTestSpinLimit.
constexpr int kLoopTestSpinLimit = 1 << 12;
std::atomic<int> g_test_pcg_loop{0};
constexpr int kLoopIters = 4096;         // iterations per launch (a multiple of 16: the buffers end where they began)

// Launch k_pcg_loop for the A.n rows: up to kLoopWarpN rows, one block per SM of
// as few warps of 64 rows as that takes (the FP64 work of a phase is spread as
// far as it goes, and no SM has two blocks for the others to wait for); else
// slots of 512 rows.  With a preconditioner, further blocks take patches.
template <bool SCHW, bool WARPS>
cudaError_t loop_launch(LoopArgs& A, cudaStream_t s) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  A.rows = !WARPS ? kLoopRows : 64 * (int)((A.n + 64 * (int64_t)sms - 1) / (64 * (int64_t)sms));
  if (A.rows > (WARPS ? RT : kLoopRows)) return cudaErrorCooperativeLaunchTooLarge;
  const int nslot = (int)((A.n + A.rows - 1) / A.rows);
  const void* fn = (const void*)k_pcg_loop<SCHW, WARPS>;
  // shared memory of one slot per block, and of all slots of a block if the grid then needs more than one
  A.slots = 1;
  int grid = 0;
  for (;;) {
    const size_t smem = SCHW ? 0 : 2 * sizeof(double) * (size_t)A.slots * A.rows;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, RT, smem);
    if (e != cudaSuccess) return e;
    grid = nslot < per_sm * sms ? nslot : per_sm * sms;
    if (grid < 1) return cudaErrorCooperativeLaunchTooLarge;
    if (SCHW || (int64_t)A.slots * grid >= nslot) break;
    ++A.slots;
  }
  if (WARPS && grid < nslot) return cudaErrorCooperativeLaunchTooLarge;
  if (SCHW) {  // one patch warp or two to a block, while blocks have an SM to themselves
    const int want = (A.wfirst[kSchwarzDense + 1] + 1) / 2;
    if (grid < want) grid = want < sms ? want : (grid < sms ? sms : grid);
  }
  const size_t smem = SCHW ? 0 : 2 * sizeof(double) * (size_t)A.slots * A.rows;
  e = cudaMemsetAsync(A.bar, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  void* args[] = {&A};
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(RT), args, smem, s);
}

cudaError_t loop_launch_any(LoopArgs& A, bool schwarz, cudaStream_t s) {
  if (A.n <= kLoopWarpN) return schwarz ? loop_launch<true, true>(A, s) : loop_launch<false, true>(A, s);
  return schwarz ? loop_launch<true, false>(A, s) : loop_launch<false, false>(A, s);
}

// The solve proper on a given workspace (shared by both entry points).
// ell_ok: the solve may allocate its ELL copy of H (not in the allocation-free
// entry point).  P: Schwarz preconditioner (y: its scratch of P->nmem
// doubles, then loop_extra(n) doubles), or null for Jacobi.
ph_status pcg_run(int64_t n, const int32_t* rowptr, const int32_t* colind, const double* values, const double* b,
                  double* x, double rtol, int32_t maxit, int32_t* iters, double* relres, double* work,
                  cudaStream_t s, bool ell_ok, const ph_schwarz* P = nullptr, double* y = nullptr) {
  const size_t nv = vec_stride(n);
  double *r = work, *p = r + nv, *q = p + nv, *dinv = q + nv, *part = dinv + nv;
  Scalars* sc = reinterpret_cast<Scalars*>(part + kPart);
  Scalars h;
  int it = 0;
  Matrix A{rowptr, colind, values, 0, nullptr, nullptr};
  void* ell = nullptr;
  // the whole iteration in one launch (k_pcg_loop) where n allows; with x not
  // 16-byte aligned the sums have another order, kept by the kernels above
  const int hook = g_test_pcg_loop.load(std::memory_order_relaxed);
  bool loop = n <= kLoopMaxN && (reinterpret_cast<uintptr_t>(x) & 15) == 0 && hook != 1;
  cudaError_t e = cudaMemsetAsync(sc, 0, sizeof(Scalars), s);
  if (e == cudaSuccess && ell_ok) {  // width of the longest row (read at the first synchronisation below)
    k_row_width<<<RB, RT, 0, s>>>(n, rowptr, &sc->done);
    e = ph::launched();
  }
  // padding entries stay zero so the pairwise direction update is defined
  if (e == cudaSuccess && nv > (size_t)n) e = cudaMemsetAsync(p + n, 0, sizeof(double) * (nv - n), s);
  if (e == cudaSuccess && nv > (size_t)n) e = cudaMemsetAsync(r + n, 0, sizeof(double) * (nv - n), s);
  if (e == cudaSuccess && nv > (size_t)n) e = cudaMemsetAsync(dinv + n, 0, sizeof(double) * (nv - n), s);
  if (e == cudaSuccess && ell_ok) e = cudaMemcpyAsync(&h, sc, sizeof h, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && ell_ok) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && ell_ok && h.done <= (unsigned)kEllMaxWidth && h.done > 0) {
    const int w = (int)h.done;
    e = ph::alloc_bytes(&ell, (sizeof(double) + sizeof(int32_t)) * (size_t)w * (size_t)n + 16, s);
    if (e == cudaSuccess) {
      double* ev = static_cast<double*>(ell);
      int32_t* ec = reinterpret_cast<int32_t*>(ev + (size_t)w * n);
      k_to_ell<<<RB, RT, 0, s>>>(n, w, rowptr, colind, values, ec, ev);
      e = ph::launched();
      A = Matrix{rowptr, colind, values, w, ec, ev};
    }
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(&sc->done, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) {
    k_pcg_init<<<RB, RT, 0, s>>>(n, rowptr, colind, values, b, x, r, p, dinv, part, sc);
    e = ph::launched();
  }
  if (e == cudaSuccess && P) {  // z = M b, p = z
    e = schwarz_apply(P, r, dinv, y, part, sc, true, s);
    if (e == cudaSuccess && !loop) {  // k_pcg_loop forms p at its first gather
      k_direction_z<<<RB, RT, 0, s>>>(n, p, dinv, sc);
      e = ph::launched();
    }
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, sc, sizeof h, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess || h.bad) {
    if (ell) ph::free_async(ell, s);
    return e != cudaSuccess ? ph::cuda_status(e, "pcg") : PH_ERR_ARG;
  }
  const double bnorm = sqrt(h.bb);
  double res = bnorm;
  while (loop && res > rtol * bnorm && it < maxit) {
    LoopArgs L;
    L.n = n;
    L.w = A.w;
    L.rowptr = rowptr;
    L.col = A.w ? A.ecol : colind;
    L.val = A.w ? A.eval : values;
    L.x = x;
    L.r = r;
    L.p = p;
    L.q = P ? q : nullptr;
    L.z = P ? dinv : nullptr;
    L.r2 = P ? y + P->nmem + (P->nmem & 1) : nullptr;
    L.p2 = P ? L.r2 + nv : q;
    L.dinv = dinv;
    L.part = part;
    L.bar = &sc->bar;
    L.sc = sc;
    L.tol = rtol * bnorm;
    L.res = res;
    L.it = it;
    L.it_stop = it + kLoopIters;
    L.maxit = maxit;
    L.spin_limit = hook == 2 ? kLoopTestSpinLimit : kLoopSpinLimit;
    L.withhold = hook == 2 ? 0 : -1;
    L.mem = P ? P->mem : nullptr;
    L.fslot = P ? P->fslot : nullptr;
    L.blk = P ? P->blk : nullptr;
    L.y = y;
    if (P) {
      L.g = P->g;
      L.wfirst[0] = L.wfirst[1] = 0;
      for (int k = 1; k <= kSchwarzDense; ++k) L.wfirst[k + 1] = L.wfirst[k] + (int)((P->g.count[k] + 31) / 32);
    }
    e = loop_launch_any(L, P != nullptr, s);
    if (e == cudaErrorCooperativeLaunchTooLarge && it == 0) {  // no room for the grid: the kernels below
      (void)cudaGetLastError();
      e = cudaSuccess;
      loop = false;
      if (P) {
        k_direction_z<<<RB, RT, 0, s>>>(n, p, dinv, sc);
        e = ph::launched();
      }
      break;
    }
    if (e == cudaSuccess) e = ph::launched();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, sc, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess || h.late) {
      if (ell) ph::free_async(ell, s);
      return e != cudaSuccess ? ph::cuda_status(e, "pcg") : PH_ERR_TIMEOUT;
    }
    it = h.it;
    res = sqrt(h.rr);
    if (iters) *iters = it;
    if (h.pq <= 0.0 && res > rtol * bnorm) break;  // breakdown (H not SPD)
  }
  if (e != cudaSuccess) {
    if (ell) ph::free_async(ell, s);
    return ph::cuda_status(e, "pcg");
  }
  while (!loop && res > rtol * bnorm && it < maxit) {
    const int batch = (maxit - it) < 8 ? (maxit - it) : 8;
    for (int i = 0; i < batch && e == cudaSuccess; ++i)
      e = pcg_iteration(n, A, x, r, p, q, dinv, part, sc, P, y, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, sc, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      if (ell) ph::free_async(ell, s);
      return ph::cuda_status(e, "pcg");
    }
    it += batch;
    res = sqrt(h.rr);
    if (iters) *iters = it;
    if (h.pq <= 0.0 && res > rtol * bnorm) break;  // breakdown (H not SPD)
  }
  if (ell) ph::free_async(ell, s);
  if (iters) *iters = it;
  if (relres) *relres = bnorm > 0.0 ? res / bnorm : 0.0;
  return res > rtol * bnorm ? PH_ERR_NOT_CONVERGED : PH_OK;
}

}  // namespace

using namespace ph;

extern "C" ph_status ph_test_pcg_loop(int mode) {
  if (mode < 0 || mode > 2) return PH_ERR_ARG;
  g_test_pcg_loop.store(mode);
  return PH_OK;
}

extern "C" ph_status ph_solve_pcg(int64_t n, const int32_t* rowptr, const int32_t* colind, const double* values,
                                  const double* b, double* x, double rtol, int32_t maxit, int32_t* iters,
                                  double* relres, void* stream) {
  if (iters) *iters = 0;
  if (relres) *relres = 0.0;
  if (n < 0 || !(rtol >= 0.0) || maxit < 0) return PH_ERR_ARG;
  if (n == 0) return PH_OK;
  if (!rowptr || !colind || !values || !b || !x) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  double* work = nullptr;
  cudaError_t e = alloc(&work, workspace_doubles(n), s);
  if (e != cudaSuccess) return cuda_status(e, "pcg alloc");
  const ph_status st = pcg_run(n, rowptr, colind, values, b, x, rtol, maxit, iters, relres, work, s, true);
  free_async(work, s);
  return st;
}

extern "C" ph_status ph_solve_pcg_schwarz(const ph_mesh* m, const double* values, const ph_schwarz* P,
                                          const double* b, double* x, double rtol, int32_t maxit, int32_t* iters,
                                          double* relres, void* stream) {
  if (iters) *iters = 0;
  if (relres) *relres = 0.0;
  if (!m || !P || P->L != m->L || !(rtol >= 0.0) || maxit < 0) return PH_ERR_ARG;
  const int64_t n = m->L;
  if (n == 0) return PH_OK;
  if (!values || !b || !x) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  double* work = nullptr;
  const size_t wd = workspace_doubles(n);
  cudaError_t e = alloc(&work, wd + (size_t)P->nmem + loop_extra(n), s);
  if (e != cudaSuccess) return cuda_status(e, "pcg alloc");
  const ph_status st =
      pcg_run(n, m->rowptr, m->colind, values, b, x, rtol, maxit, iters, relres, work, s, true, P, work + wd);
  free_async(work, s);
  return st;
}

// ---------------------------------------------------------------------------
// Iterative refinement: the solve of H x = b to fp64 accuracy.  A plain fp64
// solve stops at an error of about cond(H) eps (~3e-9 on the jittered
// checkerboard workload); refining with a residual computed in double-word
// arithmetic takes x to the fp64 rounding of the exact solution of the system
// as given (Wilkinson's iterative refinement with an extra-precise residual).
// ---------------------------------------------------------------------------
namespace {

// Knuth's TwoSum (s + e = a + b exactly) and the fma split of a product
// (p + e = a b exactly).
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// r = b - H x: each row's sum is accumulated as an unevaluated pair (sum,
// compensation), the products split exactly by fma (Ogita, Rump and Oishi's
// Dot2), so r is as accurate as a sum formed in twice the precision and
// rounded once.
__global__ void __launch_bounds__(RT) k_residual_dw(int64_t n, const int32_t* __restrict__ rowptr,
                                                    const int32_t* __restrict__ colind,
                                                    const double* __restrict__ val, const double* __restrict__ x,
                                                    const double* __restrict__ b, double* __restrict__ r) {
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    double sh = b[i], sl = 0.0;
    for (int j = rowptr[i]; j < rowptr[i + 1]; ++j) {
      const double v = val[j], xv = x[colind[j]];
      const double p = v * xv, pe = fma(v, xv, -p);
      double t, te;
      two_sum(sh, -p, t, te);
      sh = t;
      sl += te - pe;
    }
    r[i] = sh + sl;
  }
}

// x += d, with the sums d.d and x.x (new x) in a fixed order; the last block
// stores them in sc->pq (d.d) and sc->rr (x.x).
__global__ void __launch_bounds__(RT) k_add_correction(int64_t n, double* __restrict__ x,
                                                       const double* __restrict__ d, double* __restrict__ part,
                                                       Scalars* __restrict__ sc) {
  double dd = 0.0, xx = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)RB * RT) {
    const double di = d[i], xi = x[i] + di;
    x[i] = xi;
    dd = fma(di, di, dd);
    xx = fma(xi, xi, xx);
  }
  dd = block_sum(dd);
  xx = block_sum(xx);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = dd;
    part[RB + blockIdx.x] = xx;
  }
  if (last_block(&sc->done)) {
    const double dd_t = sum_partials(part, 0);
    const double xx_t = sum_partials(part, RB);
    if (threadIdx.x == 0) {
      sc->pq = dd_t;
      sc->rr = xx_t;
      sc->done = 0;
    }
  }
}

}  // namespace

extern "C" ph_status ph_solve_refined(const ph_mesh* m, const double* values, const ph_schwarz* P, const double* b,
                                      double* x, double tol, double inner_rtol, int32_t max_steps, int32_t maxit,
                                      int32_t* steps, int32_t* iters, double* correction, void* stream) {
  if (steps) *steps = 0;
  if (iters) *iters = 0;
  if (correction) *correction = 0.0;
  if (!m || (P && P->L != m->L) || !(tol >= 0.0) || !(inner_rtol >= 0.0) || max_steps < 1 || maxit < 0)
    return PH_ERR_ARG;
  const int64_t n = m->L;
  if (n == 0) return PH_OK;
  if (!values || !b || !x) return PH_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t wd = workspace_doubles(n), nv = vec_stride(n);
  // PCG workspace, its Schwarz scratch, then r, d, partial sums and scalars
  const size_t scratch = P ? ((size_t)P->nmem + loop_extra(n) + 31) & ~(size_t)31 : 0;
  const size_t total = wd + scratch + 2 * nv + kPart + (sizeof(Scalars) + 7) / 8;
  double* work = nullptr;
  cudaError_t e = alloc(&work, total, s);
  if (e != cudaSuccess) return cuda_status(e, "refine alloc");
  double* y = work + wd;
  double* r = y + scratch;
  double* d = r + nv;
  double* part = d + nv;
  Scalars* sc = reinterpret_cast<Scalars*>(part + kPart);
  ph_status st = PH_OK;
  int total_it = 0, step = 0;
  double corr = INFINITY;
  e = cudaMemsetAsync(x, 0, sizeof(double) * n, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(sc, 0, sizeof(Scalars), s);
  while (e == cudaSuccess && step < max_steps) {
    ++step;
    int32_t it = 0;
    // correction equation H d = r; an inner solve that stops at its
    // iteration cap still improves x, so only other errors end the loop
    const ph_status inner = P ? pcg_run(n, m->rowptr, m->colind, values, r, d, inner_rtol, maxit, &it, nullptr,
                                        work, s, true, P, y)
                              : pcg_run(n, m->rowptr, m->colind, values, r, d, inner_rtol, maxit, &it, nullptr,
                                        work, s, true);
    total_it += it;
    if (inner != PH_OK && inner != PH_ERR_NOT_CONVERGED) {
      st = inner;
      break;
    }
    k_add_correction<<<RB, RT, 0, s>>>(n, x, d, part, sc);
    e = launched();
    Scalars h;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, sc, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) break;
    corr = h.rr > 0.0 ? sqrt(h.pq / h.rr) : 0.0;
    if (corr <= tol) break;
    k_residual_dw<<<RB, RT, 0, s>>>(n, m->rowptr, m->colind, values, x, b, r);
    e = launched();
  }
  free_async(work, s);
  if (steps) *steps = step;
  if (iters) *iters = total_it;
  if (correction) *correction = corr;
  if (e != cudaSuccess) return cuda_status(e, "ph_solve_refined");
  if (st != PH_OK) return st;
  return corr <= tol ? PH_OK : PH_ERR_NOT_CONVERGED;
}

// y = H x
__global__ void k_spmv(int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                       const double* __restrict__ val, const double* __restrict__ x, double* __restrict__ y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int j = rowptr[i]; j < rowptr[i + 1]; ++j) s = fma(val[j], x[colind[j]], s);
  y[i] = s;
}

extern "C" ph_status ph_spmv(int64_t n, const int32_t* rowptr, const int32_t* colind, const double* values,
                             const double* x, double* y, void* stream) {
  if (n < 0) return PH_ERR_ARG;
  if (n == 0) return PH_OK;
  if (!rowptr || !colind || !values || !x || !y) return PH_ERR_ARG;
  k_spmv<<<grid_for(n), kThreads, 0, (cudaStream_t)stream>>>(n, rowptr, colind, values, x, y);
  return cuda_status(launched(), "ph_spmv");
}

// ---------------------------------------------------------------------------
// ph_solve_pcg_noalloc: the iteration above with its workspace in a fixed
// device array instead of the library's pool, for callers that must not
// allocate device memory.  It reuses the kernels above unchanged.
// ---------------------------------------------------------------------------
#include <string.h>

#include <mutex>

// r, p, q, dinv (4 vectors of PH_PCG_NOALLOC_MAX_N doubles, a multiple of 32),
// partial sums and scalars: the layout of workspace_doubles().
static_assert(PH_PCG_NOALLOC_MAX_N % 32 == 0, "vector stride");
static constexpr size_t kNoAllocDoubles = 4 * (size_t)PH_PCG_NOALLOC_MAX_N + kPart + (sizeof(Scalars) + 7) / 8;
static __device__ __align__(256) double g_pcg_noalloc_work[kNoAllocDoubles];

static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[64];

// Device address of g_pcg_noalloc_work on the current device, looked up once per
// device (the host-side symbol is only a stand-in and must not reach a kernel).
static ph_status noalloc_workspace(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_status(e, "ph_solve_pcg_noalloc: cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    ph::set_error_text("ph_solve_pcg_noalloc: device index >= 64 (the workspace address table holds 64 devices)");
    return PH_ERR_ARG;
  }
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_pcg_noalloc_work);
    if (e != cudaSuccess) return cuda_status(e, "ph_solve_pcg_noalloc: cudaGetSymbolAddress");
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return PH_OK;
}

extern "C" ph_status ph_solve_pcg_noalloc(int64_t n, const int32_t* rowptr, const int32_t* colind,
                                          const double* values, const double* b, double* x, double rtol,
                                          int32_t maxit, int32_t* iters, double* relres, void* stream) {
  if (iters) *iters = 0;
  if (relres) *relres = 0.0;
  if (n < 0 || !(rtol >= 0.0) || maxit < 0) return PH_ERR_ARG;
  if (n > PH_PCG_NOALLOC_MAX_N) {
    ph::set_error_text("ph_solve_pcg_noalloc: n exceeds PH_PCG_NOALLOC_MAX_N (the fixed workspace)");
    return PH_ERR_ARG;
  }
  if (n == 0) return PH_OK;
  if (!rowptr || !colind || !values || !b || !x) return PH_ERR_ARG;
  double* work = nullptr;
  ph_status st = noalloc_workspace(&work);
  if (st != PH_OK) return st;
  return pcg_run(n, rowptr, colind, values, b, x, rtol, maxit, iters, relres, work, (cudaStream_t)stream, false);
}
