// Deterministic grid-wide reductions shared by the bulk kernels.
//
// Each block writes its partial sums into a column-major table
//   part[col * ps + block]            (ps >= gridDim.x)
// and the last block to finish (atomic ticket) sums every column with all
// its warps: lane l adds blocks l, l+32, ... and a fixed shuffle tree
// finishes, so the result does not depend on block scheduling.
#pragma once

#include "kx_internal.cuh"

namespace kx {

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// True in every thread of the last block to finish; that block then sees
// every other block's partials.
__device__ __forceinline__ bool last_block(unsigned* counter) {
  __shared__ bool am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned t = atomicAdd(counter, 1u);
    am_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (am_last) __threadfence();
  return am_last;
}

// Block sum of one double per thread, written to part[col * ps + bid].
__device__ __forceinline__ void block_partial_at(double x, double* part, int ps, int col, int bid) {
  __shared__ double red[NWARPS];
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NWARPS; ++w) t += red[w];
    part[(int64_t)col * ps + bid] = t;
  }
  __syncthreads();
}

// Block sum of one double per thread, written to part[col * ps + blockIdx.x].
__device__ __forceinline__ void block_partial(double x, double* part, int ps, int col) {
  __shared__ double red[NWARPS];
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < NWARPS; ++w) t += red[w];
    part[(int64_t)col * ps + blockIdx.x] = t;
  }
  __syncthreads();
}

// Warp sums of eight values: lane l ends with the sum of value
// column_of_lane8(l) (four lanes hold each).  Nine additions instead of forty
// for eight separate sums: the lanes exchange halves of the values they keep.
template <typename T>
__device__ __forceinline__ T warp_sum8(T* p, int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const T keep = b4 ? p[t + 4] : p[t], send = b4 ? p[t] : p[t + 4];
    p[t] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const T keep = b3 ? p[t + 2] : p[t], send = b3 ? p[t] : p[t + 2];
    p[t] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  const T keep = b2 ? p[1] : p[0], send = b2 ? p[0] : p[1];
  T x = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x;
}
__device__ __forceinline__ int column_of_lane8(int lane) { return lane >> 2; }

// a^2 + b^2 of the phase entries, rounded alike in every kernel that adds it
// (as are the entries themselves: which kernel finalises a step depends on how
// many slots run, and the bits must not).
__device__ __forceinline__ double phase_norm2(double a, double b) { return fma(a, a, __dmul_rn(b, b)); }

// Finalisation of step j-1's pass B at the start of step j's pass A: every
// block sums the same nbb partials in the same order, so all reach the same
// h_{j,j-1} and the same breakdown decision; block 0 (rec) records them.
// Returns false where the process stops (lucky breakdown or a non-finite
// norm); *sj receives scale_j = 1/h.  An augmented process (AUG, the slot's
// aug set) also gives the two phase entries of column j their Gram-Schmidt
// update, from the raw entries that follow from column j-1's; *aj receives
// the first (the others may not read what block 0 records).
template <int AUG, typename T>
__device__ __forceinline__ bool fin_prev_b(const Slot<T>& s, int j, int ldh, int nbb, double btol, bool rec,
                                           double* sj, double* aj) {
  double x = 0.0, pa = 0.0, pb = 0.0;
  const int tid = threadIdx.x, nw = blockDim.x >> 5;
  for (int b = tid; b < nbb; b += blockDim.x) x += __ldcg(s.part + (int64_t)FINB_COL * s.ps + b);
  const bool augm = AUG && s.st->aug;
  if (AUG && augm)
    for (int col = tid; col < j; col += blockDim.x) {
      const double cc = s.H[col + (int64_t)(j - 1) * ldh] * s.scale[col];
      pa += cc * s.aug[2 * col];
      pb += cc * s.aug[2 * col + 1];
    }
  __shared__ double red[3][NWARPS];
  __shared__ double res, resa;
  __shared__ int stop;
  x = warp_sum(x);
  if (AUG) {
    pa = warp_sum(pa);
    pb = warp_sum(pb);
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = x;
    red[1][tid >> 5] = pa;
    red[2][tid >> 5] = pb;
  }
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0, a = 0.0, b = 0.0;
    for (int w = 0; w < nw; ++w) tot += red[0][w];
    if (AUG && augm) {
      double sa = 0.0, sb = 0.0;
      for (int w = 0; w < nw; ++w) {
        sa += red[1][w];
        sb += red[2][w];
      }
      const double W = s.st->omega, sp = s.scale[j - 1];
      a = __dmul_rn(-W * sp, s.aug[2 * (j - 1) + 1]) - sa;
      b = __dmul_rn(W * sp, s.aug[2 * (j - 1)]) - sb;
      tot += phase_norm2(a, b);
    }
    const double h = sqrt(tot);
    int stp = 0;
    double scl = 0.0;
    if (!isfinite(h)) stp = 2;
    else if (h <= btol * s.st->wmax) stp = 1;   // invariant subspace: the projection is exact
    else scl = 1.0 / h;
    if (rec) {
      s.H[j + (int64_t)(j - 1) * ldh] = h;
      s.st->m_done = j;
      s.scale[j] = scl;
      if (AUG) {
        s.aug[2 * j] = a;
        s.aug[2 * j + 1] = b;
      }
      if (stp == 2) s.st->status = KX_ENONFINITE;
      if (stp || abort_requested(s.st)) s.st->done = 1;
    }
    res = scl;
    resa = a;
    stop = stp;
  }
  __syncthreads();
  *sj = res;
  *aj = resa;
  return stop == 0;
}

// In the last block: tot[c] = sum over blocks of part[c * ps + b], c < ncols.
__device__ __forceinline__ void grid_columns(const double* part, int ps, int ncols, double* tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = gridDim.x;
  for (int col = warp; col < ncols; col += NWARPS) {
    const double* p = part + (int64_t)col * ps;
    double s0 = 0.0, s1 = 0.0;
    int b = lane;
    for (; b + 32 < nb; b += 64) {
      s0 += __ldcg(p + b);
      s1 += __ldcg(p + b + 32);
    }
    if (b < nb) s0 += __ldcg(p + b);
    s0 = warp_sum(s0 + s1);
    if (lane == 0) tot[col] = s0;
  }
  __syncthreads();
}

}  // namespace kx
