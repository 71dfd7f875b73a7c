// Reductions at the end of the time DFTs (last-CTA pattern: no CTA waits for another).
#pragma once

#include "pd_control.cuh"
#include "pd_internal.h"

namespace pd {

// Sum of squares of the transformed data (per thread: ss), reduced over the launch: each
// CTA stores its partial, and the last CTA to finish (no CTA waits for another) adds the
// partials in a fixed order and stores the square root into *rn.dst.
__device__ __forceinline__ void rhs_norm_finish(float ss, const RhsNorm &rn) {
  __shared__ double red[32];
  __shared__ int last;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  // binary32 within a warp (a reference scale; FP64 adds cost GB300's FP64 pipe), a quarter of it, so
  // that a warp's up to 2048 squares overflow no earlier than 512 of their size would
  ss = warp_sum(0.25f * ss);
  if (l == 0) red[w] = 4.0 * (double)ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += red[i];
    rn.part[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(rn.counter, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += __ldcg(rn.part + i);
  t = warp_sum(t);
  __syncthreads();  // red is reused
  if (l == 0) red[w] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s2 = 0.0;
    for (int i = 0; i < nw; ++i) s2 += red[i];
    *rn.dst = sqrt(s2);
    *rn.counter = 0;
  }
}

// Sums of squares of an inverse transform's output (per thread: ss, all of one column, the
// columns x0 .. x0 + TX - 1 going round the threads), per column and over the launch, and the
// refinement decision in the last CTA (fin).  blockDim.x is a multiple of 32 and of TX, at most NT.
template <int TX, int NT>
__device__ __forceinline__ void c2r_finish(double ss, int64_t x0, int64_t ncols, double *colsum, double *norm_part,
                                           const StepFinish &fin) {
  if (colsum) {
    // per-column sums of squares: blockDim.x is a multiple of TX, so every element a
    // thread wrote lies in column threadIdx.x % TX
    __shared__ double cred[NT];
    cred[threadIdx.x] = ss;
    __syncthreads();
    if ((int)threadIdx.x < TX) {
      double t = 0.0;
      for (int i = threadIdx.x; i < (int)blockDim.x; i += TX) t += cred[i];
      if (x0 + threadIdx.x < ncols) colsum[x0 + threadIdx.x] = t;
    }
  }
  if (norm_part) {
    const double sd = warp_sum(ss);
    __shared__ double red[32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = sd;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
      norm_part[blockIdx.x] = t;
    }
    if (fin.enabled) {
      // the last CTA to finish (no CTA waits) sums the squares and decides
      __shared__ int last;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) last = atomicAdd(fin.counter, 1) == (int)gridDim.x - 1;
      __syncthreads();
      if (last) {
        __threadfence();
        // every thread loads its share at once (the partials sit in L2, possibly on the
        // other die: one round trip instead of one per partial), then a fixed-order sum
        double t = 0.0;
#pragma unroll 4
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += norm_part[i];
        t = warp_sum(t);
        if (l == 0) red[w] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
          t = 0.0;
          for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
          fin.scal[S_D2] = t;
          *fin.counter = 0;
          refine_decide(fin.scal, fin.flags, fin.rc, fin.use_handle, fin.h);
        }
      }
    }
  }
}

}  // namespace pd
