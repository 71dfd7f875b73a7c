// Per-problem scaling for batched plans: `batch` independent problems share one
// plan as a block-diagonal problem (slot b = columns [b*nxm, (b+1)*nxm) of every
// time row).  The Krylov and refinement stopping rules measure the whole stack, so
// every problem is solved scaled to unit Frobenius norm (up to a factor of two).  The
// scale factors are powers of two, found here; the transforms apply them on load and
// undo them on store (SlotScale), by integer work on the exponent field.  (As passes of
// their own, scaling G and unscaling U took 184 of 2913 us on 32 x heat1d_1023x1024.)
#include <algorithm>

#include "pd_internal.h"

namespace pd {

// part[b * nc + c] = sum over time rows t = c, c + nc, ... of slot b's squares, in binary64.
//
// Bound by GB300's FP64 pipe (2 us per million squares; HBM 1.2).  W lanes (a power of two) share a row;
// eight loads are in flight per thread, and the squares go into two chains.  Measured with the exponents
// kernel, against one load at a time: 32 x 1023 x 1024 100 -> 83 us, 8 x 2048 x 256 33.6 -> 25.6 us.
// (Binary32 squares took 77 and 25 us, and lost half of the digits.)
__global__ void __launch_bounds__(256) k_batch_sumsq(const double *__restrict__ X, int64_t nt, int64_t ld, int nxm,
                                                     int nc, double *__restrict__ part, int W) {
  grid_dep_wait();
  const int c = blockIdx.x, b = blockIdx.y;
  const int i0 = (int)threadIdx.x & (W - 1);
  const int64_t dt = (int64_t)nc * (256 / W);
  const double *row = X + (int64_t)b * nxm;
  double s0 = 0.0, s1 = 0.0;
  int64_t t = c + (int64_t)nc * (threadIdx.x / W);
  int i = i0;
  while (t < nt) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = t < nt && i < nxm ? row[t * ld + i] : 0.0;
      i += W;
      if (i >= nxm) {
        i = i0;
        t += dt;
      }
    }
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      s0 = fma(v[u], v[u], s0);
      s1 = fma(v[u + 1], v[u + 1], s1);
    }
  }
  __shared__ double red[8];
  const double s = warp_sum(s0 + s1);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    part[(int64_t)b * nc + c] = t;
  }
}

// ex[b] = -round(log2 ||slot b||_F): slot b is multiplied by 2^ex[b] before the solve
// and its solution by 2^-ex[b] after it (0 for an all-zero or non-finite slot).
// zero[b] = 1 for an all-zero slot: its solution is stored as exact zeros, whatever rounding-level
// values a transform that pairs columns (the DST, the general time DFTs) leaves in its columns, and
// it takes no part in the refinement decision.
__global__ void k_batch_exponents(int batch, int nc, const double *__restrict__ part, int *__restrict__ ex,
                                  int *__restrict__ zero, const double *G, const double **gslot) {
  grid_dep_wait();
  const int b = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;  // a warp per slot
  if (blockIdx.x == 0 && threadIdx.x == 0) *gslot = G;
  if (b >= batch) return;
  double s = 0.0;
  for (int c = lane; c < nc; c += 32) s += part[(int64_t)b * nc + c];
  s = warp_sum(s);
  if (lane) return;
  int e = 0;
  if (s > 0.0 && isfinite(s)) {
    int e2;
    frexp(s, &e2);  // s = f 2^e2, f in [0.5, 1): ||x|| ~ 2^(e2/2)
    e = -(e2 / 2);
  }
  ex[b] = e;
  zero[b] = s == 0.0 ? 1 : 0;
}

void launch_batch_exponents(Ctx &c, const double *G, int64_t nt, int batch, int nxm, int nc, double *part, int *ex,
                            int *zero, const double **gslot) {
  const int64_t ld = (int64_t)batch * nxm;
  int W = 32;
  while (W < nxm && W < 256) W *= 2;
  c.launch("batch_scale", (double)nt * ld * 8.0, [&] {
    pdl_launch(c.pdl, k_batch_sumsq, dim3(nc, batch), dim3(256), 0, c.stream, G, nt, ld, nxm, nc, part, W);
  });
  c.launch("batch_scale", 0.0, [&] {
    pdl_launch(c.pdl, k_batch_exponents, dim3((batch + 7) / 8), dim3(256), 0, c.stream, batch, nc, part, ex, zero, G,
               gslot);
  });
}

// A problem joining a running batch (join[b]): its U slot starts at zero and its refinement
// state restarts; so does every unused slot (zero[b]: an all-zero right-hand side, whose U
// may hold anything).  The other slots are not touched.
__global__ void __launch_bounds__(256) k_member_join(double *U, int nt, int ld, int nxm, int batch, const int *__restrict__ join,
                                                     const int *__restrict__ zero, int *msw, double *prev, double *ref2,
                                                     int *mex, int *mconv) {
  grid_dep_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.y == 0 && j < batch && (join[j] || zero[j])) {  // (an unused slot's mex may be stale)
    msw[j] = 0;
    prev[j] = 0.0;
    ref2[j] = 0.0;
    mex[j] = 0;
    mconv[j] = 0;
  }
  if (j >= ld) return;
  const int b = j / nxm;
  if (join[b] || zero[b])
    for (int t = blockIdx.y; t < nt; t += gridDim.y) U[(int64_t)t * ld + j] = 0.0;
}

void launch_member_join(Ctx &c, double *U, int64_t nt, int batch, int nxm, const int *join, const int *zero, int *msw,
                        double *prev, double *ref2, int *mex, int *mconv) {
  const int64_t ld = (int64_t)batch * nxm;
  // enough CTAs to fill the SMs: most calls join few slots or none, and one CTA per row and 256
  // columns spent its time on CTAs that had nothing to do (8 x 2048 x 256: 14.3 -> 7.2 us)
  const unsigned gx = (unsigned)((std::max<int64_t>(ld, batch) + 255) / 256);
  const dim3 grid(gx, (unsigned)std::min<int64_t>(nt, std::max<int64_t>(1, 8 * sm_count() / gx)));
  c.launch("batch_join", (double)nt * ld * 8.0, [&] {
    pdl_launch(c.pdl, k_member_join, grid, dim3(256), 0, c.stream, U, (int)nt, (int)ld, nxm, batch, join, zero, msw, prev, ref2,
               mex, mconv);
  });
}

// out[t][j] = in[t][j] * s[j] (in place allowed): the diagonal mass matrix's symmetric
// scaling of G (s = M^{-1/2}) and of U (s = M^{-1/2}, from w = M^{1/2} u).
__global__ void k_col_scale(const double *in, double *out, int nb, const double *__restrict__ s) {
  grid_dep_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nb) return;
  const int64_t o = (int64_t)blockIdx.y * nb + j;
  out[o] = in[o] * s[j];
}

void launch_col_scale(Ctx &c, const double *in, double *out, int64_t nt, int64_t nb, const double *s) {
  const dim3 grid((unsigned)((nb + 255) / 256), (unsigned)nt);
  c.launch("mass_scale", (double)nt * nb * 16.0,
           [&] { pdl_launch(c.pdl, k_col_scale, grid, dim3(256), 0, c.stream, in, out, (int)nb, s); });
}

}  // namespace pd
