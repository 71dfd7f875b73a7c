// Parallel-in-time loop in FP64 for plans with many (frequency, block) systems: one thread per
// shifted system ((1 - pi_k) I + tau K) y = r, a Thomas sweep with factors stored per operator.
//
// Bound by GB300's FP64 pipe, so the layout is the one with the fewest FP64 operations: 10 per row
// (6 forward, 4 backward; k_pint's partitioned elimination takes about 20) and no reduction across
// lanes for the dots g_k = V_m^T h_k, which every thread keeps for its own frequency (2 per row and
// basis vector).  A warp's lanes are consecutive frequencies of one block (two at a block's end):
//  - factors 1/pivot and up/pivot, and the forward sweep's result, lie as [row][system], so a warp
//    reads and writes 512 contiguous bytes;
//  - a row of a vector (r = v_{m+1}, V_q, tau K) is one address for the whole warp;
//  - rows of a spectrum (R, Y) are 16 bytes per lane and row; a thread's kRows consecutive rows of a
//    group fill 128 bytes, merged by the caches.
// A warp needs no other warp, so it hides latency by loading a group of rows ahead.
// The weighted sum over the frequencies (b of eq. 7) is left to the column sum over the stored
// solutions (k_zsum): a reduction over lanes would cost more FP64 operations than the solve.
//
// Measured per launch, k_pint with stored factors -> here (one GB300; b pass / dots over a solve's steps):
//   255 x 255 x 256 (216 systems per SM, 255 rows)  590 / 688 us -> 197 / 324 us; floor 167 / 290 (the FP64
//                                                   operations at 1.65 per cycle and SM)
//   63 x 63 x 512 (107 per SM, 63 rows)             130 / 152 us -> 40 / 61 us
//   1023 x 63 x 512 (107 per SM, 1023 rows)         1566 / 1842 us -> 547 / 972 us
//   64 problems of 511 x 512 (108 per SM)           649 / 690 us -> 277 / 432 us
// A system is a serial chain, so too few of them leave the pipe idle: at 54 per SM 177 / 268 -> 129 / 328 us
// (255 x 63 x 256) and a solve of 32 problems of 511 x 512 took 8.00 ms instead of 7.87 ms; at 26 per SM
// 106 / 177 -> 126 / 462 us.  The line is at 96, three warps per SM (pint_sys_fits).
#include <algorithm>

#include "pd_internal.h"

namespace pd {

// One-warp CTAs spread over the SMs most evenly (255 x 255 x 256, all solves' dots: 4.9 ms; 5.4 ms in CTAs
// of 64 to 256 threads).
constexpr int kSysThreads = 32;
// Rows whose loads are issued together, one group ahead (8: 5.7 ms; 2: the b pass 253 us instead of 197)
constexpr int kSysRows = 4;
// Basis vectors whose dots ride along with the backward sweep
constexpr int kSysDots = 12;
static int64_t sys_ld(const PintGeom &g) { return ((int64_t)g.nf * g.nblk + 31) / 32 * 32; }
size_t pint_sys_scratch(const PintGeom &g) { return (size_t)sys_ld(g) * g.blen; }
bool pint_sys_fits(int nf, int nblk) { return (int64_t)nf * nblk >= (int64_t)96 * sm_count(); }

// Factors of every system: rd[e][s] = 1 / pivot, cc[e][s] = up / pivot.
__global__ void __launch_bounds__(kSysThreads) k_sys_factor(PintGeom g, PintArgs<double> a, cpx<double> *__restrict__ rd,
                                                            cpx<double> *__restrict__ cc, int64_t ld) {
  grid_dep_wait();
  const int64_t s = (int64_t)blockIdx.x * kSysThreads + threadIdx.x;
  if (s >= (int64_t)g.nf * g.nblk) return;
  const int blk = (int)(s / g.nf), k = (int)(s - (int64_t)blk * g.nf);
  const int64_t off = (int64_t)blk * g.blen;
  const double2 sk = a.shift[k];
  cpx<double> c = mk<double>(0.0, 0.0);
  for (int e = 0; e < g.blen; ++e) {
    const cpx<double> d = mk<double>(sk.x + a.tdiag[off + e], sk.y);
    const cpx<double> r = recip(e ? fnms_r(d, a.tlo[off + e], c) : d);
    c = scal(a.tup[off + e], r);
    rd[(int64_t)e * ld + s] = r;
    cc[(int64_t)e * ld + s] = c;
  }
}

// x_m = V_m y_m (before the final loop's solves, which subtract it)
__global__ void __launch_bounds__(256) k_sys_xm(PintGeom g, PintArgs<double> a) {
  grid_dep_wait();
  if (a.skip_flag && *a.skip_flag) return;
  if (a.skip_flag2 && *a.skip_flag2) return;
  const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (j >= (int64_t)g.nblk * g.blen) return;
  const int blk = (int)(j / g.blen);
  const double *y = a.xm_y + (int64_t)(blk / (a.xm_bpm > 1 ? a.xm_bpm : 1)) * a.xm_ldy;
  const int m = *a.xm_count;
  double v = 0.0;
  for (int q = 0; q < m; ++q) v += y[q] * a.V[(int64_t)q * a.ldv + j];
  a.xm_out[j] = v;
}

// Backward sweep, x_e = y_e - cc_e x_{e+1}, with the dots of the first min(m, NQ) basis vectors.
template <int NQ>
__device__ __forceinline__ void sys_backward(const cpx<double> *__restrict__ cc, const cpx<double> *y, int64_t ld,
                                             cpx<double> *Y, int blen, const double *__restrict__ V, int64_t ldv, int m,
                                             double2 *gp) {
  constexpr int U = kSysRows;
  double sx[NQ > 0 ? NQ : 1], sy[NQ > 0 ? NQ : 1];
#pragma unroll
  for (int q = 0; q < NQ; ++q) sx[q] = sy[q] = 0.0;
  cpx<double> nc[U], ny[U];
  auto load = [&](int e0) {  // rows e0, e0 - 1, ..
#pragma unroll
    for (int i = 0; i < U; ++i) {
      if (e0 - i >= 0) {
        nc[i] = cc[(int64_t)(e0 - i) * ld];
        ny[i] = y[(int64_t)(e0 - i) * ld];
      }
    }
  };
  cpx<double> x = mk<double>(0.0, 0.0);
  load(blen - 1);
  for (int e0 = blen - 1; e0 >= 0; e0 -= U) {
    cpx<double> c[U], r[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      c[i] = nc[i];
      r[i] = ny[i];
    }
    load(e0 - U);
    double vv[U][NQ > 0 ? NQ : 1];
#pragma unroll
    for (int i = 0; i < U; ++i)
#pragma unroll
      for (int q = 0; q < NQ; ++q) vv[i][q] = q < m && e0 >= i ? V[(int64_t)q * ldv + e0 - i] : 0.0;
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int e = e0 - i;
      if (e < 0) break;
      x = e == blen - 1 ? r[i] : fnms(r[i], c[i], x);
      if (Y) Y[e] = x;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        if (q < m) {
          sx[q] += vv[i][q] * x.x;
          sy[q] += vv[i][q] * x.y;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    if (q < m) gp[q] = make_double2(sx[q], sy[q]);
}

// Dots of the stored solution with the first min(m, NQ) vectors of V.
template <int NQ>
__device__ __forceinline__ void sys_dots(const cpx<double> *Y, int blen, const double *__restrict__ V, int64_t ldv, int m,
                                         double2 *gp) {
  constexpr int U = kSysRows;
  double sx[NQ], sy[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) sx[q] = sy[q] = 0.0;
  cpx<double> nx[U];
  auto load = [&](int e0) {
#pragma unroll
    for (int i = 0; i < U; ++i) nx[i] = e0 + i < blen ? Y[e0 + i] : mk<double>(0.0, 0.0);
  };
  load(0);
  for (int e0 = 0; e0 < blen; e0 += U) {
    cpx<double> x[U];
    double vv[U][NQ];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      x[i] = nx[i];
#pragma unroll
      for (int q = 0; q < NQ; ++q) vv[i][q] = q < m && e0 + i < blen ? V[(int64_t)q * ldv + e0 + i] : 0.0;
    }
    load(e0 + U);
#pragma unroll
    for (int i = 0; i < U; ++i) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        if (q < m) {
          sx[q] += vv[i][q] * x[i].x;
          sy[q] += vv[i][q] * x[i].y;
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    if (q < m) gp[q] = make_double2(sx[q], sy[q]);
}

__global__ void __launch_bounds__(kSysThreads) k_pint_sys(PintGeom g, PintArgs<double> a, const cpx<double> *__restrict__ rd,
                                                          const cpx<double> *__restrict__ cc, cpx<double> *scr,
                                                          int64_t ld) {
  grid_dep_wait();
  if (a.skip_flag && *a.skip_flag) return;
  if (a.skip_flag2 && *a.skip_flag2) return;
  constexpr int U = kSysRows;
  const int64_t s = (int64_t)blockIdx.x * kSysThreads + threadIdx.x;
  if (s >= (int64_t)g.nf * g.nblk) return;
  const int blk = (int)(s / g.nf), k = (int)(s - (int64_t)blk * g.nf), blen = g.blen;
  const int64_t off = (int64_t)blk * blen;
  const double *rv = a.rvec;
  int m = a.V ? a.mdots : 0;
  if (a.mcount) {
    const int mc = *a.mcount + 1;  // v_m of the step in progress
    rv = a.V + (int64_t)mc * a.ldv;
    m = a.want_dots ? mc : 0;
  }
  double sub = -1.0;  // with R: r = R_k - |sub| rv
  if (a.xm_count) {
    rv = a.xm_out;
    sub = -a.xm_scale;
    m = 0;
  }
  if (rv) rv += off;
  const cpx<double> *R = a.R ? a.R + (int64_t)k * a.ldr + off : nullptr;
  const double *lo = a.tlo + off;
  rd += s;
  cc += s;
  scr += s;
  // forward: y_e = (r_e - lo_e y_{e-1}) / pivot_e
  {
    cpx<double> nr[U], nb[U];
    double nl[U], nv[U];
    auto load = [&](int e0) {
#pragma unroll
      for (int i = 0; i < U; ++i) {
        nb[i] = mk<double>(0.0, 0.0);
        nv[i] = 0.0;
        if (e0 + i < blen) {
          nr[i] = rd[(int64_t)(e0 + i) * ld];
          nl[i] = lo[e0 + i];
          if (R) nb[i] = R[e0 + i];
          if (rv) nv[i] = rv[e0 + i];
        }
      }
    };
    cpx<double> y = mk<double>(0.0, 0.0);
    load(0);
    for (int e0 = 0; e0 < blen; e0 += U) {
      cpx<double> r[U], b[U];
      double l[U], v[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        r[i] = nr[i];
        b[i] = nb[i];
        l[i] = nl[i];
        v[i] = nv[i];
      }
      load(e0 + U);
#pragma unroll
      for (int i = 0; i < U; ++i) {
        if (e0 + i >= blen) break;
        cpx<double> t = b[i];
        if (!R)
          t.x = v[i];
        else if (rv)
          t.x = fma(sub, v[i], t.x);
        if (e0 + i > 0) t = fnms_r(t, l[i], y);
        y = mul(t, r[i]);
        scr[(int64_t)(e0 + i) * ld] = y;
      }
    }
  }
  cpx<double> *Y = a.Y ? a.Y + (int64_t)k * a.ldy + off : nullptr;
  const double *V = a.V ? a.V + off : nullptr;
  double2 *gp = a.gpart ? a.gpart + ((int64_t)k * g.nblk + blk) * m : nullptr;
  if (m == 0)
    sys_backward<0>(cc, scr, ld, Y, blen, V, a.ldv, 0, gp);
  else if (m <= 2)
    sys_backward<2>(cc, scr, ld, Y, blen, V, a.ldv, m, gp);
  else if (m <= 4)
    sys_backward<4>(cc, scr, ld, Y, blen, V, a.ldv, m, gp);
  else if (m <= 8)
    sys_backward<8>(cc, scr, ld, Y, blen, V, a.ldv, m, gp);
  else
    sys_backward<kSysDots>(cc, scr, ld, Y, blen, V, a.ldv, m, gp);
  for (int q0 = kSysDots; q0 < m; q0 += kSysDots)
    sys_dots<kSysDots>(Y, blen, V + (int64_t)q0 * a.ldv, a.ldv, m - q0, gp + q0);
}

// a.fac_out: the factor pass; otherwise a loop on a.fac_in with a.scratch (pint_sys_scratch values).
// a.omega is left to the caller's column sum over Y; dots of more than kSysDots vectors need Y.
void launch_pint_sys(Ctx &c, const PintGeom &g, const PintArgs<double> &a) {
  const int64_t ld = sys_ld(g), n = ld * g.blen;
  const dim3 grid((unsigned)(((int64_t)g.nf * g.nblk + kSysThreads - 1) / kSysThreads));
  if (a.fac_out) {
    c.launch("pint_factor_f64", (double)n * 32.0, [&] {
      pdl_launch(c.pdl, k_sys_factor, grid, dim3(kSysThreads), 0, c.stream, g, a, a.fac_out, a.fac_out + n, ld);
    });
    return;
  }
  if (a.xm_count)
    c.launch("pint_store_f64", (double)g.nblk * g.blen * 8.0, [&] {
      pdl_launch(c.pdl, k_sys_xm, dim3((unsigned)(((int64_t)g.nblk * g.blen + 255) / 256)), dim3(256), 0, c.stream, g, a);
    });
  const bool dots = a.mcount ? a.want_dots != 0 : a.mdots > 0;
  // factors read, the forward sweep's result written and read, spectra as requested
  const double bytes = (double)n * 16.0 * (4 + (a.R ? 1 : 0) + (a.Y ? 1 : 0));
  c.launch(dots ? "pint_dots_f64" : (a.omega ? "pint_acc_f64" : "pint_store_f64"), bytes, [&] {
    pdl_launch(c.pdl, k_pint_sys, grid, dim3(kSysThreads), 0, c.stream, g, a, a.fac_in, a.fac_in + n, a.scratch, ld);
  });
}

}  // namespace pd
