// The orthonormal DST-I along y (Sec. 6.1: it diagonalises T_y) for n_y + 1 = 64, 128 and 256:
// two passes in registers over half of the odd extension.
//
// Two columns a, b are one complex series z = a + i b of n_y values, whose DST is, but for a
// factor, the DFT of its odd extension of length N2 = 2 (n_y + 1) = R1 R2.  With z[N2 - j] =
// -z[j], the R1-point DFTs Y_r of the residues r mod R2 satisfy, with the twiddles applied,
//   T_r[k1] = w^{r k1} Y_r[k1],   T_{R2-r}[k1] = -T_r[-k1],   w = exp(-2 pi i / N2),
// so pass 1 needs r = 0 .. R2/2 only and touches every sample once, and since Z[N2 - k] = -Z[k],
// pass 2 (the R2-point DFTs over r, Z[k1 + R1 k2]) needs k1 = 0 .. R1/2 only.
//
// A CTA takes 64 columns: lane l of every warp owns columns l and l + 32 of the CTA's (of all
// (slab, x) columns in a row, so that no tile is cut off at n_x), a warp takes one r, then one
// k1.  Loads and stores run along x, the twiddles are uniform over a warp, and the exchange
// between the passes is free of bank conflicts.  Against k_dst_y (fft.cu: the full odd extension
// in shared memory, every sample read twice) this is under half the arithmetic and a fifth of
// the instructions.  Measured per launch (one GB300, k_dst_y -> k_dst2):
//   255 x 255 x 256  binary32 136 -> 68 us (mean of store and +=), binary64 1120 -> 559 us
//   127 x 127 x 512  binary32  78 -> 37 us,                        binary64  506 -> 263 us
//    63 x 63 x 512   binary32  29 -> 12 us,                        binary64  119 ->  70 us
// The binary32 transforms move 200 to 333 MB at 255 x 255 x 256 (30 to 49 us of copy bandwidth); the
// binary64 ones are bound by GB300's FP64 pipe.  With the residual on load, six FP64
// operations per element bound both (33 us each at 255 x 255 x 256): binary32 261 -> 255 us,
// binary64 1296 -> 864 us; a residual kernel of its own (231 us) beside the plain transform
// (59 us) measured slower, since here the DST's passes of one CTA run beside the FP64 work of
// the other.
#include <algorithm>

#include "pd_fft.cuh"
#include "pd_internal.h"

namespace pd {

namespace {

struct Col {  // one column of a lane
  int64_t base;  // its first element (row 0) in the (slab, y, x) array
  bool in;
  int ein, eout;  // batches: the problem's exact scaling, on binary64 input and off binary64 output
  bool dead;      // the output of an all-zero problem: exact zeros
  // residual input: problem b, x, whether its slab is the first time, the x-coefficients
  int b, x;
  bool t0;
  double cl, cu;
};

}  // namespace

// MODE 0: Y = DST X; 1: Y += DST X.  RES: the input is the FP64 residual of ResIn instead of X.
template <typename Tin, typename Tout, typename T, int R1, int R2, int NW, int MINB, int MODE, bool RES, bool SLOT>
__global__ void __launch_bounds__(NW * 32, MINB)
    k_dst2(const Tin *__restrict__ X, Tout *__restrict__ Y, int64_t ncol, int64_t nx, const cpx<T> *__restrict__ tw,
           T scale, const int *skip, ResIn rin, SlotScale sc) {
  grid_dep_wait();
  if (skip && *skip) return;  // U already holds the result (Algorithm 3's U_1 exit)
  constexpr int N = R1 * R2 / 2, NY = N - 1, S = R1 + 1;
  extern __shared__ __align__(16) unsigned char smraw[];
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw);  // T_r[k1] at ((r S + k1) 32 + lane), T_r[-k1] at k1 -> R1 - k1, T_r[-R1/2] at R1
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if constexpr (SLOT) {
    if constexpr (RES) {
      rin.G = global_ptr(sc.G);
    } else if constexpr (sizeof(Tin) == 8) {
      if (sc.G) X = global_ptr(sc.G);
    }
  }
  Col c[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t g = (int64_t)blockIdx.x * 64 + 32 * h + lane;
    c[h].in = g < ncol;
    const int64_t slab = c[h].in ? g / nx : 0;
    const int x = c[h].in ? (int)(g - slab * nx) : 0;
    c[h].base = slab * (NY * nx) + x;
    c[h].ein = c[h].eout = 0;
    c[h].dead = false;
    if constexpr (SLOT) {  // (with sc.G: a transform of the caller's G or of the residual; else one into U)
      const int b = (int)(slab % sc.batch);
      if (sc.G)
        c[h].ein = sc.ex[b];
      else
        c[h].eout = -sc.ex[b], c[h].dead = sc.zero[b] != 0;
    }
    if constexpr (RES) {
      // slabs are (time, problem) with the problems of a time row adjacent, as the rows of the
      // stacked grid are: G and U take the slab's own element index
      const int64_t tt = slab / rin.batch;
      c[h].b = (int)(slab - tt * rin.batch);
      c[h].x = x;
      c[h].t0 = tt == 0;
      const int64_t cx = (int64_t)c[h].b * nx + x;
      c[h].cl = x > 0 ? rin.rxl[cx] : 0.0;
      c[h].cu = x + 1 < nx ? rin.rxu[cx] : 0.0;
    }
  }
  // the residual r = G_t + u_{t-1} - [(I + tau T_x) u_t + tau T_y u_t] at rows y0, y0 + dy, ...: one
  // FP64 add and five FMAs, every element formed once
  const int64_t nb = RES ? (int64_t)rin.ny * nx : 0;
  constexpr int RB = 4;  // elements whose loads are in flight together
  auto residuals = [&](const Col &q, int y0, int dy, T (&v)[RB]) {
    double g[RB], um[RB], uc[RB], ul[RB], ur[RB], ud[RB], uu[RB], dd[RB];
#pragma unroll
    for (int u = 0; u < RB; ++u) {
      const int y = y0 + u * dy;
      const double *p = rin.U + q.base + (int64_t)y * nx;
      const int64_t j = (int64_t)(q.b * rin.nym + y) * nx + q.x;
      g[u] = q.in ? rin.G[q.base + (int64_t)y * nx] : 0.0;
      um[u] = q.in && !q.t0 ? p[-nb] : 0.0;
      uc[u] = q.in ? p[0] : 0.0;
      ul[u] = q.in && q.x > 0 ? p[-1] : 0.0;
      ur[u] = q.in && q.x + 1 < nx ? p[1] : 0.0;
      ud[u] = q.in && y > 0 ? p[-nx] : 0.0;
      uu[u] = q.in && y + 1 < NY ? p[nx] : 0.0;
      dd[u] = q.in ? rin.rdd[j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < RB; ++u) {
      const int iy = q.b * rin.nym + y0 + u * dy;
      double r = g[u] + um[u];
      r = fma(-dd[u], uc[u], r);
      r = fma(-q.cl, ul[u], r);
      r = fma(-q.cu, ur[u], r);
      r = fma(-rin.ryl[iy], ud[u], r);
      r = fma(-rin.ryu[iy], uu[u], r);
      if constexpr (SLOT)
        v[u] = slot_load<T>(r, q.ein + rin.mex[q.b]);
      else
        v[u] = cvt<T>(r);
    }
  };

  // pass 1
  for (int r = warp; r <= R2 / 2; r += NW) {
    cpx<T> z[R1];
    // samples r + R2 i: row r + R2 i - 1 below N, minus row N2 - (r + R2 i) - 1 above (none at 0, N)
    if constexpr (RES) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i0 = 0; i0 < R1; i0 += RB) {
          const bool upper = i0 >= R1 / 2;
          if (upper && (r == 0 || r == R2 / 2)) continue;  // mirrored below
          // rows in steps of R2, up or down; r = 0 starts at sample 0, which is zero
          T v[RB];
          const int y0 = upper ? R2 * (R1 - i0) - r - 1 : r + R2 * i0 - 1;
          residuals(c[h], y0 < 0 ? R2 - 1 : y0, upper ? -R2 : R2, v);
          if (y0 < 0) {  // (rows R2 - 1, 2 R2 - 1, ...): shift by one sample
#pragma unroll
            for (int u = RB - 1; u > 0; --u) v[u] = v[u - 1];
            v[0] = T(0);
          }
#pragma unroll
          for (int u = 0; u < RB; ++u) {
            if (h == 0)
              z[i0 + u].x = upper ? -v[u] : v[u];
            else
              z[i0 + u].y = upper ? -v[u] : v[u];
          }
        }
      if (r == 0) {
#pragma unroll
        for (int i = R1 / 2 + 1; i < R1; ++i) z[i] = mk<T>(-z[R1 - i].x, -z[R1 - i].y);
        z[R1 / 2] = mk<T>(T(0), T(0));
      } else if (r == R2 / 2) {
#pragma unroll
        for (int i = R1 / 2; i < R1; ++i) z[i] = mk<T>(-z[R1 - 1 - i].x, -z[R1 - 1 - i].y);
      }
    } else {
      Tin va[R1], vb[R1];
#pragma unroll
      for (int i = 0; i < R1; ++i) {
        const int y = i < R1 / 2 ? r + R2 * i - 1 : R2 * (R1 - i) - r - 1;
        const bool have = y >= 0 && y < NY;
        va[i] = have && c[0].in ? X[c[0].base + (int64_t)y * nx] : Tin(0);
        vb[i] = have && c[1].in ? X[c[1].base + (int64_t)y * nx] : Tin(0);
      }
#pragma unroll
      for (int i = 0; i < R1; ++i) {
        T a, b;
        if constexpr (SLOT && sizeof(Tin) == 8) {
          a = slot_load<T>(va[i], c[0].ein);
          b = slot_load<T>(vb[i], c[1].ein);
        } else {
          a = cvt<T>(va[i]);
          b = cvt<T>(vb[i]);
        }
        z[i] = i < R1 / 2 ? mk<T>(a, b) : mk<T>(-a, -b);
      }
    }
    dft_reg<T, R1>(z);
    cpx<T> *o = sm + (size_t)r * S * 32 + lane;
    o[0] = z[0];
    o[R1 * 32] = mul(conjg(tw[r * (R1 / 2)]), z[R1 / 2]);
#pragma unroll
    for (int k = 1; k < R1; ++k) {
      const int m = k <= R1 / 2 ? k : R1 - k;
      const cpx<T> w = tw[r * m];
      o[k * 32] = mul(k <= R1 / 2 ? w : conjg(w), z[k]);
    }
  }
  __syncthreads();

  // pass 2
  for (int k1 = warp; k1 <= R1 / 2; k1 += NW) {
    cpx<T> z[R2];
    const cpx<T> *p = sm + k1 * 32 + lane;
    const cpx<T> *m = sm + (k1 == 0 ? 0 : k1 == R1 / 2 ? R1 : R1 - k1) * 32 + lane;
#pragma unroll
    for (int r = 0; r < R2; ++r) {
      if (r <= R2 / 2) {
        z[r] = p[r * S * 32];
      } else {
        const cpx<T> v = m[(R2 - r) * S * 32];
        z[r] = mk<T>(-v.x, -v.y);
      }
    }
    dft_reg<T, R2>(z);
    const T sa = T(-0.5) * scale, sb = T(0.5) * scale;
    constexpr int EB = R2 / 2 < 8 ? R2 / 2 : 8;  // outputs whose old values are loaded together (MODE 1)
#pragma unroll
    for (int q0 = 0; q0 < R2; q0 += EB) {
      Tout oa[EB], ob[EB];
      // k = k1 + R1 k2 stands for row k - 1, above N for row N2 - k - 1 with the sign changed; the
      // series k1 = 0 and R1/2 hold their own mirror images
      const bool upper = q0 >= R2 / 2;
      if (upper && (k1 == 0 || k1 == R1 / 2)) continue;
#pragma unroll
      for (int u = 0; u < EB; ++u) {
        const int k = k1 + R1 * (q0 + u);
        const int row = upper ? 2 * N - k - 1 : k - 1;
        oa[u] = MODE == 1 && row >= 0 && c[0].in ? Y[c[0].base + (int64_t)row * nx] : Tout(0);
        ob[u] = MODE == 1 && row >= 0 && c[1].in ? Y[c[1].base + (int64_t)row * nx] : Tout(0);
      }
#pragma unroll
      for (int u = 0; u < EB; ++u) {
        const int k = k1 + R1 * (q0 + u);
        const int row = upper ? 2 * N - k - 1 : k - 1;
        const cpx<T> v = z[q0 + u];
        const T a = (upper ? -sa : sa) * v.y, b = (upper ? -sb : sb) * v.x;
        Tout da, db;
        if constexpr (SLOT && sizeof(Tout) == 8) {
          da = slot_store<true>(a, c[0].eout);
          db = slot_store<true>(b, c[1].eout);
        } else {
          da = cvt<Tout, true>(a);
          db = cvt<Tout, true>(b);
        }
        if (MODE == 1) {
          da = oa[u] + da;
          db = ob[u] + db;
        }
        if (row >= 0 && c[0].in) Y[c[0].base + (int64_t)row * nx] = SLOT && c[0].dead ? Tout(0) : da;
        if (row >= 0 && c[1].in) Y[c[1].base + (int64_t)row * nx] = SLOT && c[1].dead ? Tout(0) : db;
      }
    }
  }
}

// Whether k_dst2 is built for the length and the faster one.  With fewer than one CTA of 64
// columns per SM, k_dst_y's narrower tiles spread over more SMs.  The binary32 residual (bound by
// its FP64 work in either kernel) of length 127 measured 129 us here against 120 us there
// (127 x 127, n_t = 512; 255 x 255 x 256: 250 against 261, 63 x 63 x 512: 36 against 39).
bool dst2_fits(int64_t ny, int64_t ncol, bool res_f32) {
  return (ny == 63 || (ny == 127 && !res_f32) || ny == 255) && ncol >= (int64_t)64 * sm_count();
}

template <typename Tin, typename Tout, typename T, int R1, int R2, int NW, int MINB, bool RES>
static void launch_size(Ctx &c, const Tin *X, Tout *Y, int64_t ncol, int64_t ny, int64_t nx, const cpx<T> *tw, int mode,
                        const int *skip, const ResIn &rin, const SlotScale &sc, const char *fam, double bytes) {
  const size_t smem = (size_t)(R2 / 2 + 1) * (R1 + 1) * 32 * sizeof(cpx<T>);
  const T scale = (T)sqrt(2.0 / (double)(ny + 1));
  const unsigned grid = (unsigned)((ncol + 63) / 64);
  auto kern = k_dst2<Tin, Tout, T, R1, R2, NW, MINB, 0, RES, false>;
  if constexpr (!RES && sizeof(Tout) == 8) {
    if (mode) kern = k_dst2<Tin, Tout, T, R1, R2, NW, MINB, 1, RES, false>;
  }
  if constexpr (R1 * R2 < 512) {  // (batches of n_y = 255, n_x <= 32 stay with k_dst_y)
    if (sc.ex) {
      kern = k_dst2<Tin, Tout, T, R1, R2, NW, MINB, 0, RES, true>;
      if constexpr (!RES && sizeof(Tout) == 8) {
        if (mode) kern = k_dst2<Tin, Tout, T, R1, R2, NW, MINB, 1, RES, true>;
      }
    }
  }
  c.launch(fam, bytes, [&] {
    if (smem > 48 * 1024) allow_dyn_smem((const void *)kern);
    pdl_launch(c.pdl, kern, dim3(grid), dim3(NW * 32), smem, c.stream, X, Y, ncol, nx, tw, scale, skip, rin, sc);
  });
}

// Warps per CTA and CTAs per SM: nine warps take the nine pass-2 items of lengths 127 and 255
// (and the 9 or 17 of pass 1) in whole rounds, five those of length 63.  Measured against 5 and 7
// warps with 2 to 4 CTAs per SM: 255 59 us against 75 and 78, the others within 5 %.
template <typename Tin, typename Tout, typename T, bool RES>
void launch_dst2(Ctx &c, const Tin *X, Tout *Y, int64_t ncol, int64_t ny, int64_t nx, const cpx<T> *tw, int mode,
                 const int *skip, const ResIn &rin, const SlotScale &sc, const char *fam, double bytes) {
  constexpr int B = sizeof(T) == 8 ? 1 : 2;
  if (ny == 63)
    launch_size<Tin, Tout, T, 16, 8, 5, sizeof(T) == 8 ? 2 : 4, RES>(c, X, Y, ncol, ny, nx, tw, mode, skip, rin, sc, fam, bytes);
  else if (ny == 255)
    launch_size<Tin, Tout, T, 16, 32, 9, B, RES>(c, X, Y, ncol, ny, nx, tw, mode, skip, rin, sc, fam, bytes);
  else if constexpr (!(RES && sizeof(T) == 4))
    launch_size<Tin, Tout, T, 16, 16, 9, B, RES>(c, X, Y, ncol, ny, nx, tw, mode, skip, rin, sc, fam, bytes);
}

#define PD_DST2(TIN, TOUT, T, RES)                                                                                   \
  template void launch_dst2<TIN, TOUT, T, RES>(Ctx &, const TIN *, TOUT *, int64_t, int64_t, int64_t, const cpx<T> *, \
                                               int, const int *, const ResIn &, const SlotScale &, const char *, double);
PD_DST2(double, float, float, false)
PD_DST2(float, float, float, false)
PD_DST2(float, double, float, false)
PD_DST2(double, double, double, false)
PD_DST2(double, float, float, true)
PD_DST2(double, double, double, true)

}  // namespace pd
