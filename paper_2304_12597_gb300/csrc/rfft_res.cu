// Binary32, forward, of the 1D FP64 residual: the time DFT in registers (rfft.cuh) of
// r_j = G_j + u_{j-1} - (I + tau K) u_j, formed while the tile is loaded.
//
// Bound by GB300's FP64 pipe (four operations per unknown: 8 us per million), with HBM well below it
// (20 bytes per unknown, 3 us per million).  The residual needs four loads per value, so it does not
// suit pass 1, where a thread owns R1 rows and few threads run: all threads form it first, kRows
// consecutive rows of one column at a time (u_{j-1} carries over), and leave it in shared memory as
// binary32, inside the space of the exchange: residue r's R1 real values per column lie in the
// block that pass 1's R1/2 + 1 complex values of the same residue then overwrite, and the threads
// of one residue are lanes of one warp.
//
// Measured per launch (one GB300, the shared-memory passes of fft.cu -> here):
//    4095 columns of 2048  134 -> 97.5 us (FP64 floor 67: 512 tiles on 152 SMs leave a ragged last
//                          wave; four columns a tile and 160 to 256 threads: 102 to 125 us)
//   32736 columns of 1024  376 -> 300 us (floor 267)
//    1023 columns of 1024  26.6 -> 22.7 us
// Leaving out the addition of a zero G (three operations for a homogeneous equation) measured 98 -> 83
// us there, but 0.5 to 4 % more per launch wherever G is not zero: left out.
#include "rfft.cuh"

namespace pd {

// (four where the wide tile's register budget is 72)
template <typename T, int R1, int R2, int TX>
constexpr int res_rows() { return R2 < 8 || (R2 < 32 && TX == wide_tx<T, R1, R2>()) ? 4 : 8; }
// Narrow tiles (few columns): 160 threads for the residual, of which the passes use what they need
// (1023 columns of 1024 points: 22.7 us; 23.6 us with 256 threads).
template <typename T, int R1, int R2, int TX>
constexpr int res_threads() {
  constexpr int t = rfft_threads<R1, R2, TX>();
  return t < 160 && TX < wide_tx<T, R1, R2>() && R1 * R2 >= 256 ? 160 : t;
}
template <typename T, int R1, int R2, int TX>
constexpr int res_ctas() {
  return TX < wide_tx<T, R1, R2>() ? 3 : rfft_ctas<T, R1, R2, TX>();
}

template <typename T, int R1, int R2, int TX, bool SLOT>
__global__ void __launch_bounds__(res_threads<T, R1, R2, TX>(), res_ctas<T, R1, R2, TX>())
    k_rfft_res(const double *__restrict__ G, const double *__restrict__ U, int64_t ncols,
               const double *__restrict__ rxl, const double *__restrict__ rxd, const double *__restrict__ rxu,
               const cpx<T> *__restrict__ tw, cpx<T> *__restrict__ S, int64_t lds, const T *__restrict__ rs,
               const int *__restrict__ mex, int mnx, RhsNorm rn, SlotScale sc) {
  grid_dep_wait();
  constexpr int n = R1 * R2, H = R1 / 2 + 1, NIT = res_threads<T, R1, R2, TX>() / TX, RB = res_rows<T, R1, R2, TX>();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cl = (int)threadIdx.x % TX, it0 = (int)threadIdx.x / TX;
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw) + cl;  // (r, k1) at (r H + k1) TX
  T *xs = reinterpret_cast<T *>(smraw) + cl;            // (r, i) at (2 H r + i) TX
  const int64_t col = (int64_t)blockIdx.x * TX + cl;
  const bool live = col < ncols;
  if constexpr (SLOT) G = global_ptr(sc.G);
  const double ncl = live && col > 0 ? -rxl[col] : 0.0;
  const double ncd = live ? -rxd[col] : 0.0;
  const double ncu = live && col + 1 < ncols ? -rxu[col] : 0.0;
  const int64_t ol = col > 0 ? -1 : 0, ou = col + 1 < ncols ? 1 : 0;  // in-range neighbour offsets
  const int ex = SLOT && live ? mex[col / mnx] + sc.ex[col / mnx] : 0;
  float ss = 0.0f;  // squares of the residual (rn)
  // piece q: rows j0 .. j0 + RB - 1, j0 = R2 i + RB rc; the pieces side by side in a warp differ in i,
  // so that their stores hit consecutive banks
  for (int q = it0; q < n / RB; q += NIT) {
    const int i = q % R1, r0 = RB * (q / R1), j0 = R2 * i + r0;
    const int64_t o = (int64_t)j0 * ncols + col;
    double g[RB], uc[RB], ul[RB], ur[RB], um = 0.0;
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const double *u = U + o + (int64_t)k * ncols;
      g[k] = live ? G[o + (int64_t)k * ncols] : 0.0;
      uc[k] = live ? u[0] : 0.0;
      ul[k] = live ? u[ol] : 0.0;
      ur[k] = live ? u[ou] : 0.0;
    }
    if (live && j0 > 0) um = U[o - ncols];
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const double res = fma(ncu, ur[k], fma(ncl, ul[k], fma(ncd, uc[k], g[k] + um)));
      um = uc[k];
      const T v = SLOT ? slot_load<T>(res, ex) : cvt<T>(res);
      const float f = cvt<float>(v);
      ss = fmaf(f, f, ss);
      xs[(2 * H * (r0 + k) + i) * TX] = v;
    }
  }
  __syncthreads();
  const unsigned group = TX == 32 ? 0xffffffffu : ((1u << (TX & 31)) - 1u) << ((int)(threadIdx.x & 31) / TX * TX);
  for (int r = it0; r < R2; r += NIT) {
    T x[R1];
#pragma unroll
    for (int i = 0; i < R1; ++i) x[i] = xs[(2 * H * r + i) * TX];
    __syncwarp(group);  // the residue's other columns have read their values
    if (rs) {
#pragma unroll
      for (int i = 0; i < R1; ++i) x[i] *= rs[r + R2 * i];
    }
    cpx<T> z[H];
    rdft<T, R1, 1, 0, R1>(x, z);
    cpx<T> *o = sm + r * H * TX;
    o[0] = z[0];
#pragma unroll
    for (int k = 1; k < H - 1; ++k) o[k * TX] = mul(tw[r * k], z[k]);
    o[(H - 1) * TX] = scal(z[H - 1].x, tw[r * (H - 1)]);
  }
  __syncthreads();
  for (int k1 = it0; k1 < H; k1 += NIT) rfft_pass2<T, R1, R2, TX>(sm, S, lds, col, live, k1);
  if (rn.part) rhs_norm_finish(ss, rn);
}

template <>
void rfft_res_launch<float>(Ctx &c, const double *G, const double *U, int64_t ncols, int n, const double *rxl,
                            const double *rxd, const double *rxu, const cpx<float> *tw, cpx<float> *S, int64_t lds,
                            const float *rs, const int *mex, int mnx, const RhsNorm &rn, const SlotScale &sc,
                            const char *fam, double bytes) {
  using T = float;
  c.launch(fam, bytes, [&] {
    rfft_tile<T>(n, ncols, [&](auto r1, auto r2, auto tx) {
      constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value, TX = decltype(tx)::value;
      const size_t smem = (size_t)R2 * (R1 / 2 + 1) * TX * sizeof(cpx<T>);
      auto kern = sc.ex ? k_rfft_res<T, R1, R2, TX, true> : k_rfft_res<T, R1, R2, TX, false>;
      if (smem > 48 * 1024) allow_dyn_smem((const void *)kern);
      pdl_launch(c.pdl, kern, dim3((unsigned)((ncols + TX - 1) / TX)), dim3(res_threads<T, R1, R2, TX>()), smem, c.stream,
                 G, U, ncols, rxl, rxd, rxu, tw, S, lds, rs, mex, mnx, rn, sc);
    });
  });
}

}  // namespace pd
