// Time DFTs of n = R1 R2 = 32 .. 2048 points in two register passes (eq. 5: U F^T and Y F^{-T}).
//
// A thread owns one column and, in turn, one residue of the time index and one of the frequency:
//  forward  pass 1: the real R1-point DFT of the rows r + R2 i, twiddled by w_n^{r k1}, k1 = 0 .. R1/2;
//           pass 2: the complex R2-point DFT over r for one k1: the frequencies k1 + R1 k2, whose upper
//           half is the conjugate of rows n - k, so that k1 = 0 .. R1/2 is the half spectrum;
//  inverse  the same passes back to front: over k2 for one k1 (the upper half read as conjugates),
//           twiddles, then a Hermitian-to-real R1-point DFT for the rows r + R2 i.
// Real arithmetic takes the place of packing two columns into one complex series, and with it goes
// the separation pass.  One exchange through shared memory (n/2 complex values per column);
// a CTA's TX adjacent columns make every global access TX contiguous elements of a row.
//
// What bounds them: binary32, HBM and latency (about 35 thread instructions per unknown, against
// some 150 of the shared-memory passes in fft.cu); with the FP64 update on store, and in binary64,
// GB300's FP64 pipe (about 20 operations per unknown, against 25).  Measured per launch (one GB300,
// fft.cu -> here; forward / inverse):
//   65025 columns of  256, binary32   56 / 85 us -> 42 / 46 us,   binary64  614 / 669 us -> 435 / 480 us
//    4095 columns of 2048, binary32   74 / 88 us -> 42 / 53 us,   binary64  411 / 418 us -> 350 / 371 us
//   32736 columns of 1024, binary32  194 / 251 us -> 113 / 158 us
//     (forward with the norm of the input, in binary64 one FP64 operation per value: 23 of the 435 us)
//     300 columns of   32, binary32   14 / 15 us ->  8 / 12 us
// The forward transform of the 1D FP64 residual, binary32, is in rfft_res.cu.
#pragma once

#include <algorithm>

#include "pd_fft.cuh"
#include "pd_fft_tail.cuh"
#include "pd_internal.h"

namespace pd {

// Items of a CTA's TX columns that run side by side: a residue of the larger pass each.
template <int R1, int R2>
constexpr int rfft_items() { return R1 / 2 + 1 > 8 ? R1 / 2 + 1 : 8 < R2 ? 8 : R2; }
template <int R1, int R2, int TX>
constexpr int rfft_threads() { return (rfft_items<R1, R2>() * TX + 31) / 32 * 32; }
// Tiles.  Wide: as many columns as keep the exchange within about 75 KB (three CTAs per SM) and the
// CTA within 288 threads, at most 32 (one warp-wide row access).  Narrow: four columns (one 32-byte
// sector of doubles; eight for short n), taken when the wide tiles would not cover every SM twice.
template <typename T, int R1, int R2>
constexpr int wide_tx() {
  constexpr int per = R2 * (R1 / 2 + 1) * (int)sizeof(cpx<T>);
  constexpr int tx = per * 32 <= 75 * 1024 ? 32 : per * 16 <= 75 * 1024 ? 16 : per * 8 <= 75 * 1024 ? 8 : 4;
  return tx * rfft_items<R1, R2>() <= 288 ? tx : tx / 2;
}
template <typename T, int R1, int R2>
constexpr int narrow_tx() { return R1 * R2 >= 512 ? 4 : 8; }
// CTAs per SM that the register budget is set for.  Wide tiles: 72 registers a thread for passes of
// up to 16 complex values, 112 for 32 (binary64: 112 and 168); 256 points at two CTAs instead of
// three measured 50 us instead of 42.  Narrow tiles leave most SMs one or two CTAs anyway: 1023
// columns of 1024 points, inverse, 24.5 us with six CTAs' budget and its spills, 19.8 us without.
template <typename T, int R1, int R2, int TX>
constexpr int rfft_ctas() {
  constexpr int regs = R2 >= 32 || R1 >= 64 ? (sizeof(T) == 8 ? 168 : 112) : (sizeof(T) == 8 ? 112 : 72);
  constexpr int c = TX < wide_tx<T, R1, R2>() ? 2 : 65536 / (rfft_threads<R1, R2, TX>() * regs);
  return c < 1 ? 1 : c > 8 ? 8 : c;
}

// Forward, pass 2 for one k1: the frequencies k1 + R1 k2; past n/2 the conjugate of row n - k (rows 0
// and R1/2 mod R1 hold their own mirror images).
template <typename T, int R1, int R2, int TX>
__device__ __forceinline__ void rfft_pass2(const cpx<T> *sm, cpx<T> *__restrict__ S, int64_t lds, int64_t col, bool live,
                                           int k1) {
  constexpr int n = R1 * R2, H = R1 / 2 + 1;
  cpx<T> z[R2];
  const cpx<T> *p = sm + k1 * TX;
#pragma unroll
  for (int r = 0; r < R2; ++r) z[r] = p[r * H * TX];
  dft_reg<T, R2>(z);
#pragma unroll
  for (int k2 = 0; k2 < R2; ++k2) {
    const int k = k1 + R1 * k2;
    const bool up = 2 * k2 >= R2;
    if (up && (k1 == H - 1 || (k1 == 0 && 2 * k2 > R2))) continue;
    const bool mirror = up && k1 > 0;
    if (live) S[(int64_t)(mirror ? n - k : k) * lds + col] = mirror ? conjg(z[k2]) : z[k2];
  }
}

// Forward transform of X (n, ldx).
template <typename T, typename Tin, int R1, int R2, int TX, bool SLOT>
__global__ void __launch_bounds__(rfft_threads<R1, R2, TX>(), rfft_ctas<T, R1, R2, TX>())
    k_rfft(const Tin *__restrict__ X, int64_t ldx, int64_t ncols, const cpx<T> *__restrict__ tw, cpx<T> *__restrict__ S,
           int64_t lds, const T *__restrict__ rs, RhsNorm rn, SlotScale sc) {
  grid_dep_wait();
  constexpr int n = R1 * R2, H = R1 / 2 + 1, NIT = rfft_threads<R1, R2, TX>() / TX;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cl = (int)threadIdx.x % TX, it0 = (int)threadIdx.x / TX;
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw) + cl;  // (r, k1) at (r H + k1) TX
  const int64_t col = (int64_t)blockIdx.x * TX + cl;
  const bool live = col < ncols;
  T ss = T(0);  // squares of the input (rn: a reference scale)
  int ex = 0;
  if constexpr (SLOT) {
    X = global_ptr(sc.G);
    if (live) ex = sc.ex[col / sc.mnx];
  }
  for (int r = it0; r < R2; r += NIT) {
    T x[R1];
    constexpr int LB = R1 < 16 ? R1 : 16;  // rows whose loads are in flight together
#pragma unroll
    for (int i0 = 0; i0 < R1; i0 += LB) {
      Tin v[LB];
#pragma unroll
      for (int i = 0; i < LB; ++i) v[i] = live ? X[(int64_t)(r + R2 * (i0 + i)) * ldx + col] : Tin(0);
#pragma unroll
      for (int i = 0; i < LB; ++i) {
        if constexpr (SLOT)
          x[i0 + i] = slot_load<T>(v[i], ex);
        else
          x[i0 + i] = cvt<T>(v[i]);
      }
    }
    if (rn.part) {
#pragma unroll
      for (int i = 0; i < R1; ++i) ss += x[i] * x[i];
    }
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
  if (rn.part) rhs_norm_finish((float)ss, rn);
}

// Inverse: X[j] = Re((1/n) sum_k w_n^{-jk} Y[k]) with Y[n - k] = conj Y[k], times rsi[j] and, for
// batches, 2^-mex[col / mnx].  mode 0: store binary64, 1: add into binary64, 2: store binary32.
// Everything runs on conjugates: the result is real, so x_j = sum_k conj(Y[k]) w^{jk} / n.
template <typename T, int R1, int R2, int TX, int MODE, bool SLOT>
__global__ void __launch_bounds__(rfft_threads<R1, R2, TX>(), rfft_ctas<T, R1, R2, TX>())
    k_crfft(const cpx<T> *__restrict__ S, int64_t lds, int64_t ncols, const cpx<T> *__restrict__ tw,
            void *__restrict__ outv, int64_t ldo, double *__restrict__ norm_part, StepFinish fin,
            const T *__restrict__ rsi, double *__restrict__ colsum, const int *__restrict__ mex, int mnx,
            const int *skip, SlotScale sc) {
  grid_dep_wait();
  if (skip && *skip) return;  // U already holds the result (Algorithm 3's U_1 exit)
  constexpr int n = R1 * R2, H = R1 / 2 + 1, NT = rfft_threads<R1, R2, TX>(), NIT = NT / TX;
  using Tout = std::conditional_t<MODE == 2, float, double>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int cl = (int)threadIdx.x % TX, it0 = (int)threadIdx.x / TX;
  cpx<T> *sm = reinterpret_cast<cpx<T> *>(smraw) + cl;  // (r, k1) at (r H + k1) TX
  const int64_t x0 = (int64_t)blockIdx.x * TX, col = x0 + cl;
  const bool live = col < ncols;
  for (int k1 = it0; k1 < H; k1 += NIT) {
    cpx<T> z[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const int k = k1 + R1 * k2;
      const bool mirror = 2 * k > n;
      z[k2] = live ? S[(int64_t)(mirror ? n - k : k) * lds + col] : mk<T>(T(0), T(0));
    }
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const bool mirror = 2 * (k1 + R1 * k2) > n;
      z[k2].y = mirror ? z[k2].y : -z[k2].y;
    }
    dft_reg<T, R2>(z);
    cpx<T> *o = sm + k1 * TX;
    o[0] = z[0];
#pragma unroll
    for (int r = 1; r < R2; ++r) o[r * H * TX] = mul(tw[r * k1], z[r]);
  }
  __syncthreads();
  T inv_n = T(1) / T(n);
  if (mex && live) inv_n = (T)ldexp((double)inv_n, -mex[col / mnx]);
  Tout *out = reinterpret_cast<Tout *>(outv) + col;
  // batches: the store undoes the problem's scaling; columns that hold no unknown get exact zeros
  int ex = 0;
  bool dead = false;
  if (SLOT && live) {
    const int b = (int)(col / sc.mnx);
    ex = -sc.ex[b];
    dead = sc.zero[b] || col - (int64_t)b * sc.mnx >= sc.nxb[b];
  }
  // a few dozen squares per thread, in four sums of at most 16, so that binary32 overflows no earlier than
  // with the 2 to 32 values per thread of fft.cu; the stop rule needs a few digits
  float ss[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  for (int r = it0; r < R2; r += NIT) {
    cpx<T> z[H];
    const cpx<T> *p = sm + r * H * TX;
#pragma unroll
    for (int k = 0; k < H; ++k) z[k] = p[k * TX];
    T x[R1];
    hdft<T, R1, 1, 0, R1>(z, x);
    constexpr int EB = 8;  // rows whose old values are loaded together (mode 1)
#pragma unroll
    for (int i0 = 0; i0 < R1; i0 += EB) {
      Tout old[EB];
      if constexpr (MODE == 1) {
#pragma unroll
        for (int i = 0; i < EB; ++i) old[i] = live ? out[(int64_t)(r + R2 * (i0 + i)) * ldo] : Tout(0);
      }
#pragma unroll
      for (int i = 0; i < EB; ++i) {
        const int j = r + R2 * (i0 + i);
        const T v = x[i0 + i] * (rsi ? inv_n * rsi[j] : inv_n);
        if (live) {
          Tout d;
          if constexpr (SLOT)
            d = slot_store(v, ex);
          else
            d = cvt<Tout>(v);
          if constexpr (MODE == 1) d = old[i] + d;
          out[(int64_t)j * ldo] = SLOT && dead ? Tout(0) : d;
        }
        float vf;
        if constexpr (sizeof(T) == 8)
          vf = f64_to_f32_near(v);
        else
          vf = v;
        ss[i % 4] = fmaf(vf, vf, ss[i % 4]);
      }
    }
  }
  const float q = fmaf(0.25f, ss[0], 0.25f * ss[1]) + fmaf(0.25f, ss[2], 0.25f * ss[3]);
  c2r_finish<TX, NT>(live ? f32_to_f64_bits(q, 2) : 0.0, x0, ncols, colsum, norm_part, fin);
}

// ---- dispatch -------------------------------------------------------------------------------
template <typename F>
bool rfft_size(int n, F &&f) {
  switch (n) {
    case 32: f(std::integral_constant<int, 8>{}, std::integral_constant<int, 4>{}); return true;
    case 64: f(std::integral_constant<int, 8>{}, std::integral_constant<int, 8>{}); return true;
    case 128: f(std::integral_constant<int, 16>{}, std::integral_constant<int, 8>{}); return true;
    case 256: f(std::integral_constant<int, 16>{}, std::integral_constant<int, 16>{}); return true;
    case 512: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 16>{}); return true;
    case 1024: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 32>{}); return true;
    case 2048: f(std::integral_constant<int, 64>{}, std::integral_constant<int, 32>{}); return true;
    default: return false;
  }
}
// f(R1, R2, TX) for the tile of ncols columns
// (binary64 transforms of few columns stay in fft.cu, see rfft_built)
template <typename T, typename F>
void rfft_tile(int n, int64_t ncols, F &&f) {
  rfft_size(n, [&](auto r1, auto r2) {
    constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value;
    constexpr int W = wide_tx<T, R1, R2>(), NA = narrow_tx<T, R1, R2>() < W ? narrow_tx<T, R1, R2>() : W;
    if (W == NA || (ncols + W - 1) / W >= 2 * (int64_t)sm_count())
      f(r1, r2, std::integral_constant<int, W>{});
    else
      f(r1, r2, std::integral_constant<int, NA>{});
  });
}

template <typename T, typename Tin>
void rfft_launch(Ctx &c, const Tin *X, int64_t ldx, int64_t ncols, int n, const cpx<T> *tw, cpx<T> *S, int64_t lds,
                 const T *rs, const RhsNorm &rn, const SlotScale &sc, const char *fam, double bytes) {
  c.launch(fam, bytes, [&] {
    rfft_tile<T>(n, ncols, [&](auto r1, auto r2, auto tx) {
      constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value, TX = decltype(tx)::value;
      const size_t smem = (size_t)R2 * (R1 / 2 + 1) * TX * sizeof(cpx<T>);
      auto kern = k_rfft<T, Tin, R1, R2, TX, false>;
      if constexpr (sizeof(Tin) == 8) {
        if (sc.ex) kern = k_rfft<T, Tin, R1, R2, TX, true>;
      }
      if (smem > 48 * 1024) allow_dyn_smem((const void *)kern);
      pdl_launch(c.pdl, kern, dim3((unsigned)((ncols + TX - 1) / TX)), dim3(rfft_threads<R1, R2, TX>()), smem, c.stream,
                 X, ldx, ncols, tw, S, lds, rs, rn, sc);
    });
  });
}

template <typename T>
void crfft_launch(Ctx &c, const cpx<T> *S, int64_t lds, int64_t ncols, int n, const cpx<T> *tw, void *out, int64_t ldo,
                  int mode, double *norm_part, int *nparts, const StepFinish &fin, const T *rsi, double *colsum,
                  const int *mex, int mnx, const int *skip, const SlotScale &sc, const char *fam, double bytes) {
  c.launch(fam, bytes, [&] {
    rfft_tile<T>(n, ncols, [&](auto r1, auto r2, auto tx) {
      constexpr int R1 = decltype(r1)::value, R2 = decltype(r2)::value, TX = decltype(tx)::value;
      const size_t smem = (size_t)R2 * (R1 / 2 + 1) * TX * sizeof(cpx<T>);
      auto kern = sc.ex ? (mode == 1 ? k_crfft<T, R1, R2, TX, 1, true> : k_crfft<T, R1, R2, TX, 0, true>)
                        : (mode == 1 ? k_crfft<T, R1, R2, TX, 1, false> : k_crfft<T, R1, R2, TX, 0, false>);
      if constexpr (sizeof(T) == 4) {
        if (mode == 2) kern = k_crfft<T, R1, R2, TX, 2, false>;
      }
      if (smem > 48 * 1024) allow_dyn_smem((const void *)kern);
      const unsigned grid = (unsigned)((ncols + TX - 1) / TX);
      if (nparts) *nparts = (int)grid;
      pdl_launch(c.pdl, kern, dim3(grid), dim3(rfft_threads<R1, R2, TX>()), smem, c.stream, S, lds, ncols, tw, out, ldo,
                 norm_part, fin, rsi, colsum, mex, mnx, skip, sc);
    });
  });
}

}  // namespace pd
