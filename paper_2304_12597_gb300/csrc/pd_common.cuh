// Shared device helpers for the ParaDiag kernels (complex arithmetic, team
// barriers, warp reductions).  Internal header; not part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pd {

// Interleaved complex number of real type T (layout-compatible with float2 /
// double2 and with numpy complex64 / complex128).
template <typename T>
struct alignas(2 * sizeof(T)) cpx {
  T x, y;
};

template <typename T>
__host__ __device__ __forceinline__ cpx<T> mk(T a, T b) {
  cpx<T> r;
  r.x = a;
  r.y = b;
  return r;
}
template <typename T>
__device__ __forceinline__ cpx<T> add(cpx<T> a, cpx<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ cpx<T> sub(cpx<T> a, cpx<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <typename T>
__device__ __forceinline__ cpx<T> mul(cpx<T> a, cpx<T> b) {
  return mk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T>
__device__ __forceinline__ cpx<T> scal(T s, cpx<T> a) { return mk<T>(s * a.x, s * a.y); }
template <typename T>
__device__ __forceinline__ cpx<T> conjg(cpx<T> a) { return mk<T>(a.x, -a.y); }
// a - b * c
template <typename T>
__device__ __forceinline__ cpx<T> fnms(cpx<T> a, cpx<T> b, cpx<T> c) {
  return mk<T>(a.x - b.x * c.x + b.y * c.y, a.y - b.x * c.y - b.y * c.x);
}
// a - s * c with real s
template <typename T>
__device__ __forceinline__ cpx<T> fnms_r(cpx<T> a, T s, cpx<T> c) { return mk<T>(a.x - s * c.x, a.y - s * c.y); }
// 1 / a  =  conj(a) / |a|^2.  The operands met here are bounded away from zero and
// from overflow (|a| between ~1e-3 and ~1e8), so no Smith-style scaling is needed.
// binary32: the hardware approximation (rcp.approx.ftz, at most 1 ulp from 1/v) refined
// by one Newton-Raphson step, r + r (1 - v r).  The step roughly squares the relative
// error of the approximation and adds the rounding of two fused operations, so the
// result is within 1 ulp of 1/v but NOT always correctly rounded; .ftz flushes
// subnormal operands and results to zero, which normal-range operands never produce.
// paradiag_recip_f32 exposes this function so that a test can bound its error against
// the correctly rounded reciprocal.  binary64: __drcp_rn, correctly rounded.
__device__ __forceinline__ float rcp_nr(float v) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return fmaf(r, fmaf(-v, r, 1.0f), r);
}
__device__ __forceinline__ double rcp_nr(double v) { return __drcp_rn(v); }
template <typename T>
__device__ __forceinline__ cpx<T> recip(cpx<T> a) {
  const T d = rcp_nr(a.x * a.x + a.y * a.y);  // 1 / |a|^2 (within 1 ulp in binary32)
  return mk<T>(a.x * d, -a.y * d);
}
template <typename T>
__device__ __forceinline__ T abs2(cpx<T> a) { return a.x * a.x + a.y * a.y; }

template <typename T>
__device__ __forceinline__ T shfl_xor(T v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Barrier over a team of P threads (P a multiple of 32) inside a CTA that holds
// blockDim.x / P teams.  Team 0..(teams-1) use named barriers 1..teams.
__device__ __forceinline__ void team_sync(int P, int team_in_cta) {
  if (P == 32) {
    __syncwarp();
  } else if (P == (int)blockDim.x) {
    __syncthreads();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team_in_cta), "r"(P) : "memory");
  }
}

// binary64 -> binary32 by integer operations on the bit pattern: GB300 issues FP64
// instructions, conversions included, at a small fraction of its FP32 and integer rates, and
// the binary32 path converts every FP64 element it loads (in the kernels that also run FP64
// arithmetic, such as the residual, this frees the FP64 pipe; measured 8% on the 2D residual
// DST).  The significand is truncated (error below one binary32 ulp, where round-to-nearest
// gives half an ulp); magnitudes below binary32's normal range become zero, above it
// infinity; NaN stays NaN.
// SCALE: the value times 2^k (|k| < 1000).
template <bool SCALE = false>
__device__ __forceinline__ float f64_to_f32_bits(double x, int k = 0) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  int ef = e - 896;  // binary32 biased exponent: e - 1023 + 127
  if constexpr (SCALE) ef = e == 0 ? 0 : e == 0x7ff ? 255 : ef + k;
  unsigned r;
  if (ef >= 255) {
    r = sign | 0x7f800000u | ((e == 0x7ff && ((hi & 0xfffffu) | lo)) ? 0x00400000u : 0u);
  } else if (ef <= 0) {
    r = sign;
  } else {
    r = sign | ((unsigned)ef << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  }
  return __uint_as_float(r);
}
// The same rounded to nearest (ties away from zero); infinities become NaN.
__device__ __forceinline__ float f64_to_f32_near(double x) {
  return f64_to_f32_bits(__longlong_as_double(__double_as_longlong(x) + 0x10000000LL));
}
// binary32 -> binary64 by integer operations, for the same reason (the stores of the inverse
// transforms: one conversion beside the one FP64 add of U += delta).  Exact for every finite number and
// infinity; NaN stays NaN.  k: times 2^k, |k| <= 800 (every binary32 number then stays normal in
// binary64).  Subnormals are normalised by a multiplication by 2^24, or (BRANCH) take the hardware
// conversion in a branch that no ordinary value enters: faster in the DST (heat2d_255x255x256 1805 ->
// 1755 us), slower in the time DFTs (32 x heat1d_1023x1024 2455 -> 2469 us, advdiff1d_4095x2048 911 -> 923 us).
template <bool BRANCH = false>
__device__ __forceinline__ double f32_to_f64_bits(float x, int k = 0) {
  const bool sub = (__float_as_uint(x) & 0x7f800000u) == 0u;  // subnormal or zero
  const unsigned b = __float_as_uint(!BRANCH && sub ? x * 16777216.0f : x), m = b & 0x7fffffffu;
  const int e = !BRANCH && sub ? k - 24 : k;
  unsigned hi = (m >> 3) + (m >= 0x7f800000u ? 0x70000000u : 0x38000000u + ((unsigned)e << 20));  // exponent + 896 + e
  unsigned lo = m << 29;
  if constexpr (BRANCH) {
    if (sub) {
      hi = lo = 0u;
      if (m != 0u) {
        const double d = (double)x * __hiloint2double((1023 + k) << 20, 0);
        hi = (unsigned)__double2hiint(d);
        lo = (unsigned)__double2loint(d);
      }
    }
  } else if (m == 0u) {
    hi = 0u;
  }
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)lo);
}
// cvt<To>(x): x in type To, between binary64 and binary32 through the integer conversions above.
template <typename To, bool BRANCH = false, typename From>
__device__ __forceinline__ To cvt(From x) {
  if constexpr (sizeof(To) == 4 && sizeof(From) == 8)
    return f64_to_f32_bits(x);
  else if constexpr (sizeof(To) == 8 && sizeof(From) == 4)
    return f32_to_f64_bits<BRANCH>(x);
  else
    return (To)x;
}

// x * 2^k (|k| <= 1000) as ldexp gives it: an exponent-field add for a normal x whose result is normal; else
// (zero, subnormal, infinity, NaN, under- or overflow) a multiplication by the power of two, exact or
// rounded once.  8 x 63 x 63 x 128 in FP64 takes 3971 us; 4031 us with the multiplication for every value,
// an FP64 operation each; 3920 us with flushed subnormals.
__device__ __forceinline__ double pow2_scale(double x, int k) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if ((unsigned)(e - 1) < 0x7feu && (unsigned)(e + k - 1) < 0x7feu) return __hiloint2double(hi + (k << 20), __double2loint(x));
  return x * __hiloint2double((1023 + k) << 20, 0);
}
// Problem scaling of the batches on load and store: x 2^k in type T, and back to binary64.
template <typename T>
__device__ __forceinline__ T slot_load(double x, int k) {
  if constexpr (sizeof(T) == 4)
    return f64_to_f32_bits<true>(x, k);
  else
    return k ? pow2_scale(x, k) : x;
}
template <bool BRANCH = false, typename T>
__device__ __forceinline__ double slot_store(T x, int k) {
  if constexpr (sizeof(T) == 4)
    return f32_to_f64_bits<BRANCH>(x, k);
  else
    return k ? pow2_scale(x, k) : x;
}
// A pointer read from memory, known to be a global address (so that loads through it are global loads).
__device__ __forceinline__ const double *global_ptr(const double *const *p) {
  const double *q = *p;
  __builtin_assume(__isGlobal(q));
  return q;
}

// Programmatic dependent launch: every kernel of this library opens with this wait,
// so a kernel scheduled early (while its predecessor in the stream drains) reads
// nothing before the predecessor has completed; without such a launch it returns at once.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ int bitrev(int j, int logn) {
  return logn == 0 ? 0 : (int)(__brev((unsigned)j) >> (32 - logn));
}

}  // namespace pd
