// Small DFTs in registers, natural order in and out, shared by the time DFTs and the DST.
#pragma once

#include "pd_common.cuh"

namespace pd {

// X[k] = sum_i x[i] w^{ik}, w = exp(-2 pi i / 16), in place, natural order in and out:
// radix-4 over i = 4 i1 + i2 (i1 first), twiddles w^{i2 k1}, radix-4 over i2.
template <typename T>
__device__ __forceinline__ void radix4_fwd(cpx<T> &a0, cpx<T> &a1, cpx<T> &a2, cpx<T> &a3) {
  const cpx<T> t0 = add(a0, a2), t1 = sub(a0, a2), t2 = add(a1, a3), t3 = sub(a1, a3);
  const cpx<T> mt3 = mk<T>(t3.y, -t3.x);  // -i t3
  a0 = add(t0, t2);
  a2 = sub(t0, t2);
  a1 = add(t1, mt3);
  a3 = sub(t1, mt3);
}
template <typename T>
__device__ __forceinline__ cpx<T> w16(int m) {  // w^m for the products m of i2, k1 < 4
  constexpr double c = 0.92387953251128675613;  // cos(pi/8)
  constexpr double s = 0.38268343236508977173;  // sin(pi/8)
  constexpr double r = 0.70710678118654752440;  // cos(pi/4)
  switch (m) {
    case 1: return mk<T>((T)c, (T)-s);
    case 2: return mk<T>((T)r, (T)-r);
    case 3: return mk<T>((T)s, (T)-c);
    case 4: return mk<T>(T(0), T(-1));
    case 6: return mk<T>((T)-r, (T)-r);
    case 9: return mk<T>((T)-c, (T)s);
    default: return mk<T>(T(1), T(0));
  }
}
template <typename T>
__device__ __forceinline__ void dft16(cpx<T> (&x)[16]) {
#pragma unroll
  for (int i2 = 0; i2 < 4; ++i2) radix4_fwd(x[i2], x[4 + i2], x[8 + i2], x[12 + i2]);  // x[4 k1 + i2]
#pragma unroll
  for (int k1 = 1; k1 < 4; ++k1)
#pragma unroll
    for (int i2 = 1; i2 < 4; ++i2) x[4 * k1 + i2] = mul(w16<T>(i2 * k1), x[4 * k1 + i2]);
  cpx<T> y[16];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    cpx<T> b0 = x[4 * k1], b1 = x[4 * k1 + 1], b2 = x[4 * k1 + 2], b3 = x[4 * k1 + 3];
    radix4_fwd(b0, b1, b2, b3);
    y[k1] = b0;
    y[k1 + 4] = b1;
    y[k1 + 8] = b2;
    y[k1 + 12] = b3;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = y[k];
}


// X[k] = sum_i x[i] w^{ik}, w = exp(-2 pi i / 8): two 4-point DFTs of the even and odd samples.
template <typename T>
__device__ __forceinline__ void dft8(cpx<T> (&x)[8]) {
  constexpr double r = 0.70710678118654752440;  // cos(pi/4)
  radix4_fwd(x[0], x[2], x[4], x[6]);
  radix4_fwd(x[1], x[3], x[5], x[7]);
  const cpx<T> o1 = mk<T>((T)r * (x[3].x + x[3].y), (T)r * (x[3].y - x[3].x));   // w o
  const cpx<T> o2 = mk<T>(x[5].y, -x[5].x);                                      // w^2 o
  const cpx<T> o3 = mk<T>((T)r * (x[7].y - x[7].x), (T)-r * (x[7].x + x[7].y));  // w^3 o
  const cpx<T> e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1];
  x[0] = add(e0, o0);
  x[4] = sub(e0, o0);
  x[1] = add(e1, o1);
  x[5] = sub(e1, o1);
  x[2] = add(e2, o2);
  x[6] = sub(e2, o2);
  x[3] = add(e3, o3);
  x[7] = sub(e3, o3);
}

// exp(-2 pi i m / 32), 0 <= m < 16
template <typename T>
__device__ __forceinline__ cpx<T> w32(int m) {
  constexpr double c1 = 0.98078528040323044913, s1 = 0.19509032201612826785;  // pi/16
  constexpr double c2 = 0.92387953251128675613, s2 = 0.38268343236508977173;
  constexpr double c3 = 0.83146961230254523708, s3 = 0.55557023301960222474;
  constexpr double c4 = 0.70710678118654752440;
  constexpr double c[9] = {1.0, c1, c2, c3, c4, s3, s2, s1, 0.0};
  return m <= 8 ? mk<T>((T)c[m], (T)-c[8 - m]) : mk<T>((T)-c[16 - m], (T)-c[m - 8]);
}
// 32 points: two 16-point DFTs of the even and odd samples.
template <typename T>
__device__ __forceinline__ void dft32(cpx<T> (&x)[32]) {
  cpx<T> e[16], o[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    e[i] = x[2 * i];
    o[i] = x[2 * i + 1];
  }
  dft16(e);
  dft16(o);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const cpx<T> t = k == 0 ? o[0] : (k == 8 ? mk<T>(o[8].y, -o[8].x) : mul(w32<T>(k), o[k]));
    x[k] = add(e[k], t);
    x[k + 16] = sub(e[k], t);
  }
}
// exp(-2 pi i m / N), 0 <= m <= N / 4, N a power of two up to 64
template <typename T, int N>
__device__ __forceinline__ cpx<T> wn(int m) {
  constexpr double c[17] = {1.0, 0.9951847266721968862448, 0.9807852804032304491261, 0.9569403357322088649357,
                            0.9238795325112867561281, 0.8819212643483550297127, 0.8314696123025452370787,
                            0.7730104533627369608109, 0.7071067811865475244008, 0.6343932841636454982151,
                            0.5555702330196022247428, 0.4713967368259976485563, 0.3826834323650897717284,
                            0.2902846772544623676361, 0.1950903220161282678482, 0.0980171403295606019941, 0.0};
  const int t = m * (64 / N);  // c[k] = cos(pi k / 32)
  return mk<T>((T)c[t], (T)-c[16 - t]);
}

// Real input: X[k] = sum_i x[O + S i] w^{ik}, w = exp(-2 pi i / N), k = 0 .. N/2 (X[0] and X[N/2] real),
// by halving: even and odd samples, X[k] = E[k] + w^k O[k], X[N/2 - k] = conj(E[k] - w^k O[k]).
template <typename T, int N, int S, int O, int M>
__device__ __forceinline__ void rdft(const T (&x)[M], cpx<T> (&X)[N / 2 + 1]) {
  if constexpr (N == 4) {
    const T a = x[O] + x[O + 2 * S], b = x[O + S] + x[O + 3 * S];
    X[0] = mk<T>(a + b, T(0));
    X[1] = mk<T>(x[O] - x[O + 2 * S], x[O + 3 * S] - x[O + S]);
    X[2] = mk<T>(a - b, T(0));
  } else {
    cpx<T> e[N / 4 + 1], o[N / 4 + 1];
    rdft<T, N / 2, 2 * S, O, M>(x, e);
    rdft<T, N / 2, 2 * S, O + S, M>(x, o);
    X[0] = mk<T>(e[0].x + o[0].x, T(0));
    X[N / 2] = mk<T>(e[0].x - o[0].x, T(0));
    X[N / 4] = mk<T>(e[N / 4].x, -o[N / 4].x);
#pragma unroll
    for (int k = 1; k < N / 4; ++k) {
      const cpx<T> t = mul(wn<T, N>(k), o[k]);
      X[k] = add(e[k], t);
      X[N / 2 - k] = conjg(sub(e[k], t));
    }
  }
}

// Hermitian input (X[N - k] = conj X[k], given k = 0 .. N/2; the imaginary parts of X[0] and X[N/2] do
// not count), real output x[O + S i] = sum_k X[k] w^{ik}: the transpose of rdft.
template <typename T, int N, int S, int O, int M>
__device__ __forceinline__ void hdft(const cpx<T> (&X)[N / 2 + 1], T (&x)[M]) {
  if constexpr (N == 4) {
    const T s = X[0].x + X[2].x, d = X[0].x - X[2].x, p = X[1].x + X[1].x, q = X[1].y + X[1].y;
    x[O] = s + p;
    x[O + 2 * S] = s - p;
    x[O + S] = d + q;
    x[O + 3 * S] = d - q;
  } else {
    cpx<T> a[N / 4 + 1], b[N / 4 + 1];
    a[0] = mk<T>(X[0].x + X[N / 2].x, T(0));
    b[0] = mk<T>(X[0].x - X[N / 2].x, T(0));
    a[N / 4] = mk<T>(X[N / 4].x + X[N / 4].x, T(0));
    b[N / 4] = mk<T>(X[N / 4].y + X[N / 4].y, T(0));
#pragma unroll
    for (int k = 1; k < N / 4; ++k) {
      const cpx<T> v = conjg(X[N / 2 - k]);
      a[k] = add(X[k], v);
      b[k] = mul(wn<T, N>(k), sub(X[k], v));
    }
    hdft<T, N / 2, 2 * S, O, M>(a, x);
    hdft<T, N / 2, 2 * S, O + S, M>(b, x);
  }
}

template <typename T, int R>
__device__ __forceinline__ void dft_reg(cpx<T> (&x)[R]) {
  static_assert(R == 4 || R == 8 || R == 16 || R == 32, "built sizes");
  if constexpr (R == 4)
    radix4_fwd(x[0], x[1], x[2], x[3]);
  else if constexpr (R == 8)
    dft8(x);
  else if constexpr (R == 16)
    dft16(x);
  else
    dft32(x);
}

}  // namespace pd
