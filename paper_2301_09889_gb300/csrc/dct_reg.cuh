// Real cosine transforms of one line in a thread's registers, lengths 2^a and
// 3 2^a, compile-time indices and constants throughout.
//
//   dct1<N>: X_k = sum_{n=0}^{N}   x_n cos(pi k n / N)                  (N + 1 points)
//   dct2<M>: X_k = sum_{n=0}^{M-1} x_n cos(pi k (2n+1) / (2M))
//   dct3<M>: X_m = sum_{j=0}^{M-1} x_j cos(pi j (2m+1) / (2M))
//   dct4<K>: X_k = sum_{n=0}^{K-1} x_n cos(pi (2k+1) (2n+1) / (4K))
//
// Each splits by the parity of its indices into halves (the classical
// decompositions, e.g. Rao and Yip, Discrete Cosine Transform, 1990): dct1
// into a dct1 and a dct2 (or dct3) of half the length, dct2 and dct3 into
// themselves and a dct4, and dct4 into one complex DFT of a quarter of its
// 2K real degrees of freedom between two rotations: with
// z_n = x_{2n} + i x_{K-1-2n} and w_n = e^{-i pi (8n+1) / (8K)},
//   c_k = w_k sum_n z_n w_n e^{-2 pi i k n / (K/2)},  X_{2k} = Re c_k, X_{K-1-2k} = -Im c_k.
// Rotations and butterflies only (no division by small cosines), so the
// rounding error is that of an FFT.  65 real points take 539 operations,
// against 2145 for the parity-split direct sums.
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"

namespace chdns {

// cos and sin of pi k / n, 0 <= k / n <= 1/2, at compile time (Taylor series on
// [0, pi/4], reflection above)
__host__ __device__ constexpr double taylor_cos(double x) {
  double s = 0.0, x2 = x * x;
  for (int i = 13; i >= 1; --i) s = -x2 / (double)((2 * i - 1) * (2 * i)) * (1.0 + s);
  return 1.0 + s;
}
__host__ __device__ constexpr double taylor_sin(double x) {
  double s = 0.0, x2 = x * x;
  for (int i = 13; i >= 1; --i) s = -x2 / (double)((2 * i) * (2 * i + 1)) * (1.0 + s);
  return x * (1.0 + s);
}
constexpr double kPi = 3.14159265358979323846264338327950288;
__host__ __device__ constexpr double cos_pi(int k, int n) {
  return 4 * k <= n ? taylor_cos(kPi * k / n) : taylor_sin(kPi * (n - 2 * k) / (2.0 * n));
}
__host__ __device__ constexpr double sin_pi(int k, int n) {
  return 4 * k <= n ? taylor_sin(kPi * k / n) : taylor_cos(kPi * (n - 2 * k) / (2.0 * n));
}
// w_n = e^{-i pi (8n+1) / (8K)}, n < K/2
template <int K>
struct Dct4Table {
  double c[K / 2 > 0 ? K / 2 : 1] = {}, s[K / 2 > 0 ? K / 2 : 1] = {};
  constexpr Dct4Table() {
    for (int n = 0; n < K / 2; ++n) {
      c[n] = cos_pi(8 * n + 1, 8 * K);
      s[n] = sin_pi(8 * n + 1, 8 * K);
    }
  }
};

template <int K, typename R>
__device__ __forceinline__ void dct4(R (&x)[K]) {
  using C = typename cpx<R>::T;
  if constexpr (K == 1) {
    x[0] = (R)0.70710678118654752440 * x[0];
  } else if constexpr (K == 2) {
    const R c = (R)cos_pi(1, 8), s = (R)sin_pi(1, 8);
    const R a = c * x[0] + s * x[1], b = s * x[0] - c * x[1];
    x[0] = a;
    x[1] = b;
  } else if constexpr (K == 3) {
    const R c1 = (R)cos_pi(1, 12), c3 = (R)0.70710678118654752440, c5 = (R)cos_pi(5, 12);
    const R m = c3 * x[1];
    const R a = c1 * x[0] + c5 * x[2] + m, b = c3 * (x[0] - x[1] - x[2]), d = c5 * x[0] + c1 * x[2] - m;
    x[0] = a;
    x[1] = b;
    x[2] = d;
  } else {
    constexpr int H = K / 2;
    constexpr Dct4Table<K> w{};
    C z[H];
#pragma unroll
    for (int n = 0; n < H; ++n) z[n] = rot<-1, R>(mk(x[2 * n], x[K - 1 - 2 * n]), w.c[n], w.s[n]);
    dft_reg<-1, false, H, R>(z);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const C c = rot<-1, R>(z[k], w.c[k], w.s[k]);
      x[2 * k] = c.x;
      x[K - 1 - 2 * k] = -c.y;
    }
  }
}

template <int M, typename R>
__device__ __forceinline__ void dct2(R (&x)[M]) {
  if constexpr (M == 3) {
    const R s = x[0] + x[2], d = x[0] - x[2], m = x[1];
    x[0] = s + m;
    x[1] = (R)0.86602540378443864676 * d;
    x[2] = (R)0.5 * s - m;
  } else if constexpr (M > 1) {
    constexpr int H = M / 2;
    R s[H], d[H];
#pragma unroll
    for (int n = 0; n < H; ++n) {
      s[n] = x[n] + x[M - 1 - n];
      d[n] = x[n] - x[M - 1 - n];
    }
    dct2<H, R>(s);
    dct4<H, R>(d);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      x[2 * k] = s[k];
      x[2 * k + 1] = d[k];
    }
  }
}

template <int M, typename R>
__device__ __forceinline__ void dct3(R (&x)[M]) {
  if constexpr (M == 3) {
    const R a = x[0] + (R)0.5 * x[2], b = (R)0.86602540378443864676 * x[1], m = x[0] - x[2];
    x[0] = a + b;
    x[1] = m;
    x[2] = a - b;
  } else if constexpr (M > 1) {
    constexpr int H = M / 2;
    R a[H], b[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      a[j] = x[2 * j];
      b[j] = x[2 * j + 1];
    }
    dct3<H, R>(a);
    dct4<H, R>(b);
#pragma unroll
    for (int m = 0; m < H; ++m) {
      x[m] = a[m] + b[m];
      x[M - 1 - m] = a[m] - b[m];
    }
  }
}

template <int N, typename R>
__device__ __forceinline__ void dct1(R (&x)[N + 1]) {
  if constexpr (N == 1) {
    const R a = x[0] + x[1], b = x[0] - x[1];
    x[0] = a;
    x[1] = b;
  } else if constexpr (N == 2) {
    const R s = x[0] + x[2], d = x[0] - x[2], m = x[1];
    x[0] = s + m;
    x[1] = d;
    x[2] = s - m;
  } else if constexpr (N == 3) {
    const R s = x[0] + x[3], d = x[0] - x[3], p = x[1] + x[2], m = x[1] - x[2];
    x[0] = s + p;
    x[1] = d + (R)0.5 * m;
    x[2] = s - (R)0.5 * p;
    x[3] = d - m;
  } else {
    static_assert(N % 2 == 0, "length not built");
    constexpr int H = N / 2;
    R e[H + 1], o[H];
#pragma unroll
    for (int m = 0; m <= H; ++m) e[m] = x[2 * m];
#pragma unroll
    for (int m = 0; m < H; ++m) o[m] = x[2 * m + 1];
    dct1<H, R>(e);
    dct2<H, R>(o);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      x[k] = e[k] + o[k];
      x[N - k] = e[k] - o[k];
    }
    x[H] = e[H];
  }
}

// Chebyshev orders N the register transforms are built for: 2^a and 3 2^a
#define CH_DCT_ORDERS(X) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192)

}  // namespace chdns
