// Complex DFTs of one line of N = 2^a 3^b points held in a thread's registers
// (every index is a compile-time constant after unrolling, so the arrays never
// leave the register file), natural order in and out.
//
// N = P2 P3 with P2 a power of two and P3 in {1, 3, 9} goes by the prime-factor
// map (Good 1958, Thomas 1963): with n = P3 n1 + P2 n2 mod N and k1 = k mod P2,
// k2 = k mod P3,
//   X[k] = sum_{n1, n2} x[n] e^{s 2 pi i n1 k1 / P2} e^{s 2 pi i n2 k2 / P3},
// so no twiddle factor stands between the two parts.  The padded transforms of
// the 3/2 rule read (inverse) or keep (forward) only the outer two thirds of
// their points.  The radix-3 butterflies combine points N/3 apart, one from
// each third: with the 3-part first, one input of every butterfly is known to
// be zero and its operations are left out (ZP); with the 3-part last, the
// butterfly outputs of the middle third are never used and the compiler drops
// them.
#pragma once

#include "common.cuh"

namespace chdns {

// three-point DFT in place; z: index of an input known to be zero (-1: none)
template <int SIGN, typename R, typename C>
__device__ __forceinline__ void dft3(C& a, C& b, C& c, int z) {
  const R k = (R)SIGN * (R)0.86602540378443864676372317075293618;  // sin(2 pi / 3)
  const R h = (R)0.5;
  if (z == 0) {
    const C s = b + c, d = b - c;
    a = s;
    b = mk(-h * s.x - k * d.y, -h * s.y + k * d.x);
    c = mk(-h * s.x + k * d.y, -h * s.y - k * d.x);
  } else if (z == 1) {
    const C t = mk(a.x - h * c.x, a.y - h * c.y), d = c;
    a = a + c;
    b = mk(t.x + k * d.y, t.y - k * d.x);
    c = mk(t.x - k * d.y, t.y + k * d.x);
  } else if (z == 2) {
    const C t = mk(a.x - h * b.x, a.y - h * b.y), d = b;
    a = a + b;
    b = mk(t.x - k * d.y, t.y + k * d.x);
    c = mk(t.x + k * d.y, t.y - k * d.x);
  } else {
    const C s = b + c, d = b - c;
    const C t = mk(a.x - h * s.x, a.y - h * s.y);
    a = a + s;
    b = mk(t.x - k * d.y, t.y + k * d.x);
    c = mk(t.x + k * d.y, t.y - k * d.x);
  }
}

// x e^{SIGN i t} with the angle's cosine and sine
template <int SIGN, typename R, typename C>
__device__ __forceinline__ C rot(C x, double c, double s) {
  const R cr = (R)c, sr = (R)SIGN * (R)s;
  return mk(x.x * cr - x.y * sr, x.y * cr + x.x * sr);
}

// length 1, 2, 4, 8 or 16
template <int SIGN, int N, typename R, typename C>
__device__ __forceinline__ void dft_pow2(C* x) {
  if constexpr (N == 16) {
    // x[4 a + b] -> X[ka + 4 kb], twiddles e^{SIGN 2 pi i b ka / 16}
    const double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
    C t[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
#pragma unroll
      for (int a = 0; a < 4; ++a) t[b][a] = x[4 * a + b];
      small_dft_ct<SIGN, 4, C, R>(t[b]);
    }
    t[1][1] = rot<SIGN, R>(t[1][1], c1, s1);
    t[1][2] = rot<SIGN, R>(t[1][2], h, h);
    t[1][3] = rot<SIGN, R>(t[1][3], s1, c1);
    t[2][1] = rot<SIGN, R>(t[2][1], h, h);
    t[2][2] = imul((R)SIGN, t[2][2]);
    t[2][3] = rot<SIGN, R>(t[2][3], -h, h);
    t[3][1] = rot<SIGN, R>(t[3][1], s1, c1);
    t[3][2] = rot<SIGN, R>(t[3][2], -h, h);
    t[3][3] = rot<SIGN, R>(t[3][3], -c1, -s1);
#pragma unroll
    for (int ka = 0; ka < 4; ++ka) {
      C u[4] = {t[0][ka], t[1][ka], t[2][ka], t[3][ka]};
      small_dft_ct<SIGN, 4, C, R>(u);
#pragma unroll
      for (int kb = 0; kb < 4; ++kb) x[ka + 4 * kb] = u[kb];
    }
  } else if constexpr (N > 1) {
    small_dft_ct<SIGN, N, C, R>(x);
  }
}

// (a, b) <- (a + w b, a - w b) in six fused operations: a - w b = 2 a - (a + w b)
template <typename R, typename C>
__device__ __forceinline__ void bfly(C& a, C& b, C w) {
  const C s = mk(fma_rn(-w.y, b.y, fma_rn(w.x, b.x, a.x)), fma_rn(w.y, b.x, fma_rn(w.x, b.y, a.y)));
  b = mk(fma_rn((R)2.0, a.x, -s.x), fma_rn((R)2.0, a.y, -s.y));
  a = s;
}

// Length N of x_b w^b, the second half of an inverse line with its twiddles,
// natural order out; w[i] = w^(2^i).  24, 76 and 208 operations at N = 4, 8
// and 16, where the products w^b x_b and dft_pow2 take 28, 80 and 228; two,
// three and four twiddles to load instead of N - 1.  64x65x64 FP64: the passes of
// a step 587 -> 566 us.  The error of the term grows by 1 to 2 % and stays below
// that of the radix passes it replaced (8x8 to 64x64 modes, extended precision:
// 2.7e-16 to 4.1e-16 against 3.1e-16 to 6.2e-16).
template <int N, typename R, typename C>
__device__ __forceinline__ void dft_tw(C* x, const C* w) {
  if constexpr (N == 2) {
    bfly<R>(x[0], x[1], w[0]);
  } else {
    constexpr int H = N / 2;
    C e[H], o[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      e[i] = x[2 * i];
      o[i] = x[2 * i + 1];
    }
    dft_tw<H, R>(e, w + 1);
    dft_tw<H, R>(o, w + 1);
    // X_k, X_{k+H} = E_k +- w e^{2 pi i k / N} O_k
    C v = w[0];
#pragma unroll
    for (int k = 0; k < (H + 1) / 2; ++k) {
      if constexpr (N == 8) {
        if (k == 1) v = rot<+1, R>(w[0], 0.70710678118654752440, 0.70710678118654752440);
      } else if constexpr (N == 16) {
        if (k == 1) v = rot<+1, R>(w[0], 0.92387953251128675613, 0.38268343236508977173);
        if (k == 2) v = rot<+1, R>(w[0], 0.70710678118654752440, 0.70710678118654752440);
        if (k == 3) v = rot<+1, R>(w[0], 0.38268343236508977173, 0.92387953251128675613);
      }
      bfly<R>(e[k], o[k], v);
      if (H > 1) bfly<R>(e[k + H / 2], o[k + H / 2], imul((R)1.0, v));
    }
#pragma unroll
    for (int k = 0; k < H; ++k) {
      x[k] = e[k];
      x[k + H] = o[k];
    }
  }
}
// the twiddles of dft_tw: entries 1, 2, 4, ... of a table column
template <int N, int A, typename C>
__device__ __forceinline__ void load_tw(C* w, const C* tab) {
#pragma unroll
  for (int i = 0; (1 << i) < N; ++i) w[i] = tab[(1 << i) * A];
}
constexpr int log2i(int n) { return n <= 1 ? 0 : 1 + log2i(n / 2); }

// length 1, 3 or 9; z(n) says which of its inputs are known to be zero
template <int SIGN, int N, typename R, typename C, class Z>
__device__ __forceinline__ void dft_pow3(C* x, Z&& zero) {
  if constexpr (N == 3) {
    dft3<SIGN, R>(x[0], x[1], x[2], zero(0) ? 0 : zero(1) ? 1 : zero(2) ? 2 : -1);
  } else if constexpr (N == 9) {
    // x[3 a + b] -> X[ka + 3 kb], twiddles e^{SIGN 2 pi i b ka / 9}
#pragma unroll
    for (int b = 0; b < 3; ++b) dft3<SIGN, R>(x[b], x[3 + b], x[6 + b], zero(b) ? 0 : zero(3 + b) ? 1 : zero(6 + b) ? 2 : -1);
    x[4] = rot<SIGN, R>(x[4], 0.76604444311897803520, 0.64278760968653932632);   // 40 degrees
    x[7] = rot<SIGN, R>(x[7], 0.17364817766693034885, 0.98480775301220805937);   // 80
    x[5] = rot<SIGN, R>(x[5], 0.17364817766693034885, 0.98480775301220805937);   // 80
    x[8] = rot<SIGN, R>(x[8], -0.93969262078590838405, 0.34202014332566873304);  // 160
#pragma unroll
    for (int ka = 0; ka < 3; ++ka) dft3<SIGN, R>(x[3 * ka], x[3 * ka + 1], x[3 * ka + 2], -1);
    // x[3 ka + kb] holds X[ka + 3 kb]: transpose
    C t;
    t = x[1]; x[1] = x[3]; x[3] = t;
    t = x[2]; x[2] = x[6]; x[6] = t;
    t = x[5]; x[5] = x[7]; x[7] = t;
  }
}

__host__ __device__ constexpr int pow3_part(int n) { return n % 9 == 0 ? 9 : n % 3 == 0 ? 3 : 1; }

// k of the CRT: k = k1 mod p2, k = k2 mod p3
__host__ __device__ constexpr int crt_index(int p2, int p3, int k1, int k2) {
  for (int k = 0; k < p2 * p3; ++k)
    if (k % p2 == k1 && k % p3 == k2) return k;
  return 0;
}
template <int P2, int P3>
struct CrtTable {
  int k[P2 * P3] = {};
  constexpr CrtTable() {
    for (int k1 = 0; k1 < P2; ++k1)
      for (int k2 = 0; k2 < P3; ++k2) k[k1 * P3 + k2] = crt_index(P2, P3, k1, k2);
  }
};

// X[k] = sum_n x[n] e^{SIGN 2 pi i n k / N}.  ZP: the inputs N/3 <= n < 2N/3
// are zero and are not read (the 3-part goes first); otherwise the 3-part goes
// last.
template <int SIGN, bool ZP, int N, typename R, typename C>
__device__ __forceinline__ void dft_reg(C (&x)[N]) {
  constexpr int P3 = pow3_part(N), P2 = N / P3;
  static_assert(P2 == 1 || P2 == 2 || P2 == 4 || P2 == 8 || P2 == 16, "2-part not built");
  constexpr CrtTable<P2, P3> crt{};
  C y[P2][P3];
  if constexpr (ZP) {
#pragma unroll
    for (int n1 = 0; n1 < P2; ++n1) {
#pragma unroll
      for (int n2 = 0; n2 < P3; ++n2) {
        const int n = (P3 * n1 + P2 * n2) % N;
        if (n < N / 3 || n >= 2 * N / 3) y[n1][n2] = x[n];
      }
      dft_pow3<SIGN, P3, R>(y[n1], [n1](int n2) {
        const int n = (P3 * n1 + P2 * n2) % N;
        return n >= N / 3 && n < 2 * N / 3;
      });
    }
#pragma unroll
    for (int k2 = 0; k2 < P3; ++k2) {
      C u[P2];
#pragma unroll
      for (int n1 = 0; n1 < P2; ++n1) u[n1] = y[n1][k2];
      dft_pow2<SIGN, P2, R>(u);
#pragma unroll
      for (int k1 = 0; k1 < P2; ++k1) x[crt.k[k1 * P3 + k2]] = u[k1];
    }
  } else {
#pragma unroll
    for (int n2 = 0; n2 < P3; ++n2) {
      C u[P2];
#pragma unroll
      for (int n1 = 0; n1 < P2; ++n1) u[n1] = x[(P3 * n1 + P2 * n2) % N];
      dft_pow2<SIGN, P2, R>(u);
#pragma unroll
      for (int k1 = 0; k1 < P2; ++k1) y[k1][n2] = u[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < P2; ++k1) {
      dft_pow3<SIGN, P3, R>(y[k1], [](int) { return false; });
#pragma unroll
      for (int k2 = 0; k2 < P3; ++k2) x[crt.k[k1 * P3 + k2]] = y[k1][k2];
    }
  }
}

// A padded line of M points is transformed in two register steps around one
// exchange through shared memory, M = A B with 3 | A:
//   inverse: k = B a + b (kept spectrum: a outside the middle third) ->
//            A-point DFTs over a, twiddle e^{2 pi i b ka / M}, B-point DFTs
//            over b -> x = ka + A kb;
//   forward: x = ka + A kb -> B-point DFTs over kb, twiddle, A-point DFTs over
//            ka -> k = B p + s (kept: p outside the middle third).
// B = 4 leaves the fewest operations (twiddles on 3/4 of the points, one
// radix-4 butterfly) and enough independent lines per plane; longer lines take
// B = 8 and 16, so that A stays at 24 points or fewer and a step needs little
// more than 100 registers in FP64 (with A = 48 the passes over 192 and 384
// points held 6 warps per SM).
__host__ __device__ constexpr int line_b(int m) { return m == 6 || m == 18 ? 2 : m <= 96 ? 4 : m <= 192 ? 8 : 16; }
__host__ __device__ constexpr int line_a(int m) { return m / line_b(m); }
// x lines in FP32: up to eight points of all six fields fit a thread, which
// keeps the products in registers
template <typename R> __host__ __device__ constexpr int x_line_b(int m) {
  return sizeof(R) == 4 && m > 192 ? 8 : line_b(m);
}
template <typename R> __host__ __device__ constexpr int x_line_a(int m) { return m / x_line_b<R>(m); }
// padded lengths built: 3/2 of 8, 12, 16, 24, 32, 48, 64, 96, 128, 192 and 256 modes
#define CH_LINE_LENGTHS(X) X(12) X(18) X(24) X(36) X(48) X(72) X(96) X(144) X(192) X(288) X(384)

}  // namespace chdns
