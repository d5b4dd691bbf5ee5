// Shared device helpers of the channel-flow library: complex arithmetic,
// in-place mixed-radix FFT stages in shared memory, and the launch structs
// passed from the host code to the kernels.
#pragma once

#include <cmath>

#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>
#include <utility>

#include "smem_limit.h"

namespace chdns {

constexpr int kMaxNy = 201;                    // largest Chebyshev node count built
constexpr int kMaxRadixStages = 16;

// ---------------------------------------------------------------------------
// complex helpers for double2 / float2
// ---------------------------------------------------------------------------
template <typename R> struct cpx;
template <> struct cpx<double> { using T = double2; };
template <> struct cpx<float> { using T = float2; };

__host__ __device__ __forceinline__ double2 mk(double x, double y) { return make_double2(x, y); }
__host__ __device__ __forceinline__ float2 mk(float x, float y) { return make_float2(x, y); }

// Round-to-nearest multiply and fused multiply-add that the compiler never
// contracts or splits.  An expression such as a*b - c*d may be fused either
// way, and the choice can differ between kernels that inline the same code;
// the arithmetic that several kernel forms share (so that their results agree
// bit for bit) is written with these.
__host__ __device__ __forceinline__ double fma_rn(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
__host__ __device__ __forceinline__ float fma_rn(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
__host__ __device__ __forceinline__ double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

// float -> double by integer operations on the encoding: the conversion
// instruction occupies the FP64 pipe like an FP64 operation (17 of 19 cycles
// per warp and SM), and the implicit solves are bound by that pipe.  The same
// values for every argument (a NaN stays one).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  const bool sub = a < 0x00800000u;  // subnormal: exponent from 2^64 |f|
  const unsigned v = sub ? __float_as_uint(__uint_as_float(a) * 0x1p64f) : a;
  unsigned hi = (v >> 3) + (a >= 0x7f800000u ? 0x70000000u : sub ? 0x34000000u : 0x38000000u);
  if (a == 0u) hi = 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(v << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// double -> float, round to nearest even, by integer operations (as widen; a
// subnormal result is rounded once more when it is scaled back).  Taking the
// conversion instruction for subnormals, on a branch, costs a 256x193x256 step
// 20 %.
__device__ __forceinline__ float narrow(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d), a0 = h & 0x7fffffffu;
  const bool sub = a0 < 0x38100000u;                               // subnormal: rounded at 2^64 |d|, then scaled
  const unsigned a = sub ? a0 + 0x04000000u : a0;
  unsigned u = __funnelshift_l(l, a - 0x38000000u, 3);             // exponent rebiased, 23 fraction bits
  u += ((l & 0x1fffffffu) + 0x0fffffffu + (u & 1u)) >> 29;          // the 29 bits dropped
  if (a < 0x38100000u) u = 0u;
  if (a >= 0x47f00000u) u = a > 0x7ff00000u || (a == 0x7ff00000u && l) ? 0x7fffffffu : 0x7f800000u;  // NaN, else infinity
  return __uint_as_float(u | (h & 0x80000000u)) * (sub ? 0x1p-64f : 1.0f);
}

#define CH_CPX_OPS(C, R)                                                                   \
  __host__ __device__ __forceinline__ C operator+(C a, C b) { return mk(a.x + b.x, a.y + b.y); } \
  __host__ __device__ __forceinline__ C operator-(C a, C b) { return mk(a.x - b.x, a.y - b.y); } \
  __host__ __device__ __forceinline__ C operator*(R s, C a) { return mk(s * a.x, s * a.y); }     \
  __host__ __device__ __forceinline__ C cmul(C a, C b) {                                  \
    return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);                              \
  }                                                                                       \
  __host__ __device__ __forceinline__ C cconj(C a) { return mk(a.x, -a.y); }                \
  /* i * s * a */                                                                         \
  __host__ __device__ __forceinline__ C imul(R s, C a) { return mk(-s * a.y, s * a.x); }

CH_CPX_OPS(double2, double)
CH_CPX_OPS(float2, float)
#undef CH_CPX_OPS

template <typename C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }

// Asynchronous copy of one 4-, 8- or 16-byte element from global to shared
// memory (cp.async): no register holds the value, so a thread issues all its
// copies of a tile before any completes.  cp_async_wait_all() waits for the
// thread's own copies; a barrier after it publishes the tile to the CTA.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "cp.async copies 4, 8 or 16 bytes");
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(sizeof(T)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Plain stream-ordered launch.  Programmatic dependent launch was measured and
// left out: a dependent that starts early takes shared memory and registers
// from the CTAs that its predecessor still has to place.  With the trigger
// after the wait a 64x65x64 FP64 step took 25 % longer; mixed-precision steps
// took with / without it (us): 388 / 366 at 24x50x48 x 8, 402 / 391 at
// 64x65x64 x 2 (forced), 878 / 875 at 128x129x128, 1084 / 1086 at 16x65x16 x 256.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------------------
// FFT plans and in-place stages
// ---------------------------------------------------------------------------
struct FftPlan {
  int n;
  int nst;
  int radix[kMaxRadixStages];
};

// e^{SIGN 2 pi i k / n} from a table of e^{+2 pi i k / n}
template <int SIGN, typename C>
__device__ __forceinline__ C twiddle(const C* tw, int k) {
  C w = tw[k];
  if (SIGN < 0) w.y = -w.y;
  return w;
}

// Small DFT y_u = sum_t x_t e^{SIGN 2 pi i t u / r}, r in {2, 3, 4, 8}; {2, 3, 4} at run time.
template <int SIGN, int RADIX, typename C, typename R>
__device__ __forceinline__ void small_dft_ct(C* x) {
  if constexpr (RADIX == 2) {
    C a = x[0], b = x[1];
    x[0] = a + b;
    x[1] = a - b;
  } else if constexpr (RADIX == 3) {
    const R k = (R)SIGN * (R)0.86602540378443864676372317075293618;
    C s = x[1] + x[2];
    C d = x[1] - x[2];
    C t1 = x[0] - (R)0.5 * s;
    C rot = imul(k, d);
    x[0] = x[0] + s;
    x[1] = t1 + rot;
    x[2] = t1 - rot;
  } else if constexpr (RADIX == 4) {
    C a0 = x[0] + x[2], a1 = x[0] - x[2];
    C b0 = x[1] + x[3], b1 = x[1] - x[3];
    C wb1 = imul((R)SIGN, b1);
    x[0] = a0 + b0;
    x[1] = a1 + wb1;
    x[2] = a0 - b0;
    x[3] = a1 - wb1;
  } else {
    // radix 8: length-4 DFTs of the even and the odd samples, combined with
    // w^u, w = e^{SIGN 2 pi i / 8} = (1 + SIGN i) / sqrt 2
    const C a0 = x[0] + x[4], a1 = x[0] - x[4], a2 = x[2] + x[6], a3 = x[2] - x[6];
    const C e0 = a0 + a2, e2 = a0 - a2;
    const C e1 = a1 + imul((R)SIGN, a3), e3 = a1 - imul((R)SIGN, a3);
    const C b0 = x[1] + x[5], b1 = x[1] - x[5], b2 = x[3] + x[7], b3 = x[3] - x[7];
    const C o0 = b0 + b2;
    const C p2 = b0 - b2;
    const C p1 = b1 + imul((R)SIGN, b3), p3 = b1 - imul((R)SIGN, b3);
    const R h = (R)0.70710678118654752440084436210484904;
    const C o1 = mk(h * (p1.x - (R)SIGN * p1.y), h * (p1.y + (R)SIGN * p1.x));    // p1 w
    const C o2 = imul((R)SIGN, p2);                                               // p2 w^2
    const C o3 = mk(h * (-p3.x - (R)SIGN * p3.y), h * (-p3.y + (R)SIGN * p3.x));  // p3 w^3
    x[0] = e0 + o0;
    x[4] = e0 - o0;
    x[1] = e1 + o1;
    x[5] = e1 - o1;
    x[2] = e2 + o2;
    x[6] = e2 - o2;
    x[3] = e3 + o3;
    x[7] = e3 - o3;
  }
}
template <int SIGN, typename C, typename R>
__device__ __forceinline__ void small_dft(C* x, int r) {
  if (r == 2) small_dft_ct<SIGN, 2, C, R>(x);
  else if (r == 3) small_dft_ct<SIGN, 3, C, R>(x);
  else small_dft_ct<SIGN, 4, C, R>(x);
}

// Line l of a batch starts at (l / g) * (n g) + (l % g) with element stride g
// (g = 1: contiguous lines).  `bf_fastest` picks which index consecutive
// threads walk: butterflies of one line (contiguous lines) or lines
// (strided lines), so that neighbouring threads touch neighbouring words.

// Decimation in frequency: natural-order input, digit-reversed output.
template <int SIGN, typename R>
__device__ void fft_dif(typename cpx<R>::T* buf, int nlines, int g, const FftPlan& pl,
                        const typename cpx<R>::T* tw, bool bf_fastest) {
  using C = typename cpx<R>::T;
  const int n = pl.n;
  int L = n;
  for (int s = 0; s < pl.nst; ++s) {
    const int r = pl.radix[s];
    const int m = L / r;
    const int nb = n / r;
    const int tstep = n / L;
    const int total = nlines * nb;
    for (int w = threadIdx.x; w < total; w += blockDim.x) {
      int l, bf;
      if (bf_fastest) { bf = w % nb; l = w / nb; } else { l = w % nlines; bf = w / nlines; }
      C* base = buf + (l / g) * (n * g) + (l % g);
      const int blk = bf / m, q = bf % m;
      const int i0 = blk * L + q;
      C x[4];
      for (int t = 0; t < r; ++t) x[t] = base[(i0 + t * m) * g];
      small_dft<SIGN, C, R>(x, r);
      for (int u = 0; u < r; ++u) {
        C y = x[u];
        if (u > 0 && q > 0) y = cmul(y, twiddle<SIGN>(tw, q * u * tstep));
        base[(i0 + u * m) * g] = y;
      }
    }
    __syncthreads();
    L = m;
  }
}

// Decimation in time with the radices in reverse order: digit-reversed input
// (as produced by fft_dif with the same plan), natural-order output.
template <int SIGN, typename R>
__device__ void fft_dit(typename cpx<R>::T* buf, int nlines, int g, const FftPlan& pl,
                        const typename cpx<R>::T* tw, bool bf_fastest) {
  using C = typename cpx<R>::T;
  const int n = pl.n;
  int L = 1;
  for (int s = pl.nst - 1; s >= 0; --s) {
    const int r = pl.radix[s];
    const int m = L;
    L = L * r;
    const int nb = n / r;
    const int tstep = n / L;
    const int total = nlines * nb;
    for (int w = threadIdx.x; w < total; w += blockDim.x) {
      int l, bf;
      if (bf_fastest) { bf = w % nb; l = w / nb; } else { l = w % nlines; bf = w / nlines; }
      C* base = buf + (l / g) * (n * g) + (l % g);
      const int blk = bf / m, q = bf % m;
      const int i0 = blk * L + q;
      C x[4];
      for (int t = 0; t < r; ++t) {
        C v = base[(i0 + t * m) * g];
        if (t > 0 && q > 0) v = cmul(v, twiddle<SIGN>(tw, q * t * tstep));
        x[t] = v;
      }
      small_dft<SIGN, C, R>(x, r);
      for (int u = 0; u < r; ++u) base[(i0 + u * m) * g] = x[u];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// launch structs
// ---------------------------------------------------------------------------
struct Grid {
  int nx, ny, nz, nxh, P, N, mx, mz;
  // strides (complex values) of PencilBufs.Q between fields, nodes and environments
  size_t qf, qj, qb;
};

template <typename R>
struct PlaneArgs {
  using C = typename cpx<R>::T;
  // q [B][6][ny][P] and h [B][3][ny][P] in ch_nonlinear.  In a step both are
  // PencilBufs.Q, H over the first three fields: every kernel reads the part of
  // q that its writes of h cover (the columns of a pass, the plane of a CTA or a
  // cluster) before a barrier in front of them
  const C* q;
  C* h;
  size_t qf, qj, qb, hb;  // strides of fields and nodes (both), of environments (q, h)
  int nxh, nz, ny, mx, mz, P;
  int S, Lz, NP;
  // (in passes tw_x and tw_mz hold [B][A] e^{2 pi i s k / (A B)} of their line splits, fft_reg.cuh)
  const C* tw_x;       // [mx]  e^{2 pi i k / mx}
  const C* tw_z;       // [Lz]  e^{2 pi i k / Lz}
  const C* tw_mz;      // [mz]  e^{2 pi i k / mz}
  FftPlan px, pz;
  R scale;             // 1 / (mx mz)
  const int* active;   // [B] slots to process (nullptr: all)
  // planes of 16 x 16 modes (plane_small.cu): 1 in batches that fill the GPU, 2
  // on two-CTA clusters
  int team16;
  // three passes through global memory (z inverse, x transforms and products,
  // z forward; plane_pass.cuh)
  int passes;
  C* y;                // [B][ny][6][mz][nxh]: z-transformed columns, then H in fields 0..2 (PencilBufs.Q)
  int cluster;         // ch_info_t.plane_cluster
};

// Per-mode tau tables (device), mode index fastest so that threads owning
// consecutive modes read consecutive words.  Mh = N/2 + 1.
struct TauTables {
  const double* helm;      // [3][2][4][Mh][P]  e, h, b, Q of (D^2 - k^2 - 1/(beta dt nu)) per stage, parity
  const double* helm_isq;  // [3][2][P]         1 / sum Q
  const double* pois;      // [2][4][Mh][P]     same for (D^2 - k^2)
  const double* pois_isq;  // [2][P]
  const double* vh;        // [3][2][Mh][P]     homogeneous v of the influence matrix, parity-indexed
  const double* vh_idv;    // [3][2][P]         1 / sum_{n of parity} n^2 vh_n
  const double* u1;        // [3][Mh]           mean response to unit forcing (even parity)
  const double* u1_iflux;  // [3]               1 / int u1 dy
  const double* rowc;      // [3][ny]           tau row constants cA_n, cB_n, cC_n
  // the same factorisations with the row constants folded in, eA = e cA_n,
  // eB = e cB_n, eC = e cC_n, then h, b, the wall weights W (W_{M-1} = 1,
  // W_i = 1 + b_{i+1} W_{i+1}: sum_i P_i = sum_i W_i a_i) and, for the stage's
  // Helmholtz operator, E1 = (1 + alpha/beta) e and under a free-slip top W2
  // (W2_{M-1} = n^2, W2_i = n_i^2 + b_{i+1} W2_{i+1}: sum n^2 P = sum W2_i a_i)
  // eA, eB, eC, h, b, W, E1 (, W2) per stage, parity and eA, eB, eC, h, b, W per parity, the entries of a
  // row side by side for a tile of sixteen modes kz >= 0: [3][2] and [2] of [tile][rows 1 .. Mh][7 or 8, 6][16]
  const double* helm_f;
  const double* pois_f;
  const double* n2;        // [ny] n^2
  const double* n1;        // [ny] 2 (n + 1)
  const double* wint;      // [ny] int T_n dy = 2 / (1 - n^2) of the even n, 0 of the odd
  // free-slip top (top_bc = 1): the wall rows couple the parities
  const double* helm_top;  // [3][2][2][P]      sum Q, sum n^2 Q of the stage's factorisation, per parity
  const double* vh_top;    // [3][2][2][P]      A = sum n^2 (n^2 - 1) / 3 vh_n, B = sum n^2 vh_n, per parity
  const double* mean_top;  // [3][4]            mean mode: int Q_e; sum, sum n^2 and int of u1
  int Mh;
  int top_bc;              // 0 no-slip upper wall; 1 free slip (u1 then holds the affine forcing response)
};

struct StageCoef {
  double alpha, beta, gamma, zeta, dt, nu, theta, flux;
  double cc;                  // alpha / beta
  float dgaf, dzef, dgal, dzel;  // dt gamma, dt zeta as sums of two FP32 values (f + l)
  int k;
};

}  // namespace chdns
