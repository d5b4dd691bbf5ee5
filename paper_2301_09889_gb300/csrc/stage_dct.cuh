// The explicit half of a stage and the Chebyshev analysis of H with the line
// transforms in registers, for Chebyshev orders N with a register cosine
// transform (dct_reg.cuh):
//
//   stage_pre_dct : (v, omega_y, U, W) coefficients -> coefficients of u, v, w,
//                   omega_x, omega_y, omega_z -> their values at the
//                   Gauss-Lobatto nodes;
//   analysis_dct  : nodal values of H -> Chebyshev coefficients, in place.
//
// A warp holds 16 modes x 2 components of one field and one parity of its
// coefficients: loads and stores are contiguous runs, every lane runs the same
// operations, and the parity's N/2 + 1 values fit the registers up to N = 192
// in FP64.  The even and odd parts of a line meet in shared memory
// (f_j = E_j + O_j, f_{N-j} = E_j - O_j).
//
// What bounds it: FP64 lines by the FP64 pipe (539 operations per 65-point
// line and 0 to 6 per coefficient for the recurrences, against 2.2 times as
// many in the FFT form with its serial prefix sums); FP32 lines by issue and
// L2.
#pragma once

#include "common.cuh"
#include "dct_reg.cuh"
#include "internal.h"

namespace chdns {

// ---------------------------------------------------------------------------
// stage_pre_dct
//   u = (i kx Dv - i kz g)/k^2, w = (i kz Dv + i kx g)/k^2,
//   omega_x = Dw - i kz v, omega_z = i kx v - Du;  mean mode: u = U, w = W,
//   omega_x = DW, omega_z = -DU.
// Component r of (i s X) is sgn_r s X_{1-r}.  With Va, Ga the other component
// of v and omega_y, every field is
//   u, w            : cD (Dv)_n + cS S_n                      S = Ga (mean: U, W)
//   v, omega_y      : S_n                                     S = v, omega_y
//   omega_x, omega_z: cD (D^2 v)_n + cS (DS)_n + cV Va_n      S = Ga (mean: W, U)
// The derivatives are running sums from n = N down (c_m b_m = b_{m+2} +
// 2 (m+1) a_{m+1}), in the node precision.
// ---------------------------------------------------------------------------
template <typename RN> constexpr int dct_fields(int nf) { return sizeof(RN) == 4 ? nf : 1; }  // fields per CTA
// CTAs per SM the registers are held to: one parity's array and the transform
// around it
constexpr int ctas_of(int regs, int threads) { return 65536 / (regs * threads) > 0 ? 65536 / (regs * threads) : 1; }
template <typename RN, int N> constexpr int pre_dct_regs() {
  return sizeof(RN) == 8 ? (N <= 32 ? 96 : N <= 64 ? 168 : 255) : (N <= 32 ? 56 : N <= 64 ? 80 : N <= 96 ? 112 : 168);
}
template <typename RN, int N> constexpr int analysis_dct_regs() {
  return sizeof(RN) == 8 ? (N <= 32 ? 128 : 255) : (N <= 32 ? 72 : N <= 64 ? 128 : N <= 96 ? 168 : 255);
}

template <typename RN, int N, int NF>
__global__ void __launch_bounds__(64 * NF, ctas_of(pre_dct_regs<RN, N>(), 64 * NF)) stage_pre_dct_kernel(Grid g, PencilBufs pb, DevTables t,
                                                                    typename cpx<RN>::T* __restrict__ q) {
  constexpr int H = N / 2;
  // FP32 lines: v and omega_y of the tile are rounded to FP32 once, into shared
  // memory (a conversion costs as much as an FP64 operation, and every line
  // reads two of the columns); FP64 lines read them in place
  constexpr bool kTile = sizeof(RN) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P, ny = N + 1;
  const int lane = threadIdx.x & 31, fl = threadIdx.x / 64, half = (threadIdx.x / 32) & 1, f = blockIdx.z * NF + fl;
  RN* tile = reinterpret_cast<RN*>(smem_raw);  // [v, omega_y][ny][32], until the partial sums take its place
  RN* part = reinterpret_cast<RN*>(smem_raw) + fl * (N + 1) * 32;  // [E_0 .. E_H, O_0 .. O_{H-1}][32]
  const int p = blockIdx.x * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  pdl_wait_then_release();  // v, omega_y come from the previous stage
  if constexpr (kTile) {
    // a column per warp and step, every load in flight before the first store
    constexpr int KL = (2 * (N + 1) + 2 * NF - 1) / (2 * NF);
    const size_t c0 = 2 * ((size_t)b * ny * P + blockIdx.x * 16) + lane;
    const double* v0 = reinterpret_cast<const double*>(pb.V) + c0;
    const double* g0 = reinterpret_cast<const double*>(pb.G) + c0;
    size_t gs = 2 * (size_t)P;
    if (p == 0) {  // the columns of mode 0 hold W and U instead of omega_y
      g0 = (r == 0 ? pb.WM : pb.UM) + (size_t)b * ny;
      gs = 1;
    }
    constexpr int KC = KL <= 12 ? KL : (KL + (KL + 11) / 12 - 1) / ((KL + 11) / 12);  // at most 12 at a time
    for (int k0 = 0; k0 < KL; k0 += KC) {
      double d[KC];
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        const int n = threadIdx.x / 32 + 2 * NF * (k0 + k);
        d[k] = 0.0;
        if (p < P && n < 2 * ny) d[k] = n < ny ? v0[(size_t)n * 2 * P] : g0[(size_t)(n - ny) * gs];
      }
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        const int n = threadIdx.x / 32 + 2 * NF * (k0 + k);
        if (n < 2 * ny) tile[n * 32 + lane] = (RN)d[k];
      }
    }
    __syncthreads();
  }
  RN x[H + 1];
  if (p < P) {
    const int row = p / g.nxh, ix = p % g.nxh;
    const bool mean = p == 0, gen = !mean && row != g.nz / 2;
    const RN kx = (RN)t.kx[ix], kz = (RN)t.kz[row];
    const RN sg = r == 0 ? (RN)-1.0 : (RN)1.0;
    const RN ik2 = gen ? sg / (kx * kx + kz * kz) : (RN)0;
    const bool own = f == 1 || f == 4, deriv = f == 3 || f == 5;
    const size_t col = 2 * ((size_t)b * ny * P + p);  // component 0 of coefficient 0; 2 P per coefficient
    const double* Vp = reinterpret_cast<const double*>(pb.V) + col + (1 - r);
    const double* Sp;
    size_t ss = 2 * (size_t)P;
    RN cD = 0, cS = 1, cV = 0;
    if (own) {
      Sp = reinterpret_cast<const double*>(f == 1 ? pb.V : pb.G) + col + r;
    } else if (mean) {
      Sp = (f == 0 || f == 5 ? pb.UM : pb.WM) + (size_t)b * ny;
      ss = 1;
      if (f == 5) cS = (RN)-1.0;
    } else {
      Sp = reinterpret_cast<const double*>(pb.G) + col + (1 - r);
      if (f == 0) { cD = ik2 * kx; cS = -ik2 * kz; }
      if (f == 2) { cD = ik2 * kz; cS = ik2 * kx; }
      if (f == 3) { cD = ik2 * kz; cS = ik2 * kx; cV = -sg * kz; }
      if (f == 5) { cD = -ik2 * kx; cS = ik2 * kz; cV = sg * kx; }
    }
    const bool liveS = gen || (mean && !own && r == 0);
    const RN* Vt = tile + (lane ^ 1);
    const RN* St = tile + (f == 1 ? 0 : ny * 32) + (own ? lane : !mean ? lane ^ 1 : f == 0 || f == 5 ? 1 : 0);
    auto V = [&](int n) { return !gen ? (RN)0 : kTile ? Vt[n * 32] : (RN)Vp[(size_t)n * ss]; };
    auto S = [&](int n) { return !liveS ? (RN)0 : kTile ? St[n * 32] : (RN)Sp[(size_t)n * ss]; };
    // coefficients of one parity, n = 2 i + par, from the top down
    auto coefs = [&](int par, int count) {
      if (own) {
#pragma unroll
        for (int i = count - 1; i >= 0; --i) x[i] = S(2 * i + par);
      } else if (!deriv) {
        RN dv = 0;
#pragma unroll
        for (int i = count - 1; i >= 0; --i) {
          const int n = 2 * i + par;
          if (n + 1 <= N) dv = dv + (RN)(2 * (n + 1)) * V(n + 1);
          const RN d = n == 0 ? (RN)0.5 * dv : dv;
          x[i] = cD * d + cS * S(n);
        }
      } else {
        RN dv = 0, d2 = 0, ds = 0;
#pragma unroll
        for (int i = count - 1; i >= 0; --i) {
          const int n = 2 * i + par, m = n + 1;
          if (m <= N) {
            if (m + 1 <= N) dv = dv + (RN)(2 * (m + 1)) * V(m + 1);
            d2 = d2 + (RN)(2 * m) * dv;
            ds = ds + (RN)(2 * m) * S(m);
          }
          const RN h = n == 0 ? (RN)0.5 : (RN)1.0;
          x[i] = (cD * d2 + cS * ds) * h + cV * V(n);
        }
      }
    };
    if (half == 0) coefs(0, H + 1);
    else coefs(1, H);
  }
  if constexpr (kTile) __syncthreads();
  if (half == 0) {
    dct1<H, RN>(x);
#pragma unroll
    for (int j = 0; j <= H; ++j) part[j * 32 + lane] = x[j];
  } else {
    RN o[H];
#pragma unroll
    for (int j = 0; j < H; ++j) o[j] = x[j];
    dct2<H, RN>(o);
#pragma unroll
    for (int j = 0; j < H; ++j) part[(H + 1 + j) * 32 + lane] = o[j];
  }
  __syncthreads();
  if (p >= P) return;
  RN* dst = reinterpret_cast<RN*>(q) + 2 * (((size_t)b * 6 + f) * ny * P + p) + r;
  const size_t qs = 2 * (size_t)P;
#pragma unroll 16
  for (int j = half; j < H; j += 2) {
    const RN e = part[j * 32 + lane], o = part[(H + 1 + j) * 32 + lane];
    dst[(size_t)j * qs] = e + o;
    dst[(size_t)(N - j) * qs] = e - o;
  }
  if (half == 0) dst[(size_t)H * qs] = part[H * 32 + lane];
}

// a_n = 2/(N cb_n) sum_j f_j cos(pi n j / N) / cb_j (cb_0 = cb_N = 2): even n
// from f_j + f_{N-j}, odd n from f_j - f_{N-j}.  Both warps of a line have read
// their columns before either writes coefficients over them.
template <typename RN, int N, int NF>
__global__ void __launch_bounds__(64 * NF, ctas_of(analysis_dct_regs<RN, N>(), 64 * NF)) analysis_dct_kernel(Grid g, PencilBufs pb,
                                                                    typename cpx<RN>::T* __restrict__ hn) {
  constexpr int H = N / 2;
  const int P = g.P, ny = N + 1;
  const int lane = threadIdx.x & 31, half = (threadIdx.x / 32) & 1, f = blockIdx.z * NF + threadIdx.x / 64;
  const int p = blockIdx.x * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  pdl_wait_then_release();  // H comes from the nonlinear term
  RN* col = reinterpret_cast<RN*>(hn) + 2 * (((size_t)b * 3 + f) * ny * P + min(p, P - 1)) + r;
  const size_t hs = 2 * (size_t)P;
  const RN s0 = (RN)2.0 / (RN)N;
  RN x[H + 1];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const RN a = col[(size_t)j * hs], c = col[(size_t)(N - j) * hs];
    x[j] = half == 0 ? a + c : a - c;
  }
  x[0] = (RN)0.5 * x[0];
  x[H] = col[(size_t)H * hs];
  __syncthreads();
  if (p >= P) return;
  if (half == 0) {
    dct1<H, RN>(x);
#pragma unroll
    for (int i = 0; i <= H; ++i) col[(size_t)(2 * i) * hs] = ((i == 0 || i == H) ? (RN)0.5 * s0 : s0) * x[i];
  } else {
    RN o[H];
#pragma unroll
    for (int i = 0; i < H; ++i) o[i] = x[i];
    dct3<H, RN>(o);
#pragma unroll
    for (int i = 0; i < H; ++i) col[(size_t)(2 * i + 1) * hs] = s0 * o[i];
  }
}

// FP32 lines: all fields of a mode tile in one CTA, so that v and omega_y
// are shared through L1; FP64 lines: one field per
// CTA, which evens the FP64 work out over the SMs.
template <typename RN, int N>
cudaError_t pre_dct_n(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q, cudaStream_t st) {
  constexpr int NF = dct_fields<RN>(6);
  constexpr size_t smem = (size_t)NF * (N + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_dct_kernel<RN, N, NF>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_pre_dct_kernel<RN, N, NF>, dim3((g.P + 15) / 16, B, 6 / NF), dim3(64 * NF),
                                        smem, st, g, pb, t, q);
}
template <typename RN, int N>
cudaError_t analysis_dct_n(const Grid& g, int B, const PencilBufs& pb, typename cpx<RN>::T* h, cudaStream_t st) {
  return launch_pdl_if<sizeof(RN) == 4>(analysis_dct_kernel<RN, N, 1>, dim3((g.P + 15) / 16, B, 3), dim3(64), 0, st, g, pb, h);
}

}  // namespace chdns

#define CH_DCT_INSTANTIATE(RN, N)                                                                                  \
  namespace chdns {                                                                                                \
  template cudaError_t pre_dct_n<RN, N>(const Grid&, int, const PencilBufs&, const DevTables&, typename cpx<RN>::T*, \
                                        cudaStream_t);                                                             \
  template cudaError_t analysis_dct_n<RN, N>(const Grid&, int, const PencilBufs&, typename cpx<RN>::T*,             \
                                             cudaStream_t);                                                        \
  }
