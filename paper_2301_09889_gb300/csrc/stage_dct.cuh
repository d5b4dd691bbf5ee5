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
//
// The coefficients of a parity are formed by rolled loops into the thread's
// column of the exchange buffer and then read into registers: with the loops
// unrolled, the kernel's paths (three kinds of field, two parities) outgrew
// the instruction cache wherever an SM ran several of them (FP32, 256x193x256:
// 232 us by sixteen rows, 176 by eight, 180 by four).
//
// CTA: one field of a tile, two warps; the fields of a tile are neighbouring
// CTAs.  FP32 lines read the copies of v and omega_y that the implicit half
// rounded to FP32: a conversion instruction occupies the FP64 pipe as an FP64
// operation does, and the lines read every column four to five times.
// ---------------------------------------------------------------------------
constexpr int ctas_of(int regs, int threads) { return 65536 / (regs * threads) > 0 ? 65536 / (regs * threads) : 1; }
// registers a thread is held to: one parity's array and the transform around it
template <typename RN, int N> constexpr int dct_regs() {
  return sizeof(RN) == 8 ? (N <= 32 ? 96 : N <= 64 ? 168 : 255) : (N <= 32 ? 56 : N <= 64 ? 80 : N <= 96 ? 96 : N <= 128 ? 128 : 168);
}

template <typename RN, int N>
__global__ void __launch_bounds__(64, ctas_of(dct_regs<RN, N>(), 64)) stage_pre_dct_kernel(Grid g, PencilBufs pb, DevTables t,
                                                                typename cpx<RN>::T* __restrict__ q) {
  constexpr int H = N / 2, ny = N + 1;
  constexpr bool kF32 = sizeof(RN) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RN* part = reinterpret_cast<RN*>(smem_raw);  // [E_0 .. E_H, O_0 .. O_{H-1}][32]
  const int P = g.P;
  const int lane = threadIdx.x & 31, half = threadIdx.x / 32, f = blockIdx.x % 6;
  const int p = (int)blockIdx.x / 6 * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  RN* mine = part + half * (H + 1) * 32 + lane;
  if (p < P) {
    const int row = p / g.nxh, ix = p % g.nxh;
    const bool mean = p == 0, gen = !mean && row != g.nz / 2;
    const bool own = f == 1 || f == 4, deriv = f == 3 || f == 5;
    const RN kx = (RN)t.kx[ix], kz = (RN)t.kz[row];
    const RN sg = r == 0 ? (RN)-1.0 : (RN)1.0;
    const RN ik2 = gen ? sg / (kx * kx + kz * kz) : (RN)0;
    RN cD = 0, cS = 1, cV = 0;
    if (gen && !own) {
      if (f == 0) { cD = ik2 * kx; cS = -ik2 * kz; }
      if (f == 2) { cD = ik2 * kz; cS = ik2 * kx; }
      if (f == 3) { cD = ik2 * kz; cS = ik2 * kx; cV = -sg * kz; }
      if (f == 5) { cD = -ik2 * kx; cS = ik2 * kz; cV = sg * kx; }
    } else if (mean && f == 5) {
      cS = (RN)-1.0;
    }
    const bool liveM = mean && !own && r == 0;  // the columns of the mean flow
    const size_t col = 2 * ((size_t)b * ny * P + p);  // component 0 of coefficient 0; 2 P per coefficient
    const RN* v0 = reinterpret_cast<const RN*>(kF32 ? (const void*)pb.V32 : pb.V) + col;
    const RN* g0 = reinterpret_cast<const RN*>(kF32 ? (const void*)pb.G32 : pb.G) + col;
    const RN* Vp = v0 + (1 - r);
    const RN* Sp = (f == 1 ? v0 : g0) + (own ? r : 1 - r);
    const size_t vs = 2 * (size_t)P;
    size_t ss = vs;
    if (liveM) {
      // the mean flow: its own columns, or the FP32 copies in mode 0's: (W, U),
      // and (DW, DU), which the implicit half sums in FP64 (an FP32 sum loses up to
      // N / 2 roundings of the mean shear)
      if constexpr (kF32) {
        Sp = g0 + (f == 0 ? 1 : 0);
        if (deriv) {
          Vp = v0 + (f == 5 ? 1 : 0);
          cS = 0;
          cV = f == 5 ? (RN)-1.0 : (RN)1.0;
        }
      } else {
        Sp = (f == 0 || f == 5 ? pb.UM : pb.WM) + (size_t)b * ny;
        ss = 1;
      }
    }
    const bool liveV = gen || (kF32 && liveM && deriv), liveS = gen || (liveM && !(kF32 && deriv));
    // every load is unconditional (the loops batch them), dead lanes drop theirs
    auto V = [&](int n) { const RN x = __ldg(Vp + n * vs); return liveV ? x : (RN)0; };
    auto S = [&](int n) { const RN x = __ldg(Sp + n * ss); return liveS ? x : (RN)0; };
    // 2 k; from a table in FP64, where converting it would cost an operation
    auto c2 = [&](int k) {
      if constexpr (sizeof(RN) == 8) return __ldg(t.tau.n1 + k - 1);
      else return (RN)(2 * k);
    };
    // coefficients of this warp's parity, n = 2 i + half, from the top down
    const int top = half == 0 ? H : H - 1;
    if (own) {
#pragma unroll 8
      for (int i = top; i >= 0; --i) mine[i * 32] = S(2 * i + half);
    } else if (!deriv) {
      RN dv = half == 0 ? (RN)0 : (RN)(2 * N) * V(N);
      mine[top * 32] = cD * dv + cS * S(2 * top + half);
#pragma unroll 8
      for (int i = top - 1; i >= 1; --i) {
        const int n = 2 * i + half;
        dv = dv + c2(n + 1) * V(n + 1);
        mine[i * 32] = cD * dv + cS * S(n);
      }
      dv = dv + c2(half + 1) * V(half + 1);
      mine[0] = cD * (half == 0 ? (RN)0.5 * dv : dv) + cS * S(half);
    } else {
      // the step at i adds m = 2 i + half + 1 to D^2 v and DS and m + 1 to Dv
      RN dv = 0, d2 = 0, ds = 0;
      if (half == 1) {
        d2 = (RN)0;
        ds = (RN)(2 * N) * S(N);
      }
      RN vn = V(2 * top + half);
      mine[top * 32] = cD * d2 + cS * ds + cV * vn;
#pragma unroll 8
      for (int i = top - 1; i >= 1; --i) {
        const int m = 2 * i + half + 1;
        dv = dv + c2(m + 1) * vn;
        d2 = d2 + c2(m) * dv;
        ds = ds + c2(m) * S(m);
        vn = V(m - 1);
        mine[i * 32] = cD * d2 + cS * ds + cV * vn;
      }
      const int m = half + 1;
      dv = dv + c2(m + 1) * vn;
      d2 = d2 + c2(m) * dv;
      ds = ds + c2(m) * S(m);
      mine[0] = (cD * d2 + cS * ds) * (half == 0 ? (RN)0.5 : (RN)1.0) + cV * V(half);
    }
  }
  if (half == 0) {
    RN x[H + 1];
#pragma unroll
    for (int j = 0; j <= H; ++j) x[j] = mine[j * 32];
    dct1<H, RN>(x);
#pragma unroll
    for (int j = 0; j <= H; ++j) mine[j * 32] = x[j];
  } else {
    RN x[H];
#pragma unroll
    for (int j = 0; j < H; ++j) x[j] = mine[j * 32];
    dct2<H, RN>(x);
#pragma unroll
    for (int j = 0; j < H; ++j) mine[j * 32] = x[j];
  }
  __syncthreads();
  if (p >= P) return;
  RN* dst = reinterpret_cast<RN*>(q) + 2 * (b * g.qb + f * g.qf + p) + r;
  const size_t qs = 2 * g.qj;
#pragma unroll 8
  for (int j = half; j < H; j += 2) {
    const RN e = part[j * 32 + lane], o = part[(H + 1 + j) * 32 + lane];
    dst[(size_t)j * qs] = e + o;
    dst[(size_t)(N - j) * qs] = e - o;
  }
  if (half == 0) dst[(size_t)H * qs] = part[H * 32 + lane];
}

// a_n = 2/(N cb_n) sum_j f_j cos(pi n j / N) / cb_j (cb_0 = cb_N = 2): even n
// from f_j + f_{N-j}, odd n from f_j - f_{N-j}.  The columns are staged in
// shared memory, so both warps have all nodes before either writes
// coefficients over them.
template <typename RN, int N>
__global__ void __launch_bounds__(64, ctas_of(dct_regs<RN, N>(), 64)) analysis_dct_kernel(Grid g, PencilBufs pb,
                                                                    typename cpx<RN>::T* __restrict__ hn) {
  constexpr int H = N / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P;
  const int lane = threadIdx.x & 31, half = threadIdx.x / 32, f = blockIdx.z;
  const int p = blockIdx.x * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  RN* col = reinterpret_cast<RN*>(hn) + 2 * (b * g.qb + f * g.qf + min(p, P - 1)) + r;
  RN* sm = reinterpret_cast<RN*>(smem_raw) + lane;
  const size_t hs = 2 * g.qj;
#pragma unroll 16
  for (int j = half; j <= N; j += 2) sm[j * 32] = col[(size_t)j * hs];
  __syncthreads();
  const RN s0 = (RN)2.0 / (RN)N;
  if (half == 0) {
    RN x[H + 1];
#pragma unroll
    for (int j = 0; j < H; ++j) x[j] = sm[j * 32] + sm[(N - j) * 32];
    x[0] = (RN)0.5 * x[0];
    x[H] = sm[H * 32];
    dct1<H, RN>(x);
    if (p >= P) return;
#pragma unroll
    for (int i = 0; i <= H; ++i) col[(size_t)(2 * i) * hs] = ((i == 0 || i == H) ? (RN)0.5 * s0 : s0) * x[i];
  } else {
    RN x[H];
#pragma unroll
    for (int j = 0; j < H; ++j) x[j] = sm[j * 32] - sm[(N - j) * 32];
    x[0] = (RN)0.5 * x[0];
    dct3<H, RN>(x);
    if (p >= P) return;
#pragma unroll
    for (int i = 0; i < H; ++i) col[(size_t)(2 * i + 1) * hs] = s0 * x[i];
  }
}

template <typename RN, int N>
cudaError_t pre_dct_n(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q, cudaStream_t st) {
  constexpr size_t smem = (size_t)(N + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_dct_kernel<RN, N>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(stage_pre_dct_kernel<RN, N>, dim3((g.P + 15) / 16 * 6, B), dim3(64), smem, st, g, pb,
                                        t, q);
}
template <typename RN, int N>
cudaError_t analysis_dct_n(const Grid& g, int B, const PencilBufs& pb, typename cpx<RN>::T* h, cudaStream_t st) {
  constexpr size_t smem = (size_t)(N + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(analysis_dct_kernel<RN, N>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(analysis_dct_kernel<RN, N>, dim3((g.P + 15) / 16, B, 3), dim3(64), smem, st, g, pb, h);
}

}  // namespace chdns

#define CH_DCT_INSTANTIATE(RN, N)                                                                                  \
  namespace chdns {                                                                                                \
  template cudaError_t pre_dct_n<RN, N>(const Grid&, int, const PencilBufs&, const DevTables&, typename cpx<RN>::T*, \
                                        cudaStream_t);                                                             \
  template cudaError_t analysis_dct_n<RN, N>(const Grid&, int, const PencilBufs&, typename cpx<RN>::T*,             \
                                             cudaStream_t);                                                        \
  }
