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
// the instruction cache wherever an SM ran several of them.
//
// CTA: NF fields of one tile, two warps (even, odd) each.  FP32 lines of up to
// 65 nodes: all six, which share v and omega_y, rounded once into shared memory
// (a conversion instruction occupies the FP64 pipe as an FP64 operation does);
// longer and FP64 lines: one, reading its columns in place.
// ---------------------------------------------------------------------------
template <typename RN, int N> constexpr int pre_fields() { return sizeof(RN) == 4 && N <= 64 ? 6 : 1; }
constexpr int ctas_of(int regs, int threads) { return 65536 / (regs * threads) > 0 ? 65536 / (regs * threads) : 1; }
// registers a thread is held to: one parity's array and the transform around it
template <typename RN, int N> constexpr int dct_regs() {
  return sizeof(RN) == 8 ? (N <= 32 ? 96 : N <= 64 ? 168 : 255) : (N <= 32 ? 56 : N <= 64 ? 80 : N <= 96 ? 96 : N <= 128 ? 128 : 168);
}

template <typename RN, int N, int NF>
__global__ void __launch_bounds__(64 * NF, ctas_of(dct_regs<RN, N>(), 64 * NF)) stage_pre_dct_kernel(Grid g, PencilBufs pb,
                                                                DevTables t, typename cpx<RN>::T* __restrict__ q) {
  constexpr int H = N / 2, ny = N + 1;
  constexpr bool kTile = NF > 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P;
  const int lane = threadIdx.x & 31, fl = threadIdx.x / 64, half = (threadIdx.x / 32) & 1, f = blockIdx.x % (6 / NF) * NF + fl;
  RN* part = reinterpret_cast<RN*>(smem_raw) + fl * ny * 32;        // [E_0 .. E_H, O_0 .. O_{H-1}][32]
  RN* tile = reinterpret_cast<RN*>(smem_raw) + NF * ny * 32;        // [v, omega_y][ny][32]
  const int p0 = (int)blockIdx.x / (6 / NF) * 16, p = p0 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  pdl_wait_then_release();  // v, omega_y come from the previous stage
  if constexpr (kTile) {
    // a column per warp and step, every load in flight before the first store
    constexpr int KL = (2 * ny + 2 * NF - 1) / (2 * NF);
    const size_t c0 = 2 * ((size_t)b * ny * P + p0) + lane;
    const double* v0 = reinterpret_cast<const double*>(pb.V) + c0;
    const double* g0 = reinterpret_cast<const double*>(pb.G) + c0;
    size_t gs = 2 * (size_t)P;
    if (p == 0) {  // the columns of mode 0 hold W and U instead of omega_y
      g0 = (r == 0 ? pb.WM : pb.UM) + (size_t)b * ny;
      gs = 1;
    }
    double d[KL];
#pragma unroll
    for (int k = 0; k < KL; ++k) {
      const int n = threadIdx.x / 32 + 2 * NF * k;
      d[k] = 0.0;
      if (p < P && n < 2 * ny) d[k] = n < ny ? v0[(size_t)n * 2 * P] : g0[(size_t)(n - ny) * gs];
    }
#pragma unroll
    for (int k = 0; k < KL; ++k) {
      const int n = threadIdx.x / 32 + 2 * NF * k;
      if (n < 2 * ny) tile[n * 32 + lane] = (RN)d[k];
    }
    __syncthreads();
  }
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
    const bool liveS = gen || (mean && !own && r == 0);
    const size_t col = 2 * ((size_t)b * ny * P + p);  // component 0 of coefficient 0; 2 P per coefficient
    const double* Vp = reinterpret_cast<const double*>(pb.V) + col + (1 - r);
    const double* Sp = reinterpret_cast<const double*>(f == 1 ? pb.V : pb.G) + col + (own ? r : 1 - r);
    const size_t vs = 2 * (size_t)P;
    size_t ss = vs;
    if (mean && !own) {
      Sp = (f == 0 || f == 5 ? pb.UM : pb.WM) + (size_t)b * ny;
      ss = 1;
    }
    const RN* Vt = tile + (lane ^ 1);
    const RN* St = tile + (f == 1 ? 0 : ny * 32) + (own ? lane : !mean ? lane ^ 1 : f == 0 || f == 5 ? 1 : 0);
    auto V = [&](int n) { return !gen ? (RN)0 : kTile ? Vt[n * 32] : to_rn<RN>(__ldg(Vp + n * vs)); };
    auto S = [&](int n) { return !liveS ? (RN)0 : kTile ? St[n * 32] : to_rn<RN>(__ldg(Sp + n * ss)); };
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
      mine[top * 32] = cD * d2 + cS * ds + cV * V(2 * top + half);
#pragma unroll 4
      for (int i = top - 1; i >= 1; --i) {
        const int m = 2 * i + half + 1;
        dv = dv + c2(m + 1) * V(m + 1);
        d2 = d2 + c2(m) * dv;
        ds = ds + c2(m) * S(m);
        mine[i * 32] = cD * d2 + cS * ds + cV * V(m - 1);
      }
      const int m = half + 1;
      dv = dv + c2(m + 1) * V(m + 1);
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
  RN* dst = reinterpret_cast<RN*>(q) + 2 * (((size_t)b * 6 + f) * ny * P + p) + r;
  const size_t qs = 2 * (size_t)P;
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
  constexpr int H = N / 2, ny = N + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P;
  const int lane = threadIdx.x & 31, half = threadIdx.x / 32, f = blockIdx.z;
  const int p = blockIdx.x * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  pdl_wait_then_release();  // H comes from the nonlinear term
  RN* col = reinterpret_cast<RN*>(hn) + 2 * (((size_t)b * 3 + f) * ny * P + min(p, P - 1)) + r;
  RN* sm = reinterpret_cast<RN*>(smem_raw) + lane;
  const size_t hs = 2 * (size_t)P;
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
  constexpr int NF = pre_fields<RN, N>();
  constexpr size_t smem = (size_t)(NF + (NF > 1 ? 2 : 0)) * (N + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_dct_kernel<RN, N, NF>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_pre_dct_kernel<RN, N, NF>, dim3((g.P + 15) / 16 * (6 / NF), B), dim3(64 * NF),
                                        smem, st, g, pb, t, q);
}
template <typename RN, int N>
cudaError_t analysis_dct_n(const Grid& g, int B, const PencilBufs& pb, typename cpx<RN>::T* h, cudaStream_t st) {
  constexpr size_t smem = (size_t)(N + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(analysis_dct_kernel<RN, N>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(analysis_dct_kernel<RN, N>, dim3((g.P + 15) / 16, B, 3), dim3(64), smem, st, g, pb, h);
}

}  // namespace chdns

#define CH_DCT_INSTANTIATE(RN, N)                                                                                  \
  namespace chdns {                                                                                                \
  template cudaError_t pre_dct_n<RN, N>(const Grid&, int, const PencilBufs&, const DevTables&, typename cpx<RN>::T*, \
                                        cudaStream_t);                                                             \
  template cudaError_t analysis_dct_n<RN, N>(const Grid&, int, const PencilBufs&, typename cpx<RN>::T*,             \
                                             cudaStream_t);                                                        \
  }
