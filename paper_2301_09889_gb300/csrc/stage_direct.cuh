// The explicit half of a stage and the Chebyshev analysis of H by direct sums,
// for the orders N without a register cosine transform (stage_dct.cuh): the
// same lines and layouts, N at run time.
//
// Lanes hold 16 modes x 2 components of one field; the values a CTA sums over
// stand in shared memory, [n][32], and every warp forms K outputs of each line.
// A value it loads feeds K accumulators, whose factors cos(pi j n / N) are the
// same for all lanes: eight, as vectors from padded tables, in FP32; five to
// eight, whichever leaves the fewest idle sums in the last warp, in FP64 (25
// node pairs take four warps of seven, not of eight).  Node pairs j, N - j
// share their even and odd sums.
//
// What bounds it: FP64 lines by the FP64 pipe ((N/2)(N+1) operations per line,
// every lane at work; a warp per mode group took 853 us for the analysis of
// 128x148x16, a few warps per SM each on their own); FP32 lines by issue (11
// instructions for eight sums).
#pragma once

#include "common.cuh"
#include "internal.h"

namespace chdns {

template <typename RN> __device__ __forceinline__ const RN* pre_table(const DevTables& t);
template <> __device__ __forceinline__ const double* pre_table<double>(const DevTables& t) { return t.cos_pre; }
template <> __device__ __forceinline__ const float* pre_table<float>(const DevTables& t) { return t.cos_pre_f; }
template <typename RN> __device__ __forceinline__ const RN* ana_table(const DevTables& t);
template <> __device__ __forceinline__ const double* ana_table<double>(const DevTables& t) { return t.cos_ana; }
template <> __device__ __forceinline__ const float* ana_table<float>(const DevTables& t) { return t.cos_ana_f; }

// K consecutive table values (FP32: eight, 32-byte aligned)
__device__ __forceinline__ void load_k(const float* p, float (&c)[8]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  c[0] = a.x; c[1] = a.y; c[2] = a.z; c[3] = a.w;
  c[4] = b.x; c[5] = b.y; c[6] = b.z; c[7] = b.w;
}
template <int K>
__device__ __forceinline__ void load_k(const double* p, double (&c)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) c[k] = __ldg(p + k);
}

// Field f of 16 modes at node pairs; the fields' coefficients as in
// stage_pre_dct (stage_dct.cuh).  grid (6 tiles, B, groups of K W pairs)
template <typename RN, int K>
__global__ void __launch_bounds__(192) stage_pre_direct_kernel(Grid g, PencilBufs pb, DevTables t,
                                                               typename cpx<RN>::T* __restrict__ q) {
  constexpr bool kF32 = sizeof(RN) == 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RN* co = reinterpret_cast<RN*>(smem_raw);  // [ny][32]
  const int P = g.P, N = g.N, ny = g.ny, J = N / 2 + 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32, nw = blockDim.x / 32, f = blockIdx.x % 6;
  const int p = (int)blockIdx.x / 6 * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
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
    const bool liveM = mean && !own && r == 0;
    const bool liveV = gen || (kF32 && liveM && deriv), liveS = gen || (liveM && !(kF32 && deriv));
    const size_t col = 2 * ((size_t)b * ny * P + p), vs = 2 * (size_t)P;
    const RN* v0 = reinterpret_cast<const RN*>(kF32 ? (const void*)pb.V32 : pb.V) + col;
    const RN* g0 = reinterpret_cast<const RN*>(kF32 ? (const void*)pb.G32 : pb.G) + col;
    const RN* Vp = v0 + (1 - r);
    const RN* Sp = (f == 1 ? v0 : g0) + (own ? r : 1 - r);
    size_t ss = vs;
    if (liveM) {
      if constexpr (kF32) {
        // the FP32 copies in mode 0's columns: (W, U) and (DW, DU)
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
    auto V = [&](int n) { const RN x = __ldg(Vp + n * vs); return liveV ? x : (RN)0; };
    auto S = [&](int n) { const RN x = __ldg(Sp + n * ss); return liveS ? x : (RN)0; };
    auto c2 = [&](int k) {  // 2 k
      if constexpr (sizeof(RN) == 8) return __ldg(t.tau.n1 + k - 1);
      else return (RN)(2 * k);
    };
    for (int par = warp; par < 2; par += nw) {
      RN* mine = co + par * 32 + lane;  // n = 2 i + par at mine[64 i]
      const int top = (N - par) / 2, nt = 2 * top + par;
      if (own) {
#pragma unroll 8
        for (int i = top; i >= 0; --i) mine[64 * i] = S(2 * i + par);
      } else if (!deriv) {
        RN dv = nt < N ? c2(N) * V(N) : (RN)0;
        mine[64 * top] = cD * dv + cS * S(nt);
#pragma unroll 8
        for (int i = top - 1; i >= 1; --i) {
          const int n = 2 * i + par;
          dv = dv + c2(n + 1) * V(n + 1);
          mine[64 * i] = cD * dv + cS * S(n);
        }
        dv = dv + c2(par + 1) * V(par + 1);
        mine[0] = cD * (par == 0 ? (RN)0.5 * dv : dv) + cS * S(par);
      } else {
        RN dv = 0, d2 = 0, ds = nt < N ? c2(N) * S(N) : (RN)0;
        RN vn = V(nt);
        mine[64 * top] = cS * ds + cV * vn;
#pragma unroll 8
        for (int i = top - 1; i >= 1; --i) {
          const int m = 2 * i + par + 1;
          dv = dv + c2(m + 1) * vn;
          d2 = d2 + c2(m) * dv;
          ds = ds + c2(m) * S(m);
          vn = V(m - 1);
          mine[64 * i] = cD * d2 + cS * ds + cV * vn;
        }
        const int m = par + 1;
        dv = dv + c2(m + 1) * vn;
        d2 = d2 + c2(m) * dv;
        ds = ds + c2(m) * S(m);
        mine[0] = (cD * d2 + cS * ds) * (par == 0 ? (RN)0.5 : (RN)1.0) + cV * V(par);
      }
    }
  }
  __syncthreads();
  const int j0 = (blockIdx.z * nw + warp) * K;
  if (p >= P || j0 >= J) return;
  const int Jp = (J + 15) / 8 * 8;
  const RN* tab = pre_table<RN>(t) + j0;  // cos(pi j n / N) at tab[n Jp + j - j0]
  RN E[K] = {}, O[K] = {};
  if constexpr (kF32) {
    // from the highest coefficient down, the small terms first: summed upwards
    // every term rounds at the size of the lowest ones (mixed 16x148x16: omega_y
    // 2.5e-7 off after five steps, 1.6e-7 so)
    const RN* tp = tab + (size_t)N * Jp;
    const RN* cp = co + N * 32 + lane;
    if ((N & 1) == 0) {
      RN c[K];
      load_k(tp, c);
      const RN x = *cp;
#pragma unroll
      for (int k = 0; k < K; ++k) E[k] = c[k] * x;
      tp -= Jp;
      cp -= 32;
    }
#pragma unroll 1
    for (int i = (N + 1) / 2; i > 0; --i) {
      RN c[K], d[K];
      load_k(tp - Jp, c);
      load_k(tp, d);
      const RN x = cp[-32], y = *cp;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        E[k] = E[k] + c[k] * x;
        O[k] = O[k] + d[k] * y;
      }
      tp -= 2 * Jp;
      cp -= 64;
    }
  } else {
    int n = 0;
#pragma unroll 2
    for (; n + 1 <= N; n += 2) {
      RN c[K], d[K];
      load_k(tab + (size_t)n * Jp, c);
      load_k(tab + (size_t)(n + 1) * Jp, d);
      const RN x = co[n * 32 + lane], y = co[(n + 1) * 32 + lane];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        E[k] = E[k] + c[k] * x;
        O[k] = O[k] + d[k] * y;
      }
    }
    if (n == N) {
      RN c[K];
      load_k(tab + (size_t)n * Jp, c);
      const RN x = co[n * 32 + lane];
#pragma unroll
      for (int k = 0; k < K; ++k) E[k] = E[k] + c[k] * x;
    }
  }
  RN* dst = reinterpret_cast<RN*>(q) + 2 * (b * g.qb + f * g.qf + p) + r;
  const size_t qs = 2 * g.qj;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int j = j0 + k;
    if (2 * j < N) {
      dst[(size_t)j * qs] = E[k] + O[k];
      dst[(size_t)(N - j) * qs] = E[k] - O[k];
    } else if (2 * j == N) {
      dst[(size_t)j * qs] = E[k];  // the odd cosines vanish at the middle node
    }
  }
}

// The explicit half of handles with so few modes that a transform per line
// leaves most SMs idle (FP64; an operation holds its sub-partition 64 cycles, so
// one warp's line is a chain of its operations; 28 us per launch of 128 modes
// at N = 64, 21 here).  A CTA forms 12 node pairs of a field of 16 modes.
// Everything it reads arrives in one round of loads; the recurrences of the
// derivatives run on four warps (parity x the terms of d2 v or D v, and of the
// others), every CTA its own copy; then each warp sums two node pairs.
// grid (6 tiles, B, groups of 12 pairs)
constexpr int kFewWarps = 6, kFewPairs = 2 * kFewWarps;
__global__ void __launch_bounds__(32 * kFewWarps) stage_pre_few_kernel(Grid g, PencilBufs pb, DevTables t,
                                                                       double2* __restrict__ q) {
  constexpr int K = 2, KC = kFewPairs;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P, N = g.N, ny = g.ny, J = N / 2 + 1, Jp = (J + 15) / 8 * 8;
  double* co = reinterpret_cast<double*>(smem_raw);  // [ny][32] coefficients of the field
  double* sv = co + 32 * ny;                         // [ny][32] v
  double* so = sv + 32 * ny;                         // [ny][32] omega_y, the mean flow, or the field itself
  double* pd = so + 32 * ny;                         // [ny][32] terms of d2 v or D v
  double* tb = pd + 32 * ny;                         // [ny][KC] cos(pi j n / N) of the CTA's pairs
  double* c2 = tb + KC * ny;                         // [ny] 2 (n + 1)
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32, f = blockIdx.x % 6;
  const int p = (int)blockIdx.x / 6 * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y, jc = blockIdx.z * KC;
  if (pb.active && !pb.active[b]) return;
  const int pc = min(p, P - 1), row = pc / g.nxh, ix = pc % g.nxh;
  const bool mean = p == 0, gen = p > 0 && p < P && row != g.nz / 2;
  const bool own = f == 1 || f == 4, deriv = f == 3 || f == 5;
  const double kx = t.kx[ix], kz = t.kz[row];
  const double sg = r == 0 ? -1.0 : 1.0;
  const double ik2 = gen ? sg / (kx * kx + kz * kz) : 0.0;
  double cD = 0.0, cS = 1.0, cV = 0.0;
  if (gen && !own) {
    if (f == 0) { cD = ik2 * kx; cS = -ik2 * kz; }
    if (f == 2) { cD = ik2 * kz; cS = ik2 * kx; }
    if (f == 3) { cD = ik2 * kz; cS = ik2 * kx; cV = -sg * kz; }
    if (f == 5) { cD = -ik2 * kx; cS = ik2 * kz; cV = sg * kx; }
  } else if (mean && f == 5) {
    cS = -1.0;
  }
  {
    const bool liveM = mean && !own && r == 0, liveS = gen || liveM;
    const size_t col = 2 * ((size_t)b * ny * P + pc), vs = 2 * (size_t)P;
    const double* v0 = reinterpret_cast<const double*>(pb.V) + col;
    const double* Vp = v0 + (1 - r);
    const double* Sp = (f == 1 ? v0 : reinterpret_cast<const double*>(pb.G) + col) + (own ? r : 1 - r);
    size_t ss = vs;
    if (liveM) {
      Sp = (f == 0 || f == 5 ? pb.UM : pb.WM) + (size_t)b * ny;
      ss = 1;
    }
#pragma unroll 11
    for (int n = warp; n < ny; n += kFewWarps) {
      const double x = __ldg(Vp + n * vs), y = __ldg(Sp + n * ss);
      sv[n * 32 + lane] = gen ? x : 0.0;
      so[n * 32 + lane] = liveS ? y : 0.0;
    }
#pragma unroll 4
    for (int w = threadIdx.x; w < ny * KC; w += 32 * kFewWarps) {
      const int n = w / KC, j = jc + w % KC;
      tb[w] = j < J ? __ldg(t.cos_pre + (size_t)n * Jp + j) : 0.0;
    }
    for (int n = threadIdx.x; n < ny; n += 32 * kFewWarps) c2[n] = t.tau.n1[n];
  }
  __syncthreads();
  const double* src = own ? so : co;
  if (!own) {
    if (warp < 4) {
      const int par = warp & 1, top = (N - par) / 2;
      const double* V = sv + lane;
      const double* S = so + lane;
      auto two = [&](int k) { return c2[k - 1]; };  // 2 k
      if (warp < 2) {
        // cD D v, or cD D^2 v: the step at i adds m = 2 i + par + 1 (and m + 1 to D v)
        double* o = pd + par * 32 + lane;
        double dv = 0.0, d2 = 0.0;
        if (!deriv) {
          if (2 * top + par < N) dv = two(N) * V[32 * N];
          o[64 * top] = cD * dv;
#pragma unroll 4
          for (int i = top - 1; i >= 0; --i) {
            const int m = 2 * i + par + 1;
            dv = dv + two(m) * V[32 * m];
            o[64 * i] = (i == 0 && par == 0 ? 0.5 * cD : cD) * dv;
          }
        } else {
          o[64 * top] = 0.0;
#pragma unroll 4
          for (int i = top - 1; i >= 0; --i) {
            const int m = 2 * i + par + 1;
            dv = dv + two(m + 1) * V[32 * (m + 1)];
            d2 = d2 + two(m) * dv;
            o[64 * i] = (i == 0 && par == 0 ? 0.5 * cD : cD) * d2;
          }
        }
      } else {
        double* o = co + par * 32 + lane;
        if (!deriv) {
#pragma unroll 4
          for (int i = top; i >= 0; --i) o[64 * i] = cS * S[32 * (2 * i + par)];
        } else {
          double ds = 2 * top + par < N ? two(N) * S[32 * N] : 0.0;
          o[64 * top] = cS * ds + cV * V[32 * (2 * top + par)];
#pragma unroll 4
          for (int i = top - 1; i >= 0; --i) {
            const int m = 2 * i + par + 1;
            ds = ds + two(m) * S[32 * m];
            o[64 * i] = (i == 0 && par == 0 ? 0.5 * cS : cS) * ds + cV * V[32 * (m - 1)];
          }
        }
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int w = threadIdx.x; w < 32 * ny; w += 32 * kFewWarps) co[w] = co[w] + pd[w];
    __syncthreads();
  }
  const int j0 = jc + warp * K;
  if (p >= P || j0 >= J) return;
  double E[K] = {}, O[K] = {};
  const double* c = tb + warp * K;
  int n = 0;
#pragma unroll 4
  for (; n + 1 <= N; n += 2) {
    const double x = src[n * 32 + lane], y = src[(n + 1) * 32 + lane];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      E[k] = E[k] + c[n * KC + k] * x;
      O[k] = O[k] + c[(n + 1) * KC + k] * y;
    }
  }
  if (n == N) {
#pragma unroll
    for (int k = 0; k < K; ++k) E[k] = E[k] + c[n * KC + k] * src[n * 32 + lane];
  }
  double* dst = reinterpret_cast<double*>(q) + 2 * (b * g.qb + f * g.qf + p) + r;
  const size_t qs = 2 * g.qj;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int j = j0 + k;
    if (2 * j < N) {
      dst[(size_t)j * qs] = E[k] + O[k];
      dst[(size_t)(N - j) * qs] = E[k] - O[k];
    } else if (2 * j == N) {
      dst[(size_t)j * qs] = E[k];
    }
  }
}

// a_n = 2/(N cb_n) sum_j f_j cos(pi n j / N) / cb_j (cb_0 = cb_N = 2) of one
// parity of one field of 16 modes, from the nodal values hn to the coefficients
// hc (other fields of the array: the CTAs of a field share its nodes).
// grid (tiles, B, 3 fields x 2 parities x groups of 4 K)
constexpr int kAnaWarps = 4;
template <typename RN, int K>
__global__ void __launch_bounds__(32 * kAnaWarps) analysis_direct_kernel(Grid g, PencilBufs pb, DevTables t,
                                                                         const typename cpx<RN>::T* __restrict__ hn,
                                                                         typename cpx<RN>::T* __restrict__ hc, int Ip) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RN* sm = reinterpret_cast<RN*>(smem_raw);  // [N/2 + 1][32] folded nodes
  const int P = g.P, N = g.N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  const int f = blockIdx.z % 3, par = blockIdx.z / 3 % 2, i0 = (blockIdx.z / 6 * kAnaWarps + warp) * K;
  const int p = blockIdx.x * 16 + (lane >> 1), r = lane & 1;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  const size_t base = 2 * (b * g.qb + f * g.qf + min(p, P - 1)) + r, hs = 2 * g.qj;
  const RN* col = reinterpret_cast<const RN*>(hn) + base;
#pragma unroll 4
  for (int j = warp; 2 * j < N; j += kAnaWarps) {
    const RN a = __ldg(col + (size_t)j * hs), c = __ldg(col + (size_t)(N - j) * hs);
    const RN x = par == 0 ? a + c : a - c;
    sm[j * 32 + lane] = j == 0 ? (RN)0.5 * x : x;
  }
  if ((N & 1) == 0 && warp == 0) sm[(N / 2) * 32 + lane] = par == 0 ? __ldg(col + (size_t)(N / 2) * hs) : (RN)0;
  __syncthreads();
  const int I = (N - par) / 2 + 1;  // coefficients n = 2 i + par
  if (p >= P || i0 >= I) return;
  const RN* tab = ana_table<RN>(t) + (size_t)par * Ip + i0;  // cos(pi j n / N) at tab[2 Ip j + i - i0]
  RN a[K] = {};
#pragma unroll 4
  for (int j = 0; 2 * j <= N; ++j) {
    RN c[K];
    load_k(tab + (size_t)2 * Ip * j, c);
    const RN x = sm[j * 32 + lane];
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] = a[k] + c[k] * x;
  }
  RN* dst = reinterpret_cast<RN*>(hc) + base;
  const RN s0 = (RN)2.0 / (RN)N;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = i0 + k, n = 2 * i + par;
    if (i < I) dst[(size_t)n * hs] = ((n == 0 || n == N) ? (RN)0.5 * s0 : s0) * a[k];
  }
}

}  // namespace chdns
