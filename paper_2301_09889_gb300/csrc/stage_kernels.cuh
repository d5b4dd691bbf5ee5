// The two wall-normal halves of one Runge-Kutta stage, each fused over a tile
// of `ppc` Fourier modes that lives in shared memory:
//
//   stage_pre  : (v, omega_y, U, W) coefficients -> coefficients of
//                u, v, w, omega_x, omega_y, omega_z -> their values at the
//                Gauss-Lobatto nodes (input of the nonlinear plane kernel);
//   stage_post : nodal values of H = u x omega -> Chebyshev coefficients ->
//                right-hand sides -> Chebyshev-tau solves -> new state.
//
// Every global array is read and written once per stage with loads and
// stores that are contiguous over the modes of the tile; the sequential
// recurrences then run on shared memory.  RN is the precision of the nodal
// values exchanged with the plane kernel (double: all-FP64 path).
//
// Symmetry classes and components.  All wall-normal operators are real and
// map even Chebyshev coefficients to even or odd ones in a fixed pattern, so a
// mode splits into two classes (c = 0: even v, odd omega_y; c = 1: odd v,
// even omega_y) and two real components (r = 0, 1) that never interact.  The
// factors i kx, i kz only swap components: component r of (i s X) is
// sgn_r s X_{1-r} with sgn_0 = -1, sgn_1 = +1.  One thread owns one
// (mode, class, component[, equation]) and keeps one parity of its arrays in
// registers (parity index i, n = 2i + sig), bounded at compile time by MH.
//
// Chebyshev conventions: f(y) = sum_n a_n T_n(y), nodes y_j = cos(pi j / N);
// derivative recurrence c_m b_m = b_{m+2} + 2 (m+1) a_{m+1} (c_0 = 2).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "stage_launch.h"
#include "stage_scan.cuh"

namespace chdns {

// ---------------------------------------------------------------------------
// shared-memory views
// ---------------------------------------------------------------------------

// component r of a complex [n][ppc] tile: element n at p[n * stride]
template <typename T>
struct CompT {
  T* p;
  int stride;
  __device__ T& operator[](int n) const { return p[n * stride]; }
};
using CompS = CompT<double>;

// tau factor tables of one (mode, parity): element (f, i) at base[(f * Mh + i) * ppc]
struct TabSm {
  const double* base;
  int Mh, ppc;
  __device__ double e(int i) const { return base[(0 * Mh + i) * ppc]; }
  __device__ double h(int i) const { return base[(1 * Mh + i) * ppc]; }
  __device__ double b(int i) const { return base[(2 * Mh + i) * ppc]; }
  __device__ double Q(int i) const { return base[(3 * Mh + i) * ppc]; }
};

// cos(pi j n / N) table in the node precision
template <typename RN>
__device__ __forceinline__ const RN* cheb_table(const DevTables& t);
template <>
__device__ __forceinline__ const double* cheb_table<double>(const DevTables& t) { return t.cheb; }
template <>
__device__ __forceinline__ const float* cheb_table<float>(const DevTables& t) { return t.cheb_f; }

// Chebyshev coefficients a_n, n = n0 + dn k (k < KN, all of one parity), of
// one field of one mode from its nodal values col[j * stride], j = 0..N, by the
// direct sums a_n = (2 / (N c_n)) sum_j'' f_j cos(pi j n / N) over the folded
// pairs f_j + (-1)^n f_{N-j} (sg = (-1)^n), accumulated over j in ascending
// order; c_0 = c_N = 2, the end nodes weigh 1/2.
template <typename RN, int KN>
__device__ __forceinline__ void analysis_sums(const typename cpx<RN>::T* col, int stride, int N, int ny,
                                              const RN* __restrict__ cheb, int n0, int dn, RN sg,
                                              typename cpx<RN>::T (&acc)[KN]) {
  using CN = typename cpx<RN>::T;
  CN a[KN];
  const CN w0 = (RN)0.5 * (col[0] + sg * col[N * stride]);  // j = 0 and j = N weigh 1/2
#pragma unroll
  for (int k = 0; k < KN; ++k) a[k] = w0;
  for (int j = 1; 2 * j < N; ++j) {
    const CN fold = col[j * stride] + sg * col[(N - j) * stride];
#pragma unroll
    for (int k = 0; k < KN; ++k) {
      const int n = n0 + dn * k;
      a[k] = a[k] + cheb[(size_t)min(n, N) * ny + j] * fold;
    }
  }
  const RN s0 = (RN)2.0 / (RN)N;
#pragma unroll
  for (int k = 0; k < KN; ++k) {
    const int n = n0 + dn * k;
    const RN cbn = (n == 0 || n == N) ? (RN)2.0 : (RN)1.0;
    CN v = a[k];
    if ((N & 1) == 0) v = v + cheb[(size_t)min(n, N) * ny + N / 2] * col[(N / 2) * stride];
    acc[k] = (s0 / cbn) * v;
  }
}

// ---------------------------------------------------------------------------
// stage_pre
//   u = (i kx Dv - i kz g)/k^2, w = (i kz Dv + i kx g)/k^2,
//   omega_x = Dw - i kz v, omega_z = i kx v - Du;  mean mode: u = U, w = W,
//   omega_x = DW, omega_z = -DU.
// Thread (mode, class c, component r) writes component r of u, w, omega_y on
// parity 1-c and of v, omega_x, omega_z on parity c; its derivative chains run
// on component 1-r from n = N down to 0.  All threads then evaluate the six
// Chebyshev series at the nodes: f_j = E_j + O_j, f_{N-j} = E_j - O_j with the
// even/odd partial sums of a_n cos(pi n j / N), for the (N+1)/2 node pairs
// j < N/2.  For even N the middle node needs no products,
// f_{N/2} = sum_m (-1)^m a_{2m}; the thread writing the even coefficients of a
// field sums it on the way, so the node pairs divide evenly over the threads.
// ---------------------------------------------------------------------------
template <typename RN, int MH>
__global__ void __launch_bounds__(128) stage_pre_kernel(Grid g, int B, PencilBufs pb, DevTables t,
                                                        typename cpx<RN>::T* __restrict__ q, int ppc) {
  using CN = typename cpx<RN>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P, ny = g.ny, N = g.N;
  // v, omega_y coefficients in the node precision, then the six fields
  CN* sV = reinterpret_cast<CN*>(smem_raw);  // [ny][ppc]
  CN* sG = sV + ny * ppc;                    // [ny][ppc]
  CN* sC = sG + ny * ppc;                    // [6][ny][ppc]
  const int p0 = blockIdx.x * ppc;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  const int tid = threadIdx.x, nt = blockDim.x;
  pdl_wait_then_release();  // v, omega_y come from the previous stage
  for (int w = tid; w < ny * ppc; w += nt) {
    const int pl = w % ppc, n = w / ppc;
    const int p = p0 + pl;
    const size_t o = ((size_t)b * ny + n) * P + p;
    if constexpr (sizeof(RN) == 4) {
      sV[w] = (p < P) ? pb.V32[o] : czero<CN>();
      sG[w] = (p < P) ? pb.G32[o] : czero<CN>();
    } else {
      sV[w] = (p < P) ? pb.V[o] : czero<CN>();
      sG[w] = (p < P) ? pb.G[o] : czero<CN>();
    }
  }
  __syncthreads();

  // Recover: the chain of every (mode, class c, component r) is walked by
  // LC = 4 lanes (fixed, so every tile shape sums in the same order).  Lane lc
  // takes a contiguous block of the step pairs (U-step at n_u = nu0 - 2k,
  // V-step at n_u - 1), counted from the top; Dv, D omega_y and then D^2 v are
  // inclusive prefix sums of their terms over k, formed per block and
  // completed by the block totals of the lanes above (shuffles within the
  // 4-lane group); the halvings at n = 0 come last.
  {
    constexpr int LC = 4;
    constexpr int KB = (MH + 1 + LC - 1) / LC;  // step pairs per lane, bound
    const int lc = tid % LC;
    const int chain = tid / LC;  // (mode, combo) as tid did before: pl fastest
    const bool on = chain < 4 * ppc;
    const int pl = chain % ppc;
    const int combo = chain / ppc;
    const int c = combo & 1, r = combo >> 1;
    const int p = p0 + pl;
    const int row = p / g.nxh, ix = p % g.nxh;
    const int fs = 2 * ny * ppc;  // reals per field
    RN* out = reinterpret_cast<RN*>(sC) + 2 * pl + r;
    // middle node f_{N/2} = sum over even n of (-1)^(n/2) a_n, per field
    RN mid[6] = {0, 0, 0, 0, 0, 0};
    auto W = [&](int f, int n, RN x) {
      out[f * fs + n * 2 * ppc] = x;
      if ((n & 1) == 0) mid[f] = (n & 2) ? mid[f] - x : mid[f] + x;
    };
    // inclusive prefix over the 4-lane group of this lane's block total;
    // returns the exclusive offset
    auto lane_offset = [&](RN tot) {
      RN inc = tot;
#pragma unroll
      for (int o = 1; o < LC; o <<= 1) {
        const RN v = __shfl_up_sync(0xffffffffu, inc, o, LC);
        if (lc >= o) inc = inc + v;
      }
      return inc - tot;
    };
    const bool zero = !on || p >= P || row == g.nz / 2 || (p == 0 && r == 1);
    const bool mean = on && !zero && p == 0;
    if (on && zero) {
      for (int n = lc; n <= N; n += LC) {
        if ((n & 1) == 1 - c) { W(0, n, 0.0); W(2, n, 0.0); W(4, n, 0.0); }
        else { W(1, n, 0.0); W(3, n, 0.0); W(5, n, 0.0); }
      }
    } else if (mean && lc == 0) {
      const double* U = pb.UM + (size_t)b * ny;
      const double* Wm = pb.WM + (size_t)b * ny;
      double du = 0.0, dw = 0.0;
      for (int n = N; n >= 0; --n) {
        if ((n & 1) == 1 - c) {
          W(0, n, U[n]);
          W(2, n, Wm[n]);
          W(4, n, 0.0);
        } else {
          const double un = (n + 1 <= N) ? U[n + 1] : 0.0, wn = (n + 1 <= N) ? Wm[n + 1] : 0.0;
          const double t1 = du + 2.0 * (n + 1) * un, t2 = dw + 2.0 * (n + 1) * wn;
          du = (n == 0) ? 0.5 * t1 : t1;
          dw = (n == 0) ? 0.5 * t2 : t2;
          W(1, n, 0.0);
          W(3, n, dw);
          W(5, n, -du);
        }
      }
    }
    // the scans run on every lane (shuffles); only general modes use them
    const bool gen = on && !zero && !mean;
    const RN kx = gen ? (RN)t.kx[ix] : (RN)0, kz = gen ? (RN)t.kz[row] : (RN)0;
    const RN sg = (r == 0) ? (RN)-1.0 : (RN)1.0;
    const RN ik2 = gen ? sg / (kx * kx + kz * kz) : (RN)0;
    const RN skx = sg * kx, skz = sg * kz;
    const CompT<RN> V{reinterpret_cast<RN*>(sV) + 2 * pl + r, 2 * ppc};
    const CompT<RN> Va{reinterpret_cast<RN*>(sV) + 2 * pl + (1 - r), 2 * ppc};
    const CompT<RN> G{reinterpret_cast<RN*>(sG) + 2 * pl + r, 2 * ppc};
    const CompT<RN> Ga{reinterpret_cast<RN*>(sG) + 2 * pl + (1 - r), 2 * ppc};
    const int nu0 = ((N & 1) == 1 - c) ? N : N + 1;  // first U-step (N + 1: none)
    const int K = nu0 / 2 + 1;                       // step pairs
    const int Bk = (K + LC - 1) / LC;
    const int k0 = lc * Bk;
    RN dvk[KB], dgk[KB], d2k[KB];
    RN sdv = 0, sdg = 0;
#pragma unroll
    for (int j = 0; j < KB; ++j) {
      const int k = k0 + j;
      const int nu = nu0 - 2 * k;
      RN tdv = 0, tdg = 0;
      if (gen && j < Bk && k < K) {
        if (nu + 1 <= N) tdv = (RN)(2 * (nu + 1)) * Va[nu + 1];  // U-step at nu
        if (nu <= N && nu >= 1) tdg = (RN)(2 * nu) * Ga[nu];      // V-step at nu - 1
      }
      sdv = sdv + tdv;
      sdg = sdg + tdg;
      dvk[j] = sdv;
      dgk[j] = sdg;
    }
    const RN odv = lane_offset(sdv), odg = lane_offset(sdg);
    RN sd2 = 0;
#pragma unroll
    for (int j = 0; j < KB; ++j) {
      const int k = k0 + j;
      const int nu = nu0 - 2 * k;
      dvk[j] = dvk[j] + odv;
      dgk[j] = dgk[j] + odg;
      RN td2 = 0;
      if (gen && j < Bk && k < K && nu >= 1) td2 = (RN)(2 * nu) * dvk[j];  // V-step at nu - 1
      sd2 = sd2 + td2;
      d2k[j] = sd2;
    }
    const RN od2 = lane_offset(sd2);
    if (gen) {
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        const int k = k0 + j;
        if (j >= Bk || k >= K) continue;
        const int nu = nu0 - 2 * k, nv = nu - 1;
        if (nu <= N) {
          const RN dv = (nu == 0) ? (RN)0.5 * dvk[j] : dvk[j];
          const RN ga = Ga[nu];
          W(0, nu, ik2 * (kx * dv - kz * ga));  // u
          W(2, nu, ik2 * (kz * dv + kx * ga));  // w
          W(4, nu, G[nu]);                      // omega_y
        }
        if (nv >= 0) {
          const RN h = (nv == 0) ? (RN)0.5 : (RN)1.0;
          const RN d2v = h * (d2k[j] + od2), dg = h * dgk[j];
          const RN va = Va[nv];
          const RN du = ik2 * (kx * d2v - kz * dg);
          const RN dw = ik2 * (kz * d2v + kx * dg);
          W(1, nv, V[nv]);            // v
          W(3, nv, dw - skz * va);    // omega_x = Dw - i kz v
          W(5, nv, skx * va - du);    // omega_z = i kx v - Du
        }
      }
    }
    // middle node: the even coefficients of this chain's fields are spread over
    // its 4 lanes
#pragma unroll
    for (int f = 0; f < 6; ++f)
#pragma unroll
      for (int o = 1; o < LC; o <<= 1) mid[f] = mid[f] + __shfl_xor_sync(0xffffffffu, mid[f], o, LC);
    // this chain wrote the even coefficients of fields 0, 2, 4 (c = 1) or 1, 3, 5 (c = 0)
    if (on && lc == 0 && (N & 1) == 0 && p < P) {
      RN* qr = reinterpret_cast<RN*>(q);
#pragma unroll
      for (int f = 0; f < 6; ++f)
        if ((f & 1) == 1 - c) qr[2 * (((size_t)(b * 6 + f) * ny + N / 2) * P + p) + r] = mid[f];
    }
  }
  __syncthreads();

  // synthesis of the six fields at the nodes.  Thread (mode pl, group g of
  // nt / ppc) evaluates the node pairs j = g, g + ng, ... of all six fields of
  // its mode: each coefficient it loads feeds all of its outputs, which are
  // independent accumulation chains.
  {
    constexpr int KJ = (MH - 1 + 15) / 16;  // node pairs per thread (ng = nt / ppc >= 16)
    const int ng = nt / ppc;
    const int pl = tid % ppc, gq = tid / ppc;
    const int J = (N + 1) / 2;  // node pairs (j, N - j), j < N/2
    const RN* cheb = cheb_table<RN>(t);
    if (gq < ng) {
      CN E[6][KJ], O[6][KJ];
#pragma unroll
      for (int f = 0; f < 6; ++f)
#pragma unroll
        for (int k = 0; k < KJ; ++k) {
          E[f][k] = czero<CN>();
          O[f][k] = czero<CN>();
        }
      const CN* col = sC + pl;
      // even and odd n in one iteration, so that neither update is predicated
      auto accumulate = [&](int n, CN (&acc)[6][KJ]) {
        CN cf[6];
#pragma unroll
        for (int f = 0; f < 6; ++f) cf[f] = col[((size_t)f * ny + n) * ppc];
#pragma unroll
        for (int k = 0; k < KJ; ++k) {
          const int j = gq + ng * k;
          const RN c = cheb[(size_t)min(j, N) * ny + n];
#pragma unroll
          for (int f = 0; f < 6; ++f) acc[f][k] = acc[f][k] + c * cf[f];
        }
      };
      for (int n = 0; n + 1 <= N; n += 2) {
        accumulate(n, E);
        accumulate(n + 1, O);
      }
      if ((N & 1) == 0) accumulate(N, E);
      const int p = p0 + pl;
      if (p < P) {
#pragma unroll
        for (int k = 0; k < KJ; ++k) {
          const int j = gq + ng * k;
          if (j >= J) continue;
#pragma unroll
          for (int f = 0; f < 6; ++f) {
            CN* dst = q + ((size_t)(b * 6 + f) * ny) * P + p;
            dst[(size_t)j * P] = E[f][k] + O[f][k];
            dst[(size_t)(N - j) * P] = E[f][k] - O[f][k];
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// stage_post
// Analysis: a_n = 2/(N cb_n) sum_j f_j cos(pi n j / N) / cb_j (cb_0 = cb_N = 2),
// node pairs (j, N-j) folded by the parity of n.
// Implicit part, with c = alpha/beta and the shifted unknowns
// g' = g^k + c g^{k-1}, phi' = phi^k + c phi^{k-1}, v' = v^k + c v^{k-1}:
//   (D^2 - lam) g'   = -((1 + c) g + dt (gamma h_g + zeta h_g')) / (beta dt nu)
//   (D^2 - lam) phi' = -((1 + c) phi + dt (gamma h_v + zeta h_v')) / (beta dt nu),
//   (D^2 - k^2) v'   = phi',   phi = (D^2 - k^2) v^{k-1},
// lam = k^2 + 1/(beta dt nu).  (D^2 - k^2) X = (D^2 - lam) X + X/(beta dt nu)
// holds for every coefficient row, so this is the same tau discretisation as
// the plain form without derivatives of the old fields.  The solve is linear
// in its right-hand side, so the factor -1/(beta dt nu), the same for every
// coefficient of a stage, is folded into the elimination factors e of the
// Helmholtz tables on the host: the kernels form (1 + c) g + dt (...) only.
// The wall rows of g' and v' carry c times the old wall values; the influence
// matrix fixes Dv'(+-1) = c Dv^{k-1}(+-1).  Then g^k = g' - c g^{k-1},
// v^k = v' - c v^{k-1}.
//   h_g = i kz H_x - i kx H_z,  h_v = -k^2 H_y - D(i kx H_x + i kz H_z).
// Thread (mode, class c, component r, equation e): e = 0 omega_y on parity
// 1-c, e = 1 v on parity c.  The mean mode solves U at constant flow rate
// (e = 0) and W (e = 1) on parity c, real component only.
// ---------------------------------------------------------------------------
// Per-tile form: 8 systems of kLanes lanes (stage_scan.cuh), four warps, per mode
constexpr int kModeThreads = 8 * kLanes;

template <typename RN, int MH>
__global__ void __launch_bounds__(8 * kModeThreads) stage_post_kernel(Grid g, int B, PencilBufs pb, DevTables t,
                                                        const typename cpx<RN>::T* __restrict__ hn, StageCoef sc,
                                                        int ppc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = g.P, ny = g.ny, N = g.N;
  const int Mh = t.tau.Mh;
  using CN = typename cpx<RN>::T;
  double2* sH = reinterpret_cast<double2*>(smem_raw);  // [3][ny][ppc] nodes, then coefficients (RN)
  double2* sV = sH + 3 * ny * ppc;                      // [ny][ppc]
  double2* sG = sV + ny * ppc;
  // previous right-hand sides h_v', h_g' in the node precision (FP64-sized slots)
  CN* sHV = reinterpret_cast<CN*>(sG + ny * ppc);
  CN* sHG = reinterpret_cast<CN*>(sG + 2 * ny * ppc);
  double* sh = reinterpret_cast<double*>(sG + 3 * ny * ppc);  // helm [2][4][Mh][ppc] of this stage
  double* sp = sh + 2 * 4 * Mh * ppc;                        // pois [2][4][Mh][ppc]
  double* svh = sp + 2 * 4 * Mh * ppc;                       // vh [2][Mh][ppc]
  double* ss = svh + 2 * Mh * ppc;                           // helm_isq, pois_isq, vh_idv [3][2][ppc]
  const int p0 = blockIdx.x * ppc;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  const int tid = threadIdx.x, nt = blockDim.x;

  // ---- load the tile (asynchronous copies, all in flight before the wait)
  for (int w = tid; w < ny * ppc; w += nt) {
    const int pl = w % ppc, n = w / ppc;
    const int p = min(p0 + pl, P - 1);
    const size_t o = ((size_t)b * ny + n) * P + p;
    cp_async_elem(sV + w, pb.V + o);
    cp_async_elem(sG + w, pb.G + o);
    cp_async_elem(sHV + w, reinterpret_cast<const CN*>(pb.HVP) + o);
    cp_async_elem(sHG + w, reinterpret_cast<const CN*>(pb.HGP) + o);
  }
  for (int w = tid; w < 2 * 4 * Mh * ppc; w += nt) {
    const int pl = w % ppc, qq = w / ppc;  // qq = (sig * 4 + f) * Mh + i
    const int p = min(p0 + pl, P - 1);
    cp_async_elem(sh + w, t.tau.helm + ((size_t)sc.k * 2 * 4 * Mh + qq) * P + p);
    cp_async_elem(sp + w, t.tau.pois + (size_t)qq * P + p);
  }
  for (int w = tid; w < 2 * Mh * ppc; w += nt) {
    const int pl = w % ppc, qq = w / ppc;
    const int p = min(p0 + pl, P - 1);
    cp_async_elem(svh + w, t.tau.vh + ((size_t)sc.k * 2 * Mh + qq) * P + p);
  }
  for (int w = tid; w < 2 * ppc; w += nt) {
    const int pl = w % ppc, sig = w / ppc;
    const int p = min(p0 + pl, P - 1);
    cp_async_elem(ss + (0 * 2 + sig) * ppc + pl, t.tau.helm_isq + (size_t)(sc.k * 2 + sig) * P + p);
    cp_async_elem(ss + (1 * 2 + sig) * ppc + pl, t.tau.pois_isq + (size_t)sig * P + p);
    cp_async_elem(ss + (2 * 2 + sig) * ppc + pl, t.tau.vh_idv + (size_t)(sc.k * 2 + sig) * P + p);
  }
  // everything above is independent of the nonlinear term; H comes from the
  // preceding kernel
  pdl_wait_then_release();
  // nodal values in the node precision, in the first bytes of the sH region
  CN* sN = reinterpret_cast<CN*>(sH);
  for (int w = tid; w < 3 * ny * ppc; w += nt) {
    const int pl = w % ppc, fn = w / ppc;  // fn = f * ny + n
    const int p = min(p0 + pl, P - 1);
    cp_async_elem(sN + w, hn + ((size_t)b * 3 * ny + fn) * P + p);
  }
  cp_async_wait_all();
  __syncthreads();

  // ---- Chebyshev analysis of H_x, H_y, H_z by direct sums over the node pairs
  // (j, N - j), folded in place: f_j + f_{N-j} at j, f_j - f_{N-j} at N - j; j = 0
  // and N weigh 1/2.  Thread t of a mode's threads forms the values (field,
  // component, n) t, t + kModeThreads, ...; with so few modes the sums spread over
  // four warps finish before a transform in one.
  const int ml = tid / kModeThreads, mt = tid % kModeThreads;  // mode of the tile, thread of the mode
  RN* sR = reinterpret_cast<RN*>(sN);  // component r of (field, n, mode) at 2 ((f ny + n) ppc + mode) + r
  for (int w = mt; w < 6 * ((N + 1) / 2); w += kModeThreads) {
    const int j = w / 6, f = w % 6 / 2, r = w & 1;
    RN* a = sR + 2 * ((size_t)(f * ny + j) * ppc + ml) + r;
    RN* c = sR + 2 * ((size_t)(f * ny + N - j) * ppc + ml) + r;
    const RN x = j == 0 ? (RN)0.5 * *a : *a, y = j == 0 ? (RN)0.5 * *c : *c;
    *a = x + y;
    *c = x - y;
  }
  __syncthreads();
  {
    constexpr int KN = (12 * MH + kModeThreads - 1) / kModeThreads;  // values per thread, 6 (N + 1) <= 12 MH - 6
    const RN* cheb = cheb_table<RN>(t);
    const RN s0 = (RN)2.0 / (RN)N;
    RN acc[KN];
#pragma unroll
    for (int k = 0; k < KN; ++k) {
      const int w = mt + kModeThreads * k;
      acc[k] = (RN)0;
      if (w < 6 * ny) {
        // even n first, so that the lanes of a warp mostly share the folded values
        const int fr = w / ny, m = w % ny, ne = N / 2 + 1;
        const int n = m < ne ? 2 * m : 2 * (m - ne) + 1;
        const int st = m < ne ? 2 * ppc : -2 * ppc;
        const RN* x = sR + 2 * ((size_t)((fr / 2) * ny + (m < ne ? 0 : N)) * ppc + ml) + (fr & 1);
        RN a = 0;
#pragma unroll 8
        for (int j = 0; 2 * j < N; ++j) a = fma_rn(cheb[(size_t)j * ny + n], x[j * st], a);
        if (m < ne && (N & 1) == 0) a = fma_rn((n & 2) ? (RN)-1.0 : (RN)1.0, x[(N / 2) * st], a);
        acc[k] = ((n == 0 || n == N) ? (RN)0.5 * s0 : s0) * a;
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KN; ++k) {
      const int w = mt + kModeThreads * k;
      if (w < 6 * ny) {
        const int fr = w / ny, m = w % ny, ne = N / 2 + 1;
        const int n = m < ne ? 2 * m : 2 * (m - ne) + 1;
        sR[2 * ((size_t)((fr / 2) * ny + n) * ppc + ml) + (fr & 1)] = acc[k];
      }
    }
  }
  __syncthreads();

  // ---- implicit solves, system (mode, class c, component r, equation e) on
  // the lanes q of a group; e is uniform over each warp
  const int q = mt & (kLanes - 1), combo = mt / kLanes, pl = ml;
  const int p = p0 + pl;
  const int c = combo & 1, r = (combo >> 1) & 1, e = combo >> 2;
  const int row = p / g.nxh, ix = p % g.nxh;
  // a whole group is live or idle together
  if (p < P && row != g.nz / 2 && (p != 0 || r == 0)) {
    const double cc = sc.cc;
    const double* rowc = t.tau.rowc;
    const CN* Hx = reinterpret_cast<const CN*>(sH) + pl;
    const CN* Hy = Hx + ny * ppc;
    const CN* Hz = Hy + ny * ppc;
    auto helm = [&](int sig) { return TabSm{sh + sig * 4 * Mh * ppc + pl, Mh, ppc}; };
    auto comp = [](auto z, int qd) { return qd == 0 ? z.x : z.y; };
    if (p == 0) {
      mean_scan<MH, RN>(N, ny, ppc, c, e, (e == 0 ? pb.UM : pb.WM) + (size_t)b * ny,
                        (e == 0 ? pb.HXP : pb.HZP) + (size_t)b * ny, (e == 0) ? Hx : Hz, cc, sc, helm(c),
                        ss[(0 * 2 + c) * ppc + pl], rowc, t.tau.u1 + (size_t)sc.k * Mh, t.tau.u1_iflux[sc.k],
                        t.tau.wint, q);
    } else {
      const double kx = t.kx[ix], kz = t.kz[row], k2 = kx * kx + kz * kz;
      const double sgn = (r == 0) ? -1.0 : 1.0;
      if (e == 0) {
        // wall-normal vorticity, parity 1 - c
        const int sq = 1 - c;
        const CompS Gc{reinterpret_cast<double*>(sG) + 2 * pl + r, 2 * ppc};
        const CompT<RN> HGc{reinterpret_cast<RN*>(sHG) + 2 * pl + r, 2 * ppc};
        omega_scan<MH, RN>(N, ny, ppc, sq, Gc, HGc, Hx, Hz, r, sgn, kx, kz, cc, sc, helm(sq),
                           ss[(0 * 2 + sq) * ppc + pl], rowc, q);
      } else {
        // wall-normal velocity, parity c
        const int sv = c;
        const CompS Vc{reinterpret_cast<double*>(sV) + 2 * pl + r, 2 * ppc};
        const CompT<RN> HVc{reinterpret_cast<RN*>(sHV) + 2 * pl + r, 2 * ppc};
        const size_t vo = (size_t)b * P + p;
        const double vw =
            fma_rn(sc.theta, comp(pb.vw_new[vo], r) - comp(pb.vw_old[vo], r), comp(pb.vw_old[vo], r));
        const TabSm TP{sp + sv * 4 * Mh * ppc + pl, Mh, ppc};
        v_scan<MH, RN>(N, ny, ppc, sv, Vc, HVc, Hx, Hy, Hz, r, sgn, kx, kz, k2, cc, sc, helm(sv),
                       ss[(0 * 2 + sv) * ppc + pl], TP, ss[(1 * 2 + sv) * ppc + pl], svh + sv * Mh * ppc + pl,
                       ppc, ss[(2 * 2 + sv) * ppc + pl], vw, rowc, q);
      }
    }
  }
  __syncthreads();

  // ---- store the tile
  for (int w = tid; w < ny * ppc; w += nt) {
    const int pl2 = w % ppc, n = w / ppc;
    const int p2 = p0 + pl2;
    if (p2 >= P) continue;
    const size_t o = ((size_t)b * ny + n) * P + p2;
    pb.V[o] = sV[w];
    pb.G[o] = sG[w];
    if constexpr (sizeof(RN) == 4) {
      pb.V32[o] = make_float2((float)sV[w].x, (float)sV[w].y);
      const double2 gv = p2 == 0 ? mk(pb.WM[(size_t)b * ny + n], pb.UM[(size_t)b * ny + n]) : sG[w];
      pb.G32[o] = make_float2((float)gv.x, (float)gv.y);
    }
    reinterpret_cast<CN*>(pb.HVP)[o] = sHV[w];
    reinterpret_cast<CN*>(pb.HGP)[o] = sHG[w];
  }
}

// ---------------------------------------------------------------------------
// Chebyshev analysis of H by direct sums, for the orders without a register
// cosine transform: a tile of modes at a time, coefficients over the nodal
// values in place (a CTA reads all the nodes of its modes before it writes
// their coefficients).
// ---------------------------------------------------------------------------
template <typename RN, int MH>
__global__ void __launch_bounds__(256) stage_post_analysis_kernel(Grid g, int B, PencilBufs pb, DevTables t,
                                                                  typename cpx<RN>::T* __restrict__ hn, int ppc) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using CN = typename cpx<RN>::T;
  const int P = g.P, ny = g.ny, N = g.N;
  const int p0 = blockIdx.x * ppc;
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  const int tid = threadIdx.x, nt = blockDim.x;
  pdl_wait_then_release();  // H comes from the nonlinear term
  CN* hb = hn + (size_t)b * 3 * ny * P;
  // direct sums, one field at a time: thread (mode pl, group gq of 8) forms
  // the coefficients n = gq + 8 k
  constexpr int KN = (2 * MH + 7) / 8;
  CN* col0 = reinterpret_cast<CN*>(smem_raw);  // [ny][ppc]
  const int pl = tid % ppc, gq = tid / ppc;
  const RN* cheb = cheb_table<RN>(t);
  const RN sg = (gq & 1) ? (RN)-1.0 : (RN)1.0;
  for (int f = 0; f < 3; ++f) {
    CN* hf = hb + (size_t)f * ny * P;
    for (int w = tid; w < ny * ppc; w += nt) {
      const int q = w % ppc, n = w / ppc;
      col0[w] = hf[(size_t)n * P + min(p0 + q, P - 1)];
    }
    __syncthreads();
    if (gq < 8) {
      CN acc[KN];
      analysis_sums<RN, KN>(col0 + pl, ppc, N, ny, cheb, gq, 8, sg, acc);
      if (p0 + pl < P) {
#pragma unroll
        for (int k = 0; k < KN; ++k) {
          const int n = gq + 8 * k;
          if (n <= N) hf[(size_t)n * P + p0 + pl] = acc[k];
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// per-MH launchers, instantiated in the stage_mh*.cu translation units
// ---------------------------------------------------------------------------
template <typename RN, int MH>
cudaError_t pre_mh(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                          typename cpx<RN>::T* q, int ppc, size_t smem, cudaStream_t st) {
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_kernel<RN, MH>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_pre_kernel<RN, MH>, dim3((g.P + ppc - 1) / ppc, B), dim3(128), smem,
                                        st, g, B, pb, t, q, ppc);
}

template <typename RN, int MH>
cudaError_t post_mh(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                           const typename cpx<RN>::T* h, const StageCoef& sc, int ppc, size_t smem,
                           cudaStream_t st) {
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_post_kernel<RN, MH>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_post_kernel<RN, MH>, dim3((g.P + ppc - 1) / ppc, B),
                                        dim3(kModeThreads * ppc), smem, st, g, B, pb, t, h, sc, ppc);
}

template <typename RN, int MH>
cudaError_t analysis_mh(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* h,
                        cudaStream_t st) {
  constexpr int ppc = 32;  // 8 threads per mode
  const size_t smem = (size_t)g.ny * ppc * sizeof(typename cpx<RN>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_post_analysis_kernel<RN, MH>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_post_analysis_kernel<RN, MH>, dim3((g.P + ppc - 1) / ppc, B),
                                        dim3(8 * ppc), smem, st, g, B, pb, t, h, ppc);
}

}  // namespace chdns

// explicit instantiations of the launchers for one register-array bound MH,
// both node precisions, by kernel form
#define CH_STAGE_PRE(MH)                                                                                       \
  namespace chdns {                                                                                            \
  template cudaError_t pre_mh<double, MH>(const Grid&, int, const PencilBufs&, const DevTables&, double2*, int,  \
                                          size_t, cudaStream_t);                                               \
  template cudaError_t pre_mh<float, MH>(const Grid&, int, const PencilBufs&, const DevTables&, float2*, int,    \
                                         size_t, cudaStream_t);                                                \
  }
#define CH_STAGE_POST(MH)                                                                                      \
  namespace chdns {                                                                                            \
  template cudaError_t post_mh<double, MH>(const Grid&, int, const PencilBufs&, const DevTables&, const double2*, \
                                           const StageCoef&, int, size_t, cudaStream_t);                       \
  template cudaError_t post_mh<float, MH>(const Grid&, int, const PencilBufs&, const DevTables&, const float2*,  \
                                          const StageCoef&, int, size_t, cudaStream_t);                        \
  template cudaError_t analysis_mh<double, MH>(const Grid&, int, const PencilBufs&, const DevTables&, double2*,  \
                                               cudaStream_t);                                                  \
  template cudaError_t analysis_mh<float, MH>(const Grid&, int, const PencilBufs&, const DevTables&, float2*,    \
                                              cudaStream_t);                                                   \
  }
#define CH_STAGE_INSTANTIATE(MH) CH_STAGE_PRE(MH) CH_STAGE_POST(MH)
