// The implicit half of one Runge-Kutta stage for handles with few modes, fused
// over a tile of `ppc` Fourier modes that lives in shared memory: nodal values
// of H = u x omega -> Chebyshev coefficients -> right-hand sides ->
// Chebyshev-tau solves -> new state.  Every global array is read and written
// once, with accesses that are contiguous over the modes of the tile.  RN is
// the precision of the nodal values exchanged with the plane kernels (double:
// all-FP64 path).
//
// Symmetry classes and components.  All wall-normal operators are real and
// map even Chebyshev coefficients to even or odd ones in a fixed pattern, so a
// mode splits into two classes (c = 0: even v, odd omega_y; c = 1: odd v,
// even omega_y) and two real components (r = 0, 1) that never interact.  The
// factors i kx, i kz only swap components: component r of (i s X) is
// sgn_r s X_{1-r} with sgn_0 = -1, sgn_1 = +1.
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
  // nodal values in the node precision, in the first bytes of the sH region
  CN* sN = reinterpret_cast<CN*>(sH);
  for (int w = tid; w < 3 * ny * ppc; w += nt) {
    const int pl = w % ppc, fn = w / ppc;  // fn = f * ny + n
    const int p = min(p0 + pl, P - 1);
    cp_async_elem(sN + w, hn + b * g.qb + fn / ny * g.qf + fn % ny * g.qj + p);
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
                        t.tau.wint, t.tau.n1, q, reinterpret_cast<float*>(pb.V32) + 2 * (size_t)b * ny * P + (e == 0 ? 1 : 0),
                        P);
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
      if (p2 > 0) pb.V32[o] = make_float2((float)sV[w].x, (float)sV[w].y);  // mode 0: mean_scan
      const double2 gv = p2 == 0 ? mk(pb.WM[(size_t)b * ny + n], pb.UM[(size_t)b * ny + n]) : sG[w];
      pb.G32[o] = make_float2((float)gv.x, (float)gv.y);
    }
    reinterpret_cast<CN*>(pb.HVP)[o] = sHV[w];
    reinterpret_cast<CN*>(pb.HGP)[o] = sHG[w];
  }
}

// ---------------------------------------------------------------------------
// per-MH launchers, instantiated in the stage_mh*.cu translation units
// ---------------------------------------------------------------------------
template <typename RN, int MH>
cudaError_t post_mh(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                           const typename cpx<RN>::T* h, const StageCoef& sc, int ppc, size_t smem,
                           cudaStream_t st) {
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_post_kernel<RN, MH>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(stage_post_kernel<RN, MH>, dim3((g.P + ppc - 1) / ppc, B),
                                        dim3(kModeThreads * ppc), smem, st, g, B, pb, t, h, sc, ppc);
}

}  // namespace chdns

// explicit instantiations of the launcher for one register-array bound MH,
// both node precisions
#define CH_STAGE_POST(MH)                                                                                      \
  namespace chdns {                                                                                            \
  template cudaError_t post_mh<double, MH>(const Grid&, int, const PencilBufs&, const DevTables&, const double2*, \
                                           const StageCoef&, int, size_t, cudaStream_t);                       \
  template cudaError_t post_mh<float, MH>(const Grid&, int, const PencilBufs&, const DevTables&, const float2*,  \
                                          const StageCoef&, int, size_t, cudaStream_t);                        \
  }
