// The implicit solves of a stage for handles with many modes: one thread per
// (mode, class, component, equation), reading the Chebyshev coefficients of H
// that the analysis kernel left in the node array.
//
// With c = alpha/beta and the shifted unknowns g' = g^k + c g^{k-1},
// phi' = phi^k + c phi^{k-1}, v' = v^k + c v^{k-1}:
//   (D^2 - lam) g'   = -((1 + c) g + dt (gamma h_g + zeta h_g')) / (beta dt nu)
//   (D^2 - lam) phi' = -((1 + c) phi + dt (gamma h_v + zeta h_v')) / (beta dt nu)
//   (D^2 - k^2) v'   = phi',   phi = (D^2 - k^2) v^{k-1},  lam = k^2 + 1/(beta dt nu),
//   h_g = i kz H_x - i kx H_z,  h_v = -k^2 H_y - D(i kx H_x + i kz H_z).
// (D^2 - k^2) X = (D^2 - lam) X + X/(beta dt nu) holds for every coefficient
// row, so this is the tau discretisation of the plain form without derivatives
// of the old fields; -1/(beta dt nu) is folded into the tables.
//
// One parity of a tau system (parity index i, n = 2i + sig) on the folded
// tables: with row constants cA_n, cB_n, cC_n of the twice-integrated rows and
// the elimination factors e, h, b,
//   a_j = eA_j r_{j-1} - eB_j r_j + eC_j r_{j+1} - h_j a_{j+1}   (j = M-1 .. 1),
//   f_0 from the wall row,  f_i = a_i + b_i f_{i-1}.
// The particular solution P_i = a_i + b_i P_{i-1} (P_0 = 0) enters the wall rows
// through sum P = sum W_i a_i and sum n^2 P = sum W2_i a_i, so one sweep
// down and one up solve the system.  In the phi solve the stencil of D^2 v is
// v_n itself (it integrates D^2 twice): row j takes E1_j v_j, E1 = (1 + c) e,
// and the stencil of u = -(1 + c) k^2 v + dt (...), and no D^2 v is formed.
//
// No-slip walls: sum f' = c sum f_old per parity for omega_y, U, W; v' the
// same plus the wall velocity, and the influence correction c_I vh that fixes
// Dv.  Free-slip top (TOP = 1): the rows Df(+1) and f(-1) (omega_y, W), these
// and the flow rate (U), D^2 v(+1) and Dv(-1) (v) couple the parities, which
// are the two warps of a CTA: each publishes the sums of its parity and both
// solve the same closure.
//
// What bounds it: the FP64 pipe, 29 operations per coefficient and (mode,
// component), of which two convert FP32 right-hand sides.  A warp-wide FP64
// operation takes the same 64 to 76 cycles of its sub-partition whatever the
// dependences, so what counts is that every sub-partition always has a warp
// whose operands are there: the coefficient array of a thread lives in a
// column of shared memory (M doubles; up to 24 warps per SM at 65 nodes,
// where arrays in registers left ten), loads run two rows ahead, the loops
// stay rolled, and the two equations are CTAs of their own.
#pragma once

#include "common.cuh"
#include "internal.h"
#include "stage_close.cuh"

namespace chdns {

template <int TOP> constexpr int solve_tabs() { return TOP ? 8 : 7; }  // eA, eB, eC, h, b, W, E1 (, W2)
constexpr int kPoisTabs = 6;                                           // eA, eB, eC, h, b, W

// one row's table entries
struct TabRow {
  double eA, eB, eC, h, W;
};
__device__ __forceinline__ TabRow tab_row(const double* __restrict__ T, size_t MP, size_t o) {
  return TabRow{__ldg(T + o), __ldg(T + MP + o), __ldg(T + 2 * MP + o), __ldg(T + 3 * MP + o), __ldg(T + 5 * MP + o)};
}

// Solve omega_y of parity sig of one (mode, component), or the mean flow in
// the lanes of mode 0 (component 0: U at constant flow rate, 1: W).
template <typename RN, int TOP>
__device__ __forceinline__ void solve_omega(double* f, double* xch, const Grid& g, const PencilBufs& pb,
                                            const DevTables& t, const StageCoef& sc, int b, int p, int r, int sig,
                                            bool live, const RN* __restrict__ hc) {
  constexpr int NT = 64;
  const size_t P = g.P, MP = (size_t)t.tau.Mh * P;
  const int ny = g.ny, N = g.N, M = (N - sig) / 2 + 1, row = p / g.nxh, ix = p % g.nxh;
  const bool mean = p == 0;
  const double cc = sc.alpha / sc.beta;
  const double* __restrict__ T = t.tau.helm_f + (size_t)(sc.k * 2 + sig) * solve_tabs<TOP>() * MP + p;
  const double* __restrict__ n2 = t.tau.n2;
  // column: value n at xp[n xs]; H: comp of two fields at ha[2 P n], hb[2 P n]
  const size_t hP = 2 * P, base = 2 * ((size_t)b * ny * P + p) + r;
  double* xp = mean ? (r == 0 ? pb.UM : pb.WM) + (size_t)b * ny : reinterpret_cast<double*>(pb.G) + base;
  const size_t xs = mean ? 1 : hP;
  double* XP = (r == 0 ? pb.HXP : pb.HZP) + (size_t)b * ny;
  RN* HG = reinterpret_cast<RN*>(pb.HGP) + base;
  const RN* H0 = hc + 2 * ((size_t)b * 3 * ny * P + p);
  const RN* hx = mean ? H0 + (r == 0 ? 0 : 2 * (size_t)ny * hP) : H0 + 1 - r;
  const RN* hz = H0 + 2 * (size_t)ny * hP + 1 - r;
  const RN sgn = r == 0 ? (RN)-1 : (RN)1, kx = (RN)t.kx[ix], kz = (RN)t.kz[row];
  const RN dtn = (RN)sc.dt, gan = (RN)sc.gamma, zen = (RN)sc.zeta;
  double S0 = 0.0, S2 = 0.0, flux_old = 0.0, sum = 0.0, sum2 = 0.0, f0 = 0.0, fc = 0.0;
  if (live) {
    struct In {
      double x;
      RN hx, hz, hp;
      TabRow tb;
      double W2;
    };
    auto load = [&](int i) {
      In v;
      const size_t n = 2 * i + sig;
      v.x = xp[n * xs];
      v.hx = __ldg(hx + n * hP);
      v.hz = __ldg(hz + n * hP);
      v.hp = HG[n * hP];
      if (i + 1 < M) {
        v.tb = tab_row(T, MP, (size_t)(i + 1) * P);
        if (TOP) v.W2 = __ldg(T + 7 * MP + (size_t)(i + 1) * P);
      }
      return v;
    };
    double r1 = 0.0, r2 = 0.0, an = 0.0;
    auto step = [&](int i, const In& v) {
      const size_t n = 2 * i + sig;
      double q;
      if (mean) {
        const double h = (double)v.hx, hp = XP[n];
        XP[n] = h;
        q = sc.dt * fma(sc.gamma, h, sc.zeta * hp);
        if (sig == 0) flux_old = fma(t.tau.wint[n], v.x, flux_old);
      } else {
        const RN hg = sgn * (kz * v.hx - kx * v.hz);
        HG[n * hP] = hg;
        q = (double)(dtn * (gan * hg + zen * v.hp));
      }
      S0 += v.x;
      if (TOP) S2 = fma(__ldg(n2 + n), v.x, S2);
      const double r0 = fma(1.0 + cc, v.x, q);
      if (i + 1 < M) {
        const double a = fma(-v.tb.h, an, fma(v.tb.eC, r2, fma(-v.tb.eB, r1, v.tb.eA * r0)));
        f[(i + 1) * NT] = a;
        sum = fma(v.tb.W, a, sum);
        if (TOP) sum2 = fma(v.W2, a, sum2);
        an = a;
      }
      r2 = r1;
      r1 = r0;
    };
    In u = load(M - 1), v = load(M - 2);
    int i = M - 1;
    for (; i >= 3; i -= 2) {
      const In u1 = load(i - 2);
      step(i, u);
      const In v1 = load(i - 3);
      step(i - 1, v);
      u = u1;
      v = v1;
    }
    // two or three rows left: i, i - 1 (and 0)
    if (i == 2) {
      const In w = load(0);
      step(2, u);
      step(1, v);
      step(0, w);
    } else {
      step(1, u);
      step(0, v);
    }
  }
  if (TOP == 0) {
    f0 = t.tau.helm_isq[(size_t)(sc.k * 2 + sig) * P + p] * (cc * S0 - sum);
    if (mean && r == 0 && sig == 0) {
      double flux = 0.0, fp = f0;
      for (int i = 0; i < M; ++i) {
        if (i > 0) fp = fma(__ldg(T + 4 * MP + (size_t)i * P), fp, f[i * NT]);
        flux = fma(t.tau.wint[2 * i], fp, flux);
      }
      fc = (fma(cc, flux_old, sc.flux) - flux) * t.tau.u1_iflux[sc.k];
    }
  } else {
    double wp = 0.0;
    if (live && mean && sig == 0) {
      double fp = 0.0;
      for (int i = 1; i < M; ++i) {
        fp = fma(__ldg(T + 4 * MP + (size_t)i * P), fp, f[i * NT]);
        wp = fma(t.tau.wint[2 * i], fp, wp);
      }
    }
    const int me = threadIdx.x, mate = me ^ 32;
    const double mine[6] = {sum, sum2, S0, S2, wp, flux_old};
#pragma unroll
    for (int k = 0; k < 6; ++k) xch[k * NT + me] = mine[k];
    __syncthreads();
    if (!live) return;
    double se[6], so[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const double other = xch[k * NT + mate];
      se[k] = sig == 0 ? mine[k] : other;
      so[k] = sig == 0 ? other : mine[k];
    }
    auto qs = [&](int s, int w) { return t.tau.helm_top[((size_t)(sc.k * 2 + s) * 2 + w) * P + p]; };
    double xe, xo;
    if (mean && r == 0) {
      const double* m = t.tau.mean_top + 4 * sc.k;  // int Q_e; sum, sum n^2 and int of the forcing response
      close_free_slip_mean(se, so, qs(0, 0), qs(1, 0), qs(0, 1), qs(1, 1), m[0], m[1], m[2], m[3], cc, sc.flux, &xe, &xo,
                           &fc);
      if (sig != 0) fc = 0.0;
    } else {
      close_neumann_top(se, so, qs(0, 0), qs(1, 0), qs(0, 1), qs(1, 1), cc, &xe, &xo);
    }
    f0 = sig == 0 ? xe : xo;
  }
  // up: f_i = a_i + b_i f_{i-1}; x <- f - c x (+ the forced response of U)
  const double* __restrict__ u1 = t.tau.u1 + (size_t)sc.k * t.tau.Mh;
  auto out = [&](int i, double fi, double x) {
    double y = fma(-cc, x, fi);
    if (mean && r == 0 && sig == 0) y = fma(fc, u1[i], y);
    xp[(size_t)(2 * i + sig) * xs] = y;
  };
  double fp = f0;
  out(0, fp, xp[(size_t)sig * xs]);
  for (int i = 1; i < M; i += 4) {
    double bb[4], x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < M) {
        bb[k] = __ldg(T + 4 * MP + (size_t)(i + k) * P);
        x[k] = xp[(size_t)(2 * (i + k) + sig) * xs];
      }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < M) {
        fp = fma(bb[k], fp, f[(i + k) * NT]);
        out(i + k, fp, x[k]);
      }
  }
}

// Solve v of parity sig of one (mode, component).
template <typename RN, int TOP>
__device__ __forceinline__ void solve_v(double* f, double* xch, const Grid& g, const PencilBufs& pb, const DevTables& t,
                                        const StageCoef& sc, int b, int p, int r, int sig, bool live,
                                        const RN* __restrict__ hc) {
  constexpr int NT = 64;
  const size_t P = g.P, MP = (size_t)t.tau.Mh * P;
  const int ny = g.ny, N = g.N, M = (N - sig) / 2 + 1, row = p / g.nxh, ix = p % g.nxh;
  const double cc = sc.alpha / sc.beta;
  const double* __restrict__ T = t.tau.helm_f + (size_t)(sc.k * 2 + sig) * solve_tabs<TOP>() * MP + p;
  const double* __restrict__ TP = t.tau.pois_f + (size_t)sig * kPoisTabs * MP + p;
  const double* __restrict__ n2 = t.tau.n2;
  const size_t hP = 2 * P, base = 2 * ((size_t)b * ny * P + p) + r;
  double* Vp = reinterpret_cast<double*>(pb.V) + base;
  RN* HV = reinterpret_cast<RN*>(pb.HVP) + base;
  const RN* H0 = hc + 2 * ((size_t)b * 3 * ny * P + p);
  const RN* hx = H0 + 1 - r;
  const RN* hy = H0 + (size_t)ny * hP + r;
  const RN* hz = H0 + 2 * (size_t)ny * hP + 1 - r;
  const double kxd = t.kx[ix], kzd = t.kz[row], k2 = fma(kxd, kxd, kzd * kzd), ck2 = -(1.0 + cc) * k2;
  const RN sgn = r == 0 ? (RN)-1 : (RN)1, kx = (RN)kxd, kz = (RN)kzd, k2n = (RN)k2;
  const RN dtn = (RN)sc.dt, gan = (RN)sc.gamma, zen = (RN)sc.zeta;
  double Aw = 0.0, Bw = 0.0;
  if (live) {
    struct In {
      double x;
      RN hx, hy, hz, hp;
      TabRow tb;
      double E1;
    };
    auto load = [&](int i) {
      In v;
      const size_t n = 2 * i + sig;
      v.x = Vp[n * hP];
      v.hy = __ldg(hy + n * hP);
      v.hp = HV[n * hP];
      if ((int)n + 1 <= N) {
        v.hx = __ldg(hx + (n + 1) * hP);
        v.hz = __ldg(hz + (n + 1) * hP);
      } else {
        v.hx = v.hz = (RN)0;
      }
      if (i + 1 < M) {
        v.tb = tab_row(T, MP, (size_t)(i + 1) * P);
        v.E1 = __ldg(T + 6 * MP + (size_t)(i + 1) * P);
      }
      return v;
    };
    double S0 = 0.0, sum = 0.0, r1 = 0.0, r2 = 0.0, x1 = 0.0, an = 0.0;
    RN dtt = 0;  // D(i kx H_x + i kz H_z), from the top down
    auto step = [&](int i, const In& v) {
      const int n = 2 * i + sig;
      const RN t2 = (RN)(2 * (n + 1)) * (sgn * (kx * v.hx + kz * v.hz)) + dtt;
      dtt = n == 0 ? (RN)0.5 * t2 : t2;
      const RN hv = -k2n * v.hy - dtt;
      HV[(size_t)n * hP] = hv;
      const RN q = dtn * (gan * hv + zen * v.hp);
      S0 += v.x;
      const double r0 = fma(ck2, v.x, (double)q);
      if (i + 1 < M) {
        const double a =
            fma(-v.tb.h, an, fma(v.E1, x1, fma(v.tb.eC, r2, fma(-v.tb.eB, r1, v.tb.eA * r0))));
        f[(i + 1) * NT] = a;
        sum = fma(v.tb.W, a, sum);
        an = a;
      }
      r2 = r1;
      r1 = r0;
      x1 = v.x;
    };
    In u = load(M - 1), v = load(M - 2);
    int i = M - 1;
    for (; i >= 3; i -= 2) {
      const In u1 = load(i - 2);
      step(i, u);
      const In v1 = load(i - 3);
      step(i - 1, v);
      u = u1;
      v = v1;
    }
    if (i == 2) {
      const In w = load(0);
      step(2, u);
      step(1, v);
      step(0, w);
    } else {
      step(1, u);
      step(0, v);
    }
    // phi, with zero wall sum
    double fp = t.tau.helm_isq[(size_t)(sc.k * 2 + sig) * P + p] * -sum;
    f[0] = fp;
    for (int i = 1; i < M; i += 4) {
      double bb[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k < M) bb[k] = __ldg(T + 4 * MP + (size_t)(i + k) * P);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k < M) {
          fp = fma(bb[k], fp, f[(i + k) * NT]);
          f[(i + k) * NT] = fp;
        }
    }
    // (D^2 - k^2) v_p = phi, the array read at i and written at i + 1
    sum = an = r2 = 0.0;
    r1 = fp;
    for (int j = M - 1; j >= 1; j -= 2) {
      const TabRow ta = tab_row(TP, MP, (size_t)j * P);
      TabRow tb;
      if (j >= 2) tb = tab_row(TP, MP, (size_t)(j - 1) * P);
      auto row_j = [&](int jj, const TabRow& tr) {
        const double r0 = f[(jj - 1) * NT];
        const double a = fma(-tr.h, an, fma(tr.eC, r2, fma(-tr.eB, r1, tr.eA * r0)));
        f[jj * NT] = a;
        sum = fma(tr.W, a, sum);
        an = a;
        r2 = r1;
        r1 = r0;
      };
      row_j(j, ta);
      if (j >= 2) row_j(j - 1, tb);
    }
    const size_t vo = (size_t)b * P + p;
    const double* vwn = reinterpret_cast<const double*>(pb.vw_new + vo) + r;
    const double* vwo = reinterpret_cast<const double*>(pb.vw_old + vo) + r;
    const double vw = fma(sc.theta, *vwn - *vwo, *vwo);
    const double s = fma(cc, S0, (sig == 0 ? 0.5 : -0.5) * vw);
    // w = v_p - c v_old and its wall sums
    fp = t.tau.pois_isq[(size_t)sig * P + p] * (s - sum);
    auto wall = [&](int i, double fi, double x) {
      const double w = fma(-cc, x, fi), nn = __ldg(n2 + 2 * i + sig);
      f[i * NT] = w;
      Bw = fma(nn, w, Bw);
      if (TOP) Aw = fma(nn * (nn - 1.0), w, Aw);  // 3 D^2 at the wall
    };
    wall(0, fp, Vp[(size_t)sig * hP]);
    for (int i = 1; i < M; i += 4) {
      double bb[4], x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k < M) {
          bb[k] = __ldg(TP + 4 * MP + (size_t)(i + k) * P);
          x[k] = Vp[(size_t)(2 * (i + k) + sig) * hP];
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (i + k < M) {
          fp = fma(bb[k], fp, f[(i + k) * NT]);
          wall(i + k, fp, x[k]);
        }
    }
  }
  // influence coefficient: D v(+-1) = 0 per parity, or D^2 v(+1) = Dv(-1) = 0
  double cI;
  if (TOP == 0) {
    cI = -Bw * t.tau.vh_idv[(size_t)(sc.k * 2 + sig) * P + p];
  } else {
    const int me = threadIdx.x, mate = me ^ 32;
    Aw *= 1.0 / 3.0;
    xch[me] = Aw;
    xch[NT + me] = Bw;
    __syncthreads();
    if (!live) return;
    const double Ao = xch[mate], Bo = xch[NT + mate];
    const double se[4] = {sig == 0 ? Aw : Ao, sig == 0 ? Bw : Bo, 0.0, 0.0};
    const double so[4] = {sig == 0 ? Ao : Aw, sig == 0 ? Bo : Bw, 0.0, 0.0};
    auto vs = [&](int s, int w) { return t.tau.vh_top[((size_t)(sc.k * 2 + s) * 2 + w) * P + p]; };
    double ce, co;
    close_free_slip_v(se, so, vs(0, 0), vs(1, 0), vs(0, 1), vs(1, 1), cc, &ce, &co);
    cI = sig == 0 ? ce : co;
  }
  const double* __restrict__ vh = t.tau.vh + (size_t)(sc.k * 2 + sig) * MP + p;
  for (int i = 0; i < M; i += 4) {
    double h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < M) h[k] = __ldg(vh + (size_t)(i + k) * P);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < M) Vp[(size_t)(2 * (i + k) + sig) * hP] = fma(cI, h[k], f[(i + k) * NT]);
  }
}

// CTA: 16 modes x 2 components (lanes) x 2 classes (warps) of one equation;
// v (twice the work) in the first half of the grid
template <typename RN, int TOP>
__global__ void __launch_bounds__(64, 8) stage_solve_kernel(Grid g, PencilBufs pb, DevTables t,
                                                             const typename cpx<RN>::T* __restrict__ hc, StageCoef sc) {
  extern __shared__ __align__(16) double sarr[];  // [Mh][64], then the exchange slots [6][64] of a free-slip top
  const int b = blockIdx.y;
  if (pb.active && !pb.active[b]) return;
  pdl_wait_then_release();  // the coefficients of H come from the analysis
  const int lane = threadIdx.x & 31, c = threadIdx.x / 32, r = lane & 1;
  const int pr = blockIdx.x * 16 + (lane >> 1), p = min(pr, g.P - 1);
  // a free-slip top needs every thread at the exchange
  bool live = pr < g.P && p / g.nxh != g.nz / 2;  // the Nyquist row stays zero
  double* f = sarr + threadIdx.x;
  double* xch = sarr + (size_t)t.tau.Mh * 64;
  const RN* h = reinterpret_cast<const RN*>(hc);
  if (blockIdx.z == 0) {
    if (p == 0) live = false;  // the mean flow is the other equation's
    if (TOP == 0 && !live) return;
    solve_v<RN, TOP>(f, xch, g, pb, t, sc, b, p, r, c, live, h);
  } else {
    if (TOP == 0 && !live) return;
    solve_omega<RN, TOP>(f, xch, g, pb, t, sc, b, p, r, 1 - c, live, h);
  }
}

template <typename RN, int TOP>
cudaError_t solve_top(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, const typename cpx<RN>::T* h,
                      const StageCoef& sc, cudaStream_t st) {
  const size_t smem = ((size_t)t.tau.Mh + (TOP ? 6 : 0)) * 64 * sizeof(double);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_solve_kernel<RN, TOP>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(RN) == 4>(stage_solve_kernel<RN, TOP>, dim3((g.P + 15) / 16, B, 2), dim3(64), smem, st, g, pb,
                                        t, h, sc);
}

}  // namespace chdns
