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
// The mean flow is solved for its increment d = X^k - X^{k-1} instead of
// X' = X^k + c X^{k-1}: (D^2 - lam) d = -dt (...)/(beta dt nu) - (1 + c) D^2 X.
// lam is large for the mean mode, so the solve of X' would return nearly
// (1 + c) X through a system of condition ~ (N/2)^2; the increment's error is
// smaller by |d| / |X|, and X carries most of the observation.
//
// No-slip walls: sum f' = c sum f_old per parity for omega_y, U, W; v' the
// same plus the wall velocity, and the influence correction c_I vh that fixes
// Dv.  Free-slip top (TOP = 1): the rows Df(+1) and f(-1) (omega_y, W), these
// and the flow rate (U), D^2 v(+1) and Dv(-1) (v) couple the parities, which
// are the two warps of a CTA: each publishes the sums of its parity and both
// solve the same closure.
//
// What bounds it: the FP64 pipe, 27 operations per coefficient and (mode,
// component), FP32 right-hand sides apart.  A warp-wide FP64
// operation takes the same 64 to 76 cycles of its sub-partition whatever the
// dependences, so what counts is that every sub-partition always has a warp
// whose operands are there: the coefficient array of a thread lives in a
// column of shared memory (M doubles), so that registers hold the rows in flight
// only (twelve warps per SM with three rows ahead, eight with five), the loops
// stay rolled, and the two equations are CTAs of their own.
#pragma once

#include "common.cuh"
#include "internal.h"
#include "stage_close.cuh"
#include "stage_scan.cuh"

namespace chdns {

template <int TOP> constexpr int solve_tabs() { return TOP ? 8 : 7; }  // eA, eB, eC, h, b, W, E1 (, W2)
constexpr int kPoisTabs = 6;                                           // eA, eB, eC, h, b, W

// dt (gamma h + zeta h') in the node precision; in FP32 with the coefficients as
// sums of two values: one rounding of dt gamma is the same for every mode and
// step, and such errors do not average out (v of 64x65x64 after five steps
// 8.8e-8 off with one value, 7.6e-8 with two)
template <typename RN>
__device__ __forceinline__ RN explicit_rhs(const StageCoef& sc, RN h, RN hp) {
  if constexpr (sizeof(RN) == 4) return fmaf(sc.dgaf, h, fmaf(sc.dzef, hp, fmaf(sc.dgal, h, sc.dzel * hp)));
  else return sc.dt * sc.gamma * h + sc.dt * sc.zeta * hp;
}

// Rows i = M-1 .. 0 (down) or i0 .. M-1 (up) in order, the loads of a row D
// rows ahead of its step.
// The steady part is one basic block of D loads and D steps.
template <int D, class Load, class Step>
__device__ __forceinline__ void sweep_down(int top, int last, Load&& load, Step&& step) {
  decltype(load(0)) ring[D];
#pragma unroll
  for (int k = 0; k < D; ++k) ring[k] = load(max(top - k, last));
  int i = top;
#pragma unroll 1
  for (; i - 2 * D + 1 >= last; i -= D) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const auto cur = ring[k];
      ring[k] = load(i - k - D);
      step(i - k, cur);
    }
  }
  // fewer than 2 D rows left, the first D of them loaded
  decltype(load(0)) rest[D > 1 ? D - 1 : 1];
#pragma unroll
  for (int k = 0; k < D - 1; ++k) rest[k] = load(max(i - k - D, last));
#pragma unroll
  for (int k = 0; k < D; ++k)
    if (i - k >= last) step(i - k, ring[k]);
#pragma unroll
  for (int k = 0; k < D - 1; ++k)
    if (i - k - D >= last) step(i - k - D, rest[k]);
}
template <int D, class Load, class Step>
__device__ __forceinline__ void sweep_up(int first, int M, Load&& load, Step&& step) {
  sweep_down<D>(M - 1, first, [&](int i) { return load(M - 1 + first - i); },
                [&](int i, const auto& v) { step(M - 1 + first - i, v); });
}

// one row's table entries, from tables of TABS entries a row: one address serves
// all of them and, with the row stride fixed, the rows of an unrolled block (the
// solves issue three other instructions per FP64 operation: as [entry][row][mode]
// arrays the tables took six addresses a row; 256 minimal mixed channels 1090
// us per step then and 1064 so).  The tables depend on kz^2 alone and hold the
// rows kz >= 0: modes kz and -kz share theirs.
template <int TABS> __device__ __forceinline__ const double* tab_of(const double* T, int block, const Grid& g, int Mh, int p) {
  const int row = p / g.nxh, hz = g.nz / 2, pt = row > hz ? p + (2 * (hz - row)) * g.nxh : p;
  return T + ((size_t)(block * ((g.nxh * hz + 15) / 16) + pt / 16) * Mh) * (TABS * 16) + pt % 16;
}
template <int TABS> __device__ __forceinline__ double tab(const double* __restrict__ T, int row, int entry) {
  return __ldg(T + (ptrdiff_t)(row - 1) * (TABS * 16) + entry * 16);  // rows 1 .. Mh
}
struct TabRow {
  double eA, eB, eC, h, W;
};
template <int TABS> __device__ __forceinline__ TabRow tab_row(const double* __restrict__ T, int row) {
  return TabRow{tab<TABS>(T, row, 0), tab<TABS>(T, row, 1), tab<TABS>(T, row, 2), tab<TABS>(T, row, 3), tab<TABS>(T, row, 5)};
}

// what a thread's sweep down leaves for the closure
struct Wall {
  double sum = 0.0, sum2 = 0.0;  // sum P, sum n^2 P of the particular solution
  double S0 = 0.0, S2 = 0.0;     // sum x, sum n^2 x of the old field
  double wp = 0.0, wx = 0.0;     // int P, int x (mean flow, even parity)
};

struct Bw {
  double b, w;
};

// omega_y of parity sig of one (mode, component): down
template <typename RN, int TOP, int D>
__device__ __forceinline__ Wall omega_down(double* f, const Grid& g, const PencilBufs& pb, const DevTables& t,
                                           const StageCoef& sc, int b, int p, int r, int sig, const double* __restrict__ T,
                                           const RN* __restrict__ hc) {
  constexpr int NT = 64;
  constexpr int TABS = solve_tabs<TOP>();
  const size_t P = g.P;
  const int ny = g.ny, M = (g.N - sig) / 2 + 1, row = p / g.nxh, ix = p % g.nxh;
  const double cc1 = 1.0 + sc.cc;
  const double* __restrict__ n2 = t.tau.n2;
  // element n of a component column: base + 2 P n
  const size_t hP = 2 * P, base = 2 * ((size_t)b * ny * P + p) + r;
  const double* G = reinterpret_cast<const double*>(pb.G) + base;
  RN* HG = reinterpret_cast<RN*>(pb.HGP) + base;
  const RN* hx = hc + 2 * (b * g.qb + p) + 1 - r;
  const RN* hz = hx + 4 * g.qf;
  const size_t hS = 2 * g.qj;
  const RN sgn = r == 0 ? (RN)-1 : (RN)1, kx = sgn * (RN)t.kx[ix], kz = sgn * (RN)t.kz[row];
  struct In {
    double x;
    RN hx, hz, hp;
    TabRow tb;
    double W2;
  };
  Wall w;
  double r1 = 0.0, r2 = 0.0, an = 0.0;
  sweep_down<D>(
      M - 1, 0,
      [&](int i) {
        In v;
        const size_t n = 2 * i + sig;
        v.x = G[n * hP];
        v.hx = __ldg(hx + n * hS);
        v.hz = __ldg(hz + n * hS);
        v.hp = HG[n * hP];
        v.tb = tab_row<TABS>(T, i + 1);  // row i + 1 of the elimination (row M is not used)
        if (TOP) v.W2 = tab<TABS>(T, i + 1, 7);
        return v;
      },
      [&](int i, const In& v) {
        const size_t n = 2 * i + sig;
        const RN hg = kz * v.hx - kx * v.hz;
        HG[n * hP] = hg;
        w.S0 += v.x;
        if (TOP) w.S2 = fma(__ldg(n2 + n), v.x, w.S2);
        const double r0 = fma(cc1, v.x, widen(explicit_rhs<RN>(sc, hg, v.hp)));
        if (i + 1 < M) {
          const double a = fma(-v.tb.h, an, fma(v.tb.eC, r2, fma(-v.tb.eB, r1, v.tb.eA * r0)));
          f[(i + 1) * NT] = a;
          w.sum = fma(v.tb.W, a, w.sum);
          if (TOP) w.sum2 = fma(v.W2, a, w.sum2);
          an = a;
        }
        r2 = r1;
        r1 = r0;
      });
  return w;
}

// The mean flow (component 0: U, 1: W) of parity sig, in the lanes of mode 0:
// down, for the increment.  X: coefficients, XP: previous plane means of H,
// hm: its new ones (2 qj apart).
template <typename RN, int TOP>
__device__ __forceinline__ Wall mean_down(double* f, const DevTables& t, const StageCoef& sc, int N, size_t qj, int sig,
                                       const double* __restrict__ T, const double* X, double* XP,
                                       const RN* __restrict__ hm) {
  constexpr int NT = 64;
  constexpr int TABS = solve_tabs<TOP>();
  const int M = (N - sig) / 2 + 1;
  const double bdn = sc.beta * sc.dt * sc.nu;
  Wall w;
  double r1 = 0.0, r2 = 0.0, an = 0.0, x1 = 0.0;
  struct In {
    double x, hp, n2, wi;
    RN h;
    TabRow tb;
    double E1, W2;
  };
  sweep_down<4>(
      M - 1, 0,
      [&](int i) {
        In v;
        const int n = 2 * i + sig;
        v.x = X[n];
        v.hp = XP[n];
        v.h = __ldg(hm + 2 * qj * n);
        v.wi = __ldg(t.tau.wint + n);
        v.tb = tab_row<TABS>(T, i + 1);
        v.E1 = tab<TABS>(T, i + 1, 6);
        if (TOP) {
          v.n2 = __ldg(t.tau.n2 + n);
          v.W2 = tab<TABS>(T, i + 1, 7);
        }
        return v;
      },
      [&](int i, const In& v) {
        const double h = widen(v.h);
        XP[2 * i + sig] = h;
        w.S0 += v.x;
        if (TOP) w.S2 = fma(v.n2, v.x, w.S2);
        w.wx = fma(v.wi, v.x, w.wx);
        const double r0 = sc.dt * fma(sc.gamma, h, sc.zeta * v.hp);
        if (i + 1 < M) {
          const double a = fma(v.E1, bdn * x1, fma(-v.tb.h, an, fma(v.tb.eC, r2, fma(-v.tb.eB, r1, v.tb.eA * r0))));
          f[(i + 1) * NT] = a;
          w.sum = fma(v.tb.W, a, w.sum);
          if (TOP) w.sum2 = fma(v.W2, a, w.sum2);
          an = a;
        }
        r2 = r1;
        r1 = r0;
        x1 = v.x;
      });
  if (TOP && sig == 0) {
    double fp = 0.0;
    sweep_up<4>(
        1, M, [&](int i) { return Bw{tab<TABS>(T, i, 4), __ldg(t.tau.wint + 2 * i)}; },
        [&](int i, const Bw& v) {
          fp = fma(v.b, fp, f[i * NT]);
          w.wp = fma(v.w, fp, w.wp);
        });
  }
  return w;
}

// up: X <- X + d (+ the response u1 to the forcing of U).  X32 (mixed precision):
// FP32 copies of X, 2 P apart; X then also takes its column f.
template <int TOP>
__device__ __forceinline__ void mean_up(double* f, const DevTables& t, const StageCoef& sc, int N, size_t P, int sig,
                                     bool forced, const double* __restrict__ T, double* X, float* X32, double f0,
                                     double fc, double wx) {
  constexpr int NT = 64;
  constexpr int TABS = solve_tabs<TOP>();
  const int M = (N - sig) / 2 + 1;
  double fp = f0, flux = t.tau.wint[0] * f0;
  f[0] = f0;
  sweep_up<4>(
      1, M, [&](int i) { return Bw{tab<TABS>(T, i, 4), __ldg(t.tau.wint + 2 * i)}; },
      [&](int i, const Bw& v) {
        fp = fma(v.b, fp, f[i * NT]);
        f[i * NT] = fp;
        flux = fma(v.w, fp, flux);
      });
  if (TOP == 0) fc = (sc.flux - wx - flux) * t.tau.u1_iflux[sc.k];
  if (!forced || sig != 0) fc = 0.0;
  const double* u1 = t.tau.u1 + (size_t)sc.k * t.tau.Mh;
  sweep_up<4>(
      0, M, [&](int i) { return Bw{X[2 * i + sig], __ldg(u1 + i)}; },
      [&](int i, const Bw& v) {
        const double x = fma(fc, v.w, v.b + f[i * NT]);
        X[2 * i + sig] = x;
        if (X32) {
          X32[2 * P * (2 * i + sig)] = narrow(x);
          f[i * NT] = x;
        }
      });
}

// mean_shear (stage_scan.cuh) of a column x of up to 16 K coefficients
template <int K>
__device__ __forceinline__ void mean_shear_of(const double* x, const DevTables& t, int N, size_t P, int sig, int q, float* D32) {
  constexpr int NT = 64;
  static_assert(7 * kLanes > kMaxNy / 2, "a column fits the lanes");
  const int M = (N - sig) / 2 + 1, i0 = (kLanes - q) * K - 1;
  double v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = i0 - k < M ? x[(i0 - k) * NT] : 0.0;
  mean_shear<K>(v, N, sig, i0, t.tau.n1, q, D32, P);
}

// Solve omega_y of parity sig of one (mode, component), or (MEAN) the mean flow
// (component 0: U at constant flow rate, 1: W).
template <typename RN, int TOP, int D, bool MEAN>
__device__ __forceinline__ void solve_omega(double* f, double* xch, const Grid& g, const PencilBufs& pb,
                                            const DevTables& t, const StageCoef& sc, int b, int p, int r, int sig,
                                            bool live, const RN* __restrict__ hc) {
  constexpr int NT = 64;
  constexpr int TABS = solve_tabs<TOP>();
  const size_t P = g.P;
  const int ny = g.ny, M = (g.N - sig) / 2 + 1;
  const double* __restrict__ T = tab_of<TABS>(t.tau.helm_f, sc.k * 2 + sig, g, t.tau.Mh, p);
  double* X = (r == 0 ? pb.UM : pb.WM) + (size_t)b * ny;
  Wall w;
  if (live) {
    if constexpr (MEAN) {
      const RN* hm = hc + 2 * b * g.qb + (r == 0 ? 0 : 4 * g.qf);
      w = mean_down<RN, TOP>(f, t, sc, g.N, g.qj, sig, T, X, (r == 0 ? pb.HXP : pb.HZP) + (size_t)b * ny, hm);
    } else {
      w = omega_down<RN, TOP, D>(f, g, pb, t, sc, b, p, r, sig, T, hc);
    }
  }
  const double cx = MEAN ? -1.0 : sc.cc;  // the wall rows of X' take c X, those of d take -X
  double f0, fc = 0.0;
  if (TOP == 0) {
    f0 = t.tau.helm_isq[(size_t)(sc.k * 2 + sig) * P + p] * (cx * w.S0 - w.sum);
  } else {
    const int me = threadIdx.x, mate = me ^ 32;
    const double mine[6] = {w.sum, w.sum2, w.S0, w.S2, w.wp, w.wx};
#pragma unroll
    for (int k = 0; k < 6; ++k) xch[k * NT + me] = mine[k];
    __syncthreads();
    if (!live && !(MEAN && sizeof(RN) == 4)) return;
    double se[6], so[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const double other = xch[k * NT + mate];
      se[k] = sig == 0 ? mine[k] : other;
      so[k] = sig == 0 ? other : mine[k];
    }
    auto qs = [&](int s, int w) { return t.tau.helm_top[((size_t)(sc.k * 2 + s) * 2 + w) * P + p]; };
    double xe, xo;
    if (MEAN && r == 0) {
      const double* m = t.tau.mean_top + 4 * sc.k;  // int Q_e; sum, sum n^2 and int of the forcing response
      close_free_slip_mean(se, so, qs(0, 0), qs(1, 0), qs(0, 1), qs(1, 1), m[0], m[1], m[2], m[3], cx, sc.flux, &xe, &xo,
                           &fc);
    } else {
      close_neumann_top(se, so, qs(0, 0), qs(1, 0), qs(0, 1), qs(1, 1), cx, &xe, &xo);
    }
    f0 = sig == 0 ? xe : xo;
  }
  if constexpr (MEAN) {
    // the FP32 copies go to the columns of mode 0: (W, U) and (DW, DU)
    const size_t col = 2 * (size_t)b * ny * P;
    float* X32 = sizeof(RN) == 4 ? reinterpret_cast<float*>(pb.G32) + col + (1 - r) : nullptr;
    if (live) mean_up<TOP>(f, t, sc, g.N, P, sig, r == 0, T, X, X32, f0, fc, w.wx);
    if constexpr (sizeof(RN) == 4) {
      // sixteen lanes of the warp on each of its two columns (as a loop of the two
      // threads the mean flow outlasted v: 16x201x16 x 8 557 us a step, 583 so)
      __syncwarp();
      const int q = threadIdx.x % kLanes, c = threadIdx.x % 32 / kLanes;
      const double* x = f - threadIdx.x % 32 + c;
      float* D32 = reinterpret_cast<float*>(pb.V32) + col + (1 - c);
      if (M <= 3 * kLanes) mean_shear_of<3>(x, t, g.N, P, sig, q, D32);
      else mean_shear_of<7>(x, t, g.N, P, sig, q, D32);
    }
    return;
  }
  // up: f_i = a_i + b_i f_{i-1}; g <- f - c g
  const size_t hP = 2 * P;
  const size_t base = 2 * ((size_t)b * ny * P + p) + r + (size_t)sig * hP;
  double* G = reinterpret_cast<double*>(pb.G) + base;
  float* G32 = reinterpret_cast<float*>(pb.G32) + base;
  const double cc = sc.cc;
  double fp = f0;
  auto put = [&](int i, double v) {
    G[(size_t)i * 2 * hP] = v;
    if constexpr (sizeof(RN) == 4) G32[(size_t)i * 2 * hP] = narrow(v);
  };
  put(0, fma(-cc, G[0], fp));
  struct Up {
    double b, x;
  };
  sweep_up<2 * D>(
      1, M, [&](int i) { return Up{tab<TABS>(T, i, 4), G[(size_t)i * 2 * hP]}; },
      [&](int i, const Up& u) {
        fp = fma(u.b, fp, f[i * NT]);
        put(i, fma(-cc, u.x, fp));
      });
}

// Solve v of parity sig of one (mode, component).
template <typename RN, int TOP, int D>
__device__ __forceinline__ void solve_v(double* f, double* xch, const Grid& g, const PencilBufs& pb, const DevTables& t,
                                        const StageCoef& sc, int b, int p, int r, int sig, bool live,
                                        const RN* __restrict__ hc) {
  constexpr int NT = 64;
  const size_t P = g.P, MP = (size_t)t.tau.Mh * P;
  const int ny = g.ny, N = g.N, M = (N - sig) / 2 + 1, row = p / g.nxh, ix = p % g.nxh;
  const double cc = sc.cc;
  constexpr int TABS = solve_tabs<TOP>();
  const double* __restrict__ T = tab_of<TABS>(t.tau.helm_f, sc.k * 2 + sig, g, t.tau.Mh, p);
  const double* __restrict__ TP = tab_of<kPoisTabs>(t.tau.pois_f, sig, g, t.tau.Mh, p);
  const double* __restrict__ n2 = t.tau.n2;
  const size_t hP = 2 * P, base = 2 * ((size_t)b * ny * P + p) + r;
  double* Vp = reinterpret_cast<double*>(pb.V) + base;
  RN* HV = reinterpret_cast<RN*>(pb.HVP) + base;
  float* V32 = reinterpret_cast<float*>(pb.V32) + base;
  const RN* H0 = hc + 2 * (b * g.qb + p);
  const RN* hx = H0 + 1 - r;
  const RN* hy = H0 + 2 * g.qf + r;
  const RN* hz = H0 + 4 * g.qf + 1 - r;
  const size_t hS = 2 * g.qj;
  const double kxd = t.kx[ix], kzd = t.kz[row], k2 = fma(kxd, kxd, kzd * kzd), ck2 = -(1.0 + cc) * k2;
  const RN sgn = r == 0 ? (RN)-1 : (RN)1, kx = sgn * (RN)kxd, kz = sgn * (RN)kzd, k2n = (RN)k2;
  double Aw = 0.0, Bw = 0.0;
  if (live) {
    struct In {
      double x;
      RN hx, hy, hz, hp, fac;
      TabRow tb;
      double E1;
    };
    auto load = [&](int i) {
      In v;
      const size_t n = 2 * i + sig;
      v.x = Vp[n * hP];
      v.hy = __ldg(hy + n * hS);
      v.hp = HV[n * hP];
      if constexpr (sizeof(RN) == 8) v.fac = __ldg(t.tau.n1 + n);
      else v.fac = (RN)(2 * ((int)n + 1));
      const size_t no = min((int)n + 1, N);
      v.hx = __ldg(hx + no * hS);
      v.hz = __ldg(hz + no * hS);
      v.tb = tab_row<TABS>(T, i + 1);
      v.E1 = tab<TABS>(T, i + 1, 6);
      return v;
    };
    double S0 = 0.0, sum = 0.0, r1 = 0.0, r2 = 0.0, x1 = 0.0, an = 0.0;
    RN dtt = 0;  // D(i kx H_x + i kz H_z), from the top down
    auto step = [&](int i, const In& v) {
      const int n = 2 * i + sig;
      const RN tt = n + 1 <= N ? kx * v.hx + kz * v.hz : (RN)0;
      const RN t2 = v.fac * tt + dtt;
      dtt = n == 0 ? (RN)0.5 * t2 : t2;
      const RN hv = -k2n * v.hy - dtt;
      HV[(size_t)n * hP] = hv;
      const RN q = explicit_rhs<RN>(sc, hv, v.hp);
      S0 += v.x;
      const double r0 = fma(ck2, v.x, widen(q));
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
    sweep_down<D>(M - 1, 0, load, step);
    // phi, with zero wall sum
    double fp = t.tau.helm_isq[(size_t)(sc.k * 2 + sig) * P + p] * -sum;
    f[0] = fp;
    sweep_up<2 * D>(
        1, M, [&](int i) { return tab<TABS>(T, i, 4); },
        [&](int i, double bi) {
          fp = fma(bi, fp, f[i * NT]);
          f[i * NT] = fp;
        });
    // (D^2 - k^2) v_p = phi, the array read at i and written at i + 1
    sum = an = r2 = 0.0;
    r1 = fp;
    sweep_down<D>(
        M - 1, 1, [&](int j) { return tab_row<kPoisTabs>(TP, j); },
        [&](int j, const TabRow& tr) {
          const double r0 = f[(j - 1) * NT];
          const double a = fma(-tr.h, an, fma(tr.eC, r2, fma(-tr.eB, r1, tr.eA * r0)));
          f[j * NT] = a;
          sum = fma(tr.W, a, sum);
          an = a;
          r2 = r1;
          r1 = r0;
        });
    const size_t vo = (size_t)b * P + p;
    const double* vwn = reinterpret_cast<const double*>(pb.vw_new + vo) + r;
    const double* vwo = reinterpret_cast<const double*>(pb.vw_old + vo) + r;
    const double vw = fma(sc.theta, *vwn - *vwo, *vwo);
    const double s = fma(cc, S0, (sig == 0 ? 0.5 : -0.5) * vw);
    // w = v_p - c v_old and its wall sums
    fp = t.tau.pois_isq[(size_t)sig * P + p] * (s - sum);
    auto wall = [&](int i, double fi, double x, double nn) {
      const double w = fma(-cc, x, fi);
      f[i * NT] = w;
      Bw = fma(nn, w, Bw);
      if (TOP) Aw = fma(nn * (nn - 1.0), w, Aw);  // 3 D^2 at the wall
    };
    wall(0, fp, Vp[(size_t)sig * hP], __ldg(n2 + sig));
    struct Up {
      double b, x, nn;
    };
    sweep_up<D>(
        1, M,
        [&](int i) {
          return Up{tab<kPoisTabs>(TP, i, 4), Vp[(size_t)(2 * i + sig) * hP], __ldg(n2 + 2 * i + sig)};
        },
        [&](int i, const Up& u) {
          fp = fma(u.b, fp, f[i * NT]);
          wall(i, fp, u.x, u.nn);
        });
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
  sweep_up<2 * D>(
      0, M, [&](int i) { return __ldg(vh + (size_t)i * P); },
      [&](int i, double h) {
        const size_t o = (size_t)(2 * i + sig) * hP;
        const double v = fma(cI, h, f[i * NT]);
        Vp[o] = v;
        if constexpr (sizeof(RN) == 4) V32[o] = narrow(v);
      });
}

// CTA: 16 modes x 2 components (lanes) x 2 classes (warps) of one equation:
// the mean flow, then v (twice the work of omega_y), then omega_y.  D rows are
// loaded ahead: three on 168 registers (six CTAs per SM up to 147 nodes, five up
// to 175), five on up to 255 where the grid or the columns leave four or fewer.
// us per step with 3 / 5, the implicit half and all else: 16x65x16 x 256 mixed
// 1205 / 1302, 128x129x128 mixed 764 / 807, 16x171x16 x 128 mixed 3584 / 3660,
// 64x65x64 x 4 FP64 2970 / 3066; 64x148x64 x 2 mixed 963 / 938, 24x50x48 x 8
// mixed 316 / 314, 64x65x64 FP64 945 / 946.  Under a free-slip top, where three
// rows spill (344 bytes mixed, 520 FP64): 16x65x16 x 128 mixed 781 / 812,
// 64x65x64 x 4 mixed 479 / 560 and FP64 3014 / 3104, 16x65x16 x 128 FP64 4732 /
// 4704.
template <typename RN, int TOP, int D>
__global__ void __launch_bounds__(64, D == 3 ? 6 : 4) stage_solve_kernel(Grid g, PencilBufs pb, DevTables t,
                                                            const typename cpx<RN>::T* __restrict__ hc, StageCoef sc) {
  extern __shared__ __align__(16) double sarr[];  // [Mh][64], then the exchange slots [6][64] of a free-slip top
  const int b = blockIdx.y, tiles = (g.P + 15) / 16;
  if (pb.active && !pb.active[b]) return;
  const int lane = threadIdx.x & 31, c = threadIdx.x / 32, r = lane & 1;
  const int z = (blockIdx.x + tiles - 1) / tiles;  // 0: mean, 1: v, 2: omega_y
  const int pr = z == 0 ? lane >> 1 : ((int)(blockIdx.x - 1) % tiles) * 16 + (lane >> 1), p = min(pr, g.P - 1);
  // the mean flow is mode 0; the Nyquist row stays zero
  const bool live = z == 0 ? lane < 2 : pr > 0 && pr < g.P && p / g.nxh != g.nz / 2;
  // a free-slip top needs every thread at the exchange, the FP32 copy of the mean
  // shear every lane
  if (TOP == 0 && !live && !(z == 0 && sizeof(RN) == 4)) return;
  double* f = sarr + threadIdx.x;
  double* xch = sarr + (size_t)t.tau.Mh * 64;
  const RN* h = reinterpret_cast<const RN*>(hc);
  if (z == 0) solve_omega<RN, TOP, D, true>(f, xch, g, pb, t, sc, b, p, r, c, live, h);
  else if (z == 1) solve_v<RN, TOP, D>(f, xch, g, pb, t, sc, b, p, r, c, live, h);
  else solve_omega<RN, TOP, D, false>(f, xch, g, pb, t, sc, b, p, r, 1 - c, live, h);
}

template <typename RN, int TOP, int D>
cudaError_t solve_ahead(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, const typename cpx<RN>::T* h,
                        const StageCoef& sc, dim3 grid, size_t smem, cudaStream_t st) {
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_solve_kernel<RN, TOP, D>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(stage_solve_kernel<RN, TOP, D>, grid, dim3(64), smem, st, g, pb, t, h, sc);
}

template <typename RN, int TOP>
cudaError_t solve_top(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, const typename cpx<RN>::T* h,
                      const StageCoef& sc, cudaStream_t st) {
  const size_t smem = ((size_t)t.tau.Mh + (TOP ? 6 : 0)) * 64 * sizeof(double);
  const dim3 grid(1 + 2 * ((g.P + 15) / 16), B);
  if ((long)grid.x * grid.y > 4 * 152 && smem <= (size_t)44 * 1024)
    return solve_ahead<RN, TOP, 3>(g, B, pb, t, h, sc, grid, smem, st);
  return solve_ahead<RN, TOP, 5>(g, B, pb, t, h, sc, grid, smem, st);
}

}  // namespace chdns
