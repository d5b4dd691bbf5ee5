// The no-slip implicit solves of one (mode, class, component, equation) spread
// over a group of kLanes lanes, for handles with too few modes to fill the GPU
// with one thread per system (fewer than 768 in a batch).
//
// Lane q of the group holds the block of coefficient indices
//   i = MH - 1 - q K - k,  k = 0 .. K - 1,  K = ceil(MH / kLanes),
// so lane 0 holds the top of the spectrum.  Every sequential sweep of the
// single-thread solve becomes a block sweep plus a combination across the
// lanes:
//   - sums (wall rows, influence and flux sums): block sums, then a fixed
//     butterfly over the group;
//   - running sums from the top (the derivative walk of t): block prefix sums
//     plus the inclusive prefix of the block totals of the lanes above;
//   - the first-order recurrences of the tau elimination, a_j = alpha_j -
//     h_j a_{j+1} (downwards) and P_i = b_i P_{i-1} + a_i (upwards): each
//     block composes its affine maps, a Kogge-Stone scan composes the maps of
//     the lanes before it, and the block is swept again from its true input.
// A warp-wide FP64 operation takes 64 cycles of its sub-partition whatever its
// dependences and active lanes, so the time of such a handle is the number of
// operations a warp issues: sixteen lanes (three coefficients each at 65
// nodes) and four warps per mode, one per sub-partition, in place of four
// lanes and one warp take 190 operations for v instead of 344 and run omega_y
// beside it instead of before it.  Sums are formed in another order than the
// single-thread form, so the two forms agree to rounding, not bitwise.
#pragma once

#include "common.cuh"

namespace chdns {

constexpr int kLanes = 16;

namespace scanl {

// the lanes of this thread's group (groups of a warp may take different
// paths: every shuffle names only its own group)
__device__ __forceinline__ unsigned group_mask() {
  return (kLanes == 32 ? 0xffffffffu : (1u << kLanes) - 1u) << (threadIdx.x & (32u - kLanes));
}

// sum over the lanes of the group, the same bits on every lane
__device__ __forceinline__ double lane_sum(double x) {
  const unsigned m = group_mask();
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) x = x + __shfl_xor_sync(m, x, o, kLanes);
  return x;
}

// exclusive prefix over lanes 0 .. q - 1 of a per-lane total
template <typename T>
__device__ __forceinline__ T lanes_above(T tot, int q) {
  const unsigned m = group_mask();
  T inc = tot;
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
    const T v = __shfl_up_sync(m, inc, o, kLanes);
    if (q >= o) inc = inc + v;
  }
  const T ex = __shfl_up_sync(m, inc, 1, kLanes);
  return q == 0 ? (T)0 : ex;
}

// The input of lane q's block for a chain x -> A + B x composed block by
// block: downwards (lane 0 first, down = true) or upwards (the last lane first); the
// first block's input is 0.
__device__ __forceinline__ double chain_input(double A, double B, int q, bool down) {
  const unsigned m = group_mask();
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
    const double Ap = down ? __shfl_up_sync(m, A, o, kLanes) : __shfl_down_sync(m, A, o, kLanes);
    const double Bp = down ? __shfl_up_sync(m, B, o, kLanes) : __shfl_down_sync(m, B, o, kLanes);
    if (down ? q >= o : q + o < kLanes) {
      A = fma_rn(B, Ap, A);  // (A, B) after (Ap, Bp)
      B = mul_rn(B, Bp);
    }
  }
  const double in = down ? __shfl_up_sync(m, A, 1, kLanes) : __shfl_down_sync(m, A, 1, kLanes);
  return (down ? q == 0 : q == kLanes - 1) ? 0.0 : in;
}

}  // namespace scanl

template <int MH>
struct Blk {
  static constexpr int K = (MH + kLanes - 1) / kLanes;
  __device__ static constexpr int i_of(int q, int k) { return MH - 1 - q * K - k; }
};

// Chebyshev-tau Dirichlet solve (tau_seq's rows) over a lane group.  On
// entry f[k] holds r at i = i_of(q, k) (0 outside 0 .. M - 1); on return the
// solution f_i, with the wall row sum_i f_i = wall.
// With DIAG, row j also takes diag[k] (a term whose stencil is its own value).
template <int MH, bool DIAG = false, class Tab>
__device__ __forceinline__ void tau_scan(int N, int ny, int sig, double (&f)[Blk<MH>::K], const Tab& T, double isq,
                                         double wall, const double* __restrict__ rowc, int q,
                                         const double* diag = nullptr) {
  constexpr int K = Blk<MH>::K;
  const int M = (N - sig) / 2 + 1;
  // neighbours across the block edges: r at hi + 1 (bottom of the lane above)
  // and at lo - 1 (top of the lane below)
  const unsigned m = scanl::group_mask();
  const double above = __shfl_up_sync(m, f[K - 1], 1, kLanes), below = __shfl_down_sync(m, f[0], 1, kLanes);
  const double r_above = q == 0 ? 0.0 : above;
  const double r_below = q == kLanes - 1 ? 0.0 : below;
  // alpha_j = e_j R_j in place (r_{j+1} kept from the previous step), and the
  // block's map a_bottom = A + B a_in
  double A = 0.0, B = 1.0;
  double r_up = r_above;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int j = Blk<MH>::i_of(q, k);
    const double rj = f[k];
    const double rlo = k + 1 < K ? f[k + 1] : r_below;
    if (j >= 1 && j < M) {
      const int n = 2 * j + sig;
      double R = fma_rn(-rowc[ny + n], rj, mul_rn(rowc[n], rlo));
      if (j + 1 < M) R = fma_rn(rowc[2 * ny + n], r_up, R);
      if (DIAG) R = R + diag[k];
      const double al = mul_rn(T.e(j), R);
      const double be = -T.h(j);
      f[k] = al;
      A = fma_rn(be, A, al);
      B = mul_rn(be, B);
    }
    r_up = rj;
  }
  double a = scanl::chain_input(A, B, q, true);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int j = Blk<MH>::i_of(q, k);
    if (j >= 1 && j < M) {
      a = fma_rn(-T.h(j), a, f[k]);
      f[k] = a;
    }
  }
  // upwards: P_i = b_i P_{i-1} + a_i from P_0 = 0; the block map and then the sweep
  A = 0.0;
  B = 1.0;
#pragma unroll
  for (int k = K - 1; k >= 0; --k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 1 && i < M) {
      A = fma_rn(T.b(i), A, f[k]);
      B = mul_rn(T.b(i), B);
    }
  }
  double Pp = scanl::chain_input(A, B, q, false);
  double s = 0.0;
#pragma unroll
  for (int k = K - 1; k >= 0; --k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 1 && i < M) {
      Pp = fma_rn(T.b(i), Pp, f[k]);
      f[k] = Pp;
      s += Pp;
    }
  }
  const double f0 = mul_rn(isq, wall - scanl::lane_sum(s));
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i == 0) f[k] = f0;
    else if (i >= 1 && i < M) f[k] = fma_rn(T.Q(i), f0, f[k]);
  }
}

// omega_y of parity sq over a lane group
template <int MH, typename RN, class GV, class HV, class Tab>
__device__ __forceinline__ void omega_scan(int N, int ny, int ppc, int sq, const GV& Gc, const HV& HGc,
                                           const typename cpx<RN>::T* Hx, const typename cpx<RN>::T* Hz, int r,
                                           double sgn, double kx, double kz, double cc, const StageCoef& sc,
                                           const Tab& T, double isq, const double* __restrict__ rowc, int q) {
  using CN = typename cpx<RN>::T;
  constexpr int K = Blk<MH>::K;
  const int ra = 1 - r;
  auto comp = [](const CN z, int qd) { return qd == 0 ? z.x : z.y; };
  const RN sgnn = (RN)sgn, kxn = (RN)kx, kzn = (RN)kz;
  const RN dtn = (RN)sc.dt, gan = (RN)sc.gamma, zen = (RN)sc.zeta;
  const int M = (N - sq) / 2 + 1;
  double f[K];
  double sum = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    f[k] = 0.0;
    if (i >= 0 && i < M) {
      const int n = 2 * i + sq;
      const double gn = Gc[n];
      const RN hg = mul_rn(sgnn, fma_rn(-kxn, comp(Hz[n * ppc], ra), mul_rn(kzn, comp(Hx[n * ppc], ra))));
      const RN hp = HGc[n];
      HGc[n] = hg;
      const RN qv = mul_rn(dtn, fma_rn(gan, hg, mul_rn(zen, hp)));
      f[k] = fma_rn(1.0 + cc, gn, (double)qv);
      sum += gn;
    }
  }
  tau_scan<MH>(N, ny, sq, f, T, isq, mul_rn(cc, scanl::lane_sum(sum)), rowc, q);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 0 && i < M) {
      const int n = 2 * i + sq;
      Gc[n] = fma_rn(-cc, Gc[n], f[k]);
    }
  }
}

// v of parity sv over a lane group: the derivative walk as running sums from
// the top, the phi solve, the Poisson solve and the influence correction
template <int MH, typename RN, class VV, class HV, class Tab, class TabP>
__device__ __forceinline__ void v_scan(int N, int ny, int ppc, int sv, const VV& Vc, const HV& HVc,
                                       const typename cpx<RN>::T* Hx, const typename cpx<RN>::T* Hy,
                                       const typename cpx<RN>::T* Hz, int r, double sgn, double kx, double kz,
                                       double k2, double cc, const StageCoef& sc, const Tab& Th, double isq_h,
                                       const TabP& Tp, double isq_p, const double* vh, int vhs, double idv,
                                       double vw, const double* __restrict__ rowc, int q) {
  using CN = typename cpx<RN>::T;
  constexpr int K = Blk<MH>::K;
  const int ra = 1 - r;
  auto comp = [](const CN z, int qd) { return qd == 0 ? z.x : z.y; };
  const RN dsvn = (RN)(2 * sv);
  const RN sgnn = (RN)sgn, kxn = (RN)kx, kzn = (RN)kz, k2n = (RN)k2;
  const RN dtn = (RN)sc.dt, gan = (RN)sc.gamma, zen = (RN)sc.zeta;
  const int M = (N - sv) / 2 + 1;
  const double ck2 = -(1.0 + cc) * k2;
  double f[K], dg[K], nn[K];  // nn: n^2
  RN tk[K];
  // Dt: running sum from the top of 2 (n + 1) t_{n+1}
  RN dtt = (RN)0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    const int no = 2 * i + sv + 1;
    if (i >= 0 && i < M && no <= N) {
      const RN t = mul_rn(sgnn, fma_rn(kxn, comp(Hx[no * ppc], ra), mul_rn(kzn, comp(Hz[no * ppc], ra))));
      dtt = fma_rn((RN)(4 * i + 2) + dsvn, t, dtt);
    }
    tk[k] = dtt;
  }
  const RN dt_off = scanl::lanes_above(dtt, q);
  // right-hand sides of the phi solve: the stencil of D^2 v is v itself, a
  // diagonal term (stage_solve.cuh), and u = -(1 + c) k^2 v + dt (...); the wall
  // sums of the old field
  double S0 = 0.0, S2 = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    const int n = 2 * i + sv;
    f[k] = dg[k] = nn[k] = 0.0;
    if (i >= 0 && i < M) {
      nn[k] = (double)(n * n);
      RN dt2 = tk[k] + dt_off;
      if (n == 0) dt2 = (RN)0.5 * dt2;
      const double vn = Vc[n];
      S0 += vn;
      S2 = fma_rn(nn[k], vn, S2);
      const RN hv = fma_rn(-k2n, comp(Hy[n * ppc], r), -dt2);
      const RN hp = HVc[n];
      HVc[n] = hv;
      const RN qv = mul_rn(dtn, fma_rn(gan, hv, mul_rn(zen, hp)));
      f[k] = fma_rn(ck2, vn, (double)qv);
      dg[k] = mul_rn(1.0 + cc, vn);
    }
  }
  S0 = scanl::lane_sum(S0);
  S2 = scanl::lane_sum(S2);
  tau_scan<MH, true>(N, ny, sv, f, Th, isq_h, 0.0, rowc, q, dg);
  const double s = fma_rn(cc, S0, ((sv == 0) ? 0.5 : -0.5) * vw);
  tau_scan<MH>(N, ny, sv, f, Tp, isq_p, s, rowc, q);
  double dp = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 0 && i < M) dp = fma_rn(nn[k], f[k], dp);
  }
  const double cI = mul_rn(fma_rn(cc, S2, -scanl::lane_sum(dp)), idv);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 0 && i < M) {
      const int n = 2 * i + sv;
      Vc[n] = fma_rn(-cc, Vc[n], fma_rn(cI, vh[i * vhs], f[k]));
    }
  }
}

// The FP32 copy of the derivative of the mean flow from the coefficients x[k] of
// index i0 - k (n = 2 i + s; 0 outside the parity) on the lanes of a group: sums
// of 2 n X_n from the top in FP64, each rounded once.  Coefficients 2 P apart;
// n1[n] = 2 (n + 1).
template <int K>
__device__ __forceinline__ void mean_shear(double (&x)[K], int N, int s, int i0, const double* __restrict__ n1, int q,
                                           float* D32, size_t P) {
  const int M = (N - s) / 2 + 1;
  double d = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int n = 2 * (i0 - k) + s;
    d = fma_rn(__ldg(n1 + min(max(n - 1, 0), N)), x[k], d);
    x[k] = d;
  }
  const double above = scanl::lanes_above(d, q);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = i0 - k, n = 2 * i + s;
    if (i < 0 || i >= M || n < 1) continue;
    double b = x[k] + above;
    if (n == 1) b = 0.5 * b;
    D32[2 * P * (n - 1)] = narrow(b);
  }
  if (q == 0 && ((N - s) & 1)) D32[2 * P * N] = 0.0f;
}

// mean flow of parity s over a lane group, solved for its increment
// d = X^k - X^{k-1} (see stage_solve.cuh): right-hand side dt (...), and
// (1 + c) beta dt nu X on the diagonal for (1 + c) D^2 X.  D32, mixed precision:
// mean_shear
template <int MH, typename RN, class Tab>
__device__ __forceinline__ void mean_scan(int N, int ny, int ppc, int s, int e, double* X, double* XP,
                                          const typename cpx<RN>::T* Hm, double cc, const StageCoef& sc,
                                          const Tab& T, double isq, const double* __restrict__ rowc,
                                          const double* __restrict__ u1, double u1_iflux,
                                          const double* __restrict__ wint, const double* __restrict__ n1, int q,
                                          float* D32, size_t P) {
  constexpr int K = Blk<MH>::K;
  const int M = (N - s) / 2 + 1;
  double f[K], dg[K];
  const double cb = (1.0 + cc) * sc.beta * sc.dt * sc.nu;
  double sum = 0.0, flux_old = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    f[k] = dg[k] = 0.0;
    if (i >= 0 && i < M) {
      const int n = 2 * i + s;
      const double xn = X[n];
      const double hv = (double)Hm[n * ppc].x;
      const double hp = XP[n];
      XP[n] = hv;
      sum += xn;
      if (s == 0) flux_old = fma_rn(wint[n], xn, flux_old);
      f[k] = mul_rn(sc.dt, fma_rn(sc.gamma, hv, mul_rn(sc.zeta, hp)));
      dg[k] = mul_rn(cb, xn);
    }
  }
  flux_old = scanl::lane_sum(flux_old);
  tau_scan<MH, true>(N, ny, s, f, T, isq, -scanl::lane_sum(sum), rowc, q, dg);
  double fc = 0.0;
  if (e == 0 && s == 0) {
    double flux = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = Blk<MH>::i_of(q, k);
      if (i >= 0 && i < M) flux = fma_rn(wint[2 * i], f[k], flux);
    }
    fc = mul_rn(sc.flux - flux_old - scanl::lane_sum(flux), u1_iflux);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = Blk<MH>::i_of(q, k);
    if (i >= 0 && i < M) {
      const int n = 2 * i + s;
      double v = X[n] + f[k];
      if (e == 0 && s == 0) v = fma_rn(fc, u1[i], v);
      X[n] = v;
      f[k] = v;
    }
  }
  if constexpr (sizeof(RN) == 4) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = Blk<MH>::i_of(q, k);
      if (i < 0 || i >= M) f[k] = 0.0;
    }
    mean_shear<K>(f, N, s, MH - 1 - q * K, n1, q, D32, P);
  }
}

}  // namespace chdns
