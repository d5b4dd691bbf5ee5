// The small kernels of the environment step (action, observation, wall shear,
// reward) and the stateless Chebyshev-tau entry points.  The Runge-Kutta stage
// itself lives in stage_kernels.cuh (wall-normal work) and plane.cu (nonlinear term).
//
// Chebyshev conventions: f(y) = sum_n a_n T_n(y), nodes y_j = cos(pi j / N).
// Derivative recurrence (coefficient space): c_m b_m = b_{m+2} + 2 (m+1) a_{m+1}
// with c_0 = 2, c_m = 1 otherwise, walked from m = N down to 0.
#include <algorithm>
#include <mutex>

#include "../../include/channel_dns.h"
#include "common.cuh"
#include "internal.h"

namespace chdns {

// ---------------------------------------------------------------------------
// Chebyshev-tau Dirichlet problem (D^2 - lam) f = r, split by parity.
//
// For n >= 2 the tau rows are equivalent to the quasi-tridiagonal rows
//   -lam c_{n-2}/(4n(n-1)) f_{n-2} + (1 + lam b_n/(2(n^2-1))) f_n
//   - lam b_{n+2}/(4n(n+1)) f_{n+2}
//     = c_{n-2}/(4n(n-1)) r_{n-2} - b_n/(2(n^2-1)) r_n + b_{n+2}/(4n(n+1)) r_{n+2}
// (b_m = 1 for m <= N-2, else 0: the two highest rows of r are dropped), obtained
// by integrating D^2 f = r + lam f twice.  With parity index i (n = 2i + sig) the
// rows i >= 1 are tridiagonal; the wall row sum_i f_i = s closes the system.
// Elimination from the bottom gives f_i = a_i + b_i f_{i-1}; all f_i are then
// affine in f_0, which the wall row fixes.  The lam-dependent factors
// e_i = 1/den_i, h_i = U_i/den_i, b_i = -L_i/den_i, Q_i = prod b and 1/sum Q
// are precomputed per mode and stage.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double tau_cA(int n) { return (n == 2 ? 2.0 : 1.0) / (4.0 * n * (n - 1)); }
__device__ __forceinline__ double tau_cB(int n, int N) { return n <= N - 2 ? 1.0 / (2.0 * ((double)n * n - 1.0)) : 0.0; }
__device__ __forceinline__ double tau_cC(int n, int N) { return n + 2 <= N - 2 ? 1.0 / (4.0 * n * (n + 1)) : 0.0; }

struct TabLocal {
  const double *pe, *ph, *pb, *pQ;
  __device__ double e(int i) const { return pe[i]; }
  __device__ double h(int i) const { return ph[i]; }
  __device__ double b(int i) const { return pb[i]; }
  __device__ double Q(int i) const { return pQ[i]; }
};

// r[i] = r_{2i+sig}; f[i] receives f_{2i+sig}.  r and f must not alias.
template <class Tab>
__device__ void tau_solve(int N, int sig, const double2* r, double2* f, const Tab& T, double isq, double2 s) {
  const int M = (N - sig) / 2 + 1;
  double2 anext = mk(0.0, 0.0);
  for (int i = M - 1; i >= 1; --i) {
    const int n = 2 * i + sig;
    double2 R = tau_cA(n) * r[i - 1] - tau_cB(n, N) * r[i];
    if (i + 1 < M) R = R + tau_cC(n, N) * r[i + 1];
    const double2 a = T.e(i) * R - T.h(i) * anext;
    f[i] = a;
    anext = a;
  }
  double2 Pp = mk(0.0, 0.0), sum = mk(0.0, 0.0);
  for (int i = 1; i < M; ++i) {
    Pp = f[i] + T.b(i) * Pp;
    f[i] = Pp;
    sum = sum + Pp;
  }
  const double2 f0 = isq * (s - sum);
  f[0] = f0;
  for (int i = 1; i < M; ++i) f[i] = f[i] + T.Q(i) * f0;
}

// on-the-fly factorisation of one parity (for the stateless entry point)
__device__ void tau_factor(int N, int sig, double lam, double* e, double* h, double* b, double* Q, double* isq) {
  const int M = (N - sig) / 2 + 1;
  double bnext = 0.0;
  e[0] = h[0] = b[0] = 0.0;
  for (int i = M - 1; i >= 1; --i) {
    const int n = 2 * i + sig;
    const double L = -lam * tau_cA(n);
    const double Dg = 1.0 + lam * tau_cB(n, N);
    const double U = (i + 1 < M) ? -lam * tau_cC(n, N) : 0.0;
    const double den = Dg + U * bnext;
    e[i] = 1.0 / den;
    h[i] = U / den;
    b[i] = -L / den;
    bnext = b[i];
  }
  Q[0] = 1.0;
  double sq = 1.0;
  for (int i = 1; i < M; ++i) {
    Q[i] = b[i] * Q[i - 1];
    sq += Q[i];
  }
  *isq = 1.0 / sq;
}

// ---------------------------------------------------------------------------
// wall shear of the lower wall: tau_w = nu sum_n U_n T_n'(-1), T_n'(-1) = (-1)^(n+1) n^2
// one warp per environment, fixed summation order
// ---------------------------------------------------------------------------
__global__ void wall_shear_kernel(int ny, int B, const double* UM, double nu, double* acc, const int* active) {
  const int b = blockIdx.x;
  if (b >= B || (active && !active[b])) return;
  const int lane = threadIdx.x;
  double s = 0.0;
  for (int n = lane; n < ny; n += 32) {
    const double d = (double)n * n * ((n & 1) ? 1.0 : -1.0);
    s += d * UM[(size_t)b * ny + n];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) acc[b] += nu * s;
}

// ---------------------------------------------------------------------------
// sensing plane: Fourier coefficients of u and v at node js (and, for
// opposition control, the wall spectrum -alpha v(y_s) with the mean removed,
// paper Sec. 4.1).  v(y_s) = sum_n v_n T_n(y_s), Dv(y_s) = sum_n v_n T_n'(y_s),
// omega_y(y_s) likewise.  L lanes per (mode, component q) share the sums;
// component q of Dv and omega_y makes component 1 - q of u = (i kx Dv - i kz
// omega_y) / k^2, so a lane group exchanges nothing with the other component.
// FP64-bound: three operations per coefficient and component.  One lane per
// system where the batch fills the SMs that way; four or eight (shorter chains
// of loads, a few operations more) for fewer systems or longer columns (us of a
// step's small kernels with 1 / 4 / 8 lanes: 16x65x16 x 16 70 / 54 / 52, x 128 81 /
// 72 / 81, x 256 92 / 94 / 106, 16x129x16 x 256 137 / 123 / 130, 64x33x64 x 16 91 /
// 101 / 119).
// ---------------------------------------------------------------------------
template <int L>
__global__ void __launch_bounds__(128) sense_kernel(Grid g, int B, PencilBufs pb, DevTables t, int js, double alpha,
                                                    int opposition) {
  const int P = g.P, ny = g.ny;
  const int lane = threadIdx.x & (L - 1);
  const long sys = (blockIdx.x * (long)blockDim.x + threadIdx.x) / L;  // (b, p, q), q fastest
  const bool inside = sys < 2L * P * B;
  const int q = (int)(sys & 1);
  const int p = inside ? (int)(sys / 2 % P) : 0;
  const int b = inside ? (int)(sys / 2 / P) : 0;
  const bool act = inside && !(pb.active && !pb.active[b]);
  const int row = p / g.nxh, ix = p % g.nxh;
  const double* cj = t.cheb + (size_t)js * ny;
  const bool gen = act && p > 0 && row != g.nz / 2, mean = act && p == 0 && q == 0;
  // partial sums (only the loads are conditional; every lane of the warp then
  // takes part in the same shuffles)
  double vs = 0.0, gs = 0.0, ds = 0.0;
  if (gen) {
    const size_t o = 2 * ((size_t)b * ny * P + p) + q;
    const double* V = reinterpret_cast<const double*>(pb.V) + o;
    const double* G = reinterpret_cast<const double*>(pb.G) + o;
#pragma unroll 8
    for (int n = lane; n < ny; n += L) {
      const double vn = V[(size_t)n * 2 * P], gn = G[(size_t)n * 2 * P], c = __ldg(cj + n);
      vs = fma(c, vn, vs);
      gs = fma(c, gn, gs);
      ds = fma(__ldg(t.dts + n), vn, ds);
    }
  } else if (mean) {
#pragma unroll 8
    for (int n = lane; n < ny; n += L) gs = fma(__ldg(cj + n), pb.UM[(size_t)b * ny + n], gs);
  }
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) {
    vs += __shfl_xor_sync(0xffffffffu, vs, o, L);
    gs += __shfl_xor_sync(0xffffffffu, gs, o, L);
    ds += __shfl_xor_sync(0xffffffffu, ds, o, L);
  }
  if (!act || lane != 0) return;
  const size_t o = (size_t)b * P + p;
  if (opposition) {
    // new action: the previous one becomes the start of the ramp, the wall
    // shear average restarts
    double* old = reinterpret_cast<double*>(pb.vw_old + o) + q;
    double* now = reinterpret_cast<double*>(pb.vw_new + o) + q;
    *old = *now;
    *now = p == 0 ? 0.0 : -alpha * vs;
    if (p == 0 && q == 0) pb.tau_acc[b] = 0.0;
  } else {
    double us = 0.0;
    int ru = 1 - q;  // component of u this thread makes
    if (gen) {
      const double kx = t.kx[ix], kz = t.kz[row];
      us = (q == 0 ? 1.0 : -1.0) * (kx * ds - kz * gs) / (kx * kx + kz * kz);
    } else if (p == 0) {
      us = gs;  // U in the real part, zero in the imaginary one
      ru = q;
    }
    reinterpret_cast<double*>(pb.planes + ((size_t)b * 2 + 0) * P + p)[ru] = us;
    reinterpret_cast<double*>(pb.planes + ((size_t)b * 2 + 1) * P + p)[q] = vs;
  }
}

// ---------------------------------------------------------------------------
// observation planes: unpadded inverse transform of the two sensing-plane
// spectra, f(x_a, z_b) = Re sum_kz F[kz,0] e^{i kz z} + 2 Re sum_{kx>0} F e^{i(kx x + kz z)}.
// One CTA per (block of zblk output rows, field, environment); each row has
// nt / zblk threads.  The z sums t[z_b][kx] are split over nq parts (rows
// q, q + nq, ...) and the x sums of every output over nr parts (kx = 1 + q,
// 1 + q + nr, ...); the parts are added in ascending order.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) obs_kernel(int nx, int nz, int nxh, int zblk, const double2* planes,
                                                  const double2* tw_nx, const double2* tw_nz, double* out,
                                                  size_t out_stride, const int* active) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int tpr = nt / zblk;                 // threads per output row
  const int nq = max(1, tpr / nxh), nr = max(1, tpr / nx);
  double2* part = reinterpret_cast<double2*>(smem_raw);  // [zblk][nq][nxh] z partial sums
  double2* tmp = part + (size_t)zblk * nq * nxh;         // [zblk][nxh]
  double* pr = reinterpret_cast<double*>(tmp + (size_t)zblk * nxh);  // [zblk][nr][nx] x partial sums
  const int z0 = blockIdx.x * zblk, f = blockIdx.y, b = blockIdx.z;
  if (active && !active[b]) return;
  const int P = nz * nxh;
  const double2* F = planes + ((size_t)b * 2 + f) * P;
  for (int w = tid; w < zblk * nq * nxh; w += nt) {
    const int zl = w / (nq * nxh), q = (w / nxh) % nq, i = w % nxh, zb = min(z0 + zl, nz - 1);
    double2 acc = mk(0.0, 0.0);
    int e = (q * zb) % nz;  // (row zb) mod nz; m = row - nz for row > nz/2 gives the same index
    const int step = (nq * zb) % nz;
#pragma unroll 4
    for (int row = q; row < nz; row += nq) {
      if (row != nz / 2) acc = acc + cmul(F[row * nxh + i], tw_nz[e]);
      e += step;
      if (e >= nz) e -= nz;
    }
    part[w] = acc;
  }
  __syncthreads();
  for (int w = tid; w < zblk * nxh; w += nt) {
    const int zl = w / nxh, i = w % nxh;
    const double2* pz = part + (size_t)zl * nq * nxh + i;
    double2 acc = pz[0];
    for (int q = 1; q < nq; ++q) acc = acc + pz[q * nxh];
    tmp[w] = acc;
  }
  __syncthreads();
  for (int w = tid; w < zblk * nr * nx; w += nt) {
    const int zl = w / (nr * nx), q = (w / nx) % nr, xa = w % nx;
    const double2* t = tmp + (size_t)zl * nxh;
    double s = 0.0;
    int e = ((1 + q) * xa) % nx;  // (kx xa) mod nx
    const int step = (nr * xa) % nx;
    for (int i = 1 + q; i < nxh; i += nr) {
      const double2 tw = tw_nx[e];
      const double2 v = t[i];
      s += v.x * tw.x - v.y * tw.y;
      e += step;
      if (e >= nx) e -= nx;
    }
    pr[w] = s;
  }
  __syncthreads();
  for (int w = tid; w < zblk * nx; w += nt) {
    const int zl = w / nx, xa = w % nx, zb = z0 + zl;
    if (zb >= nz) continue;
    const double* px = pr + (size_t)zl * nr * nx + xa;
    double s = 0.0;
    for (int q = 0; q < nr; ++q) s += px[q * nx];
    out[(size_t)b * out_stride + (size_t)f * nz * nx + (size_t)zb * nx + xa] = tmp[zl * nxh].x + 2.0 * s;
  }
}

// ---------------------------------------------------------------------------
// wall action -> wall spectrum: clip to [-u_tau, u_tau] (paper Sec. 3.2),
// forward transform of the kept modes; the mean mode (zero net mass flux,
// Sec. 4.1) and the Nyquist row are zero.  Removing the plane mean before the
// transform changes only the mean mode, which is set to zero, so it is not
// computed.  Two passes through a scratch plane tx[b][z][kx], one thread per
// output coefficient, each sum in ascending order:
//   action_x_kernel: x transform of the clipped rows; also starts the new
//                    action (the previous spectrum becomes the start of the
//                    ramp, the wall-shear average restarts);
//   action_z_kernel: z transform.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) action_x_kernel(int nx, int nz, int nxh, int B, const double* act,
                                                       double u_tau, const double2* tw_nx, double2* tx,
                                                       double2* vw_old, const double2* vw, double* acc,
                                                       const int* active) {
  const int P = nz * nxh;
  const long w = blockIdx.x * (long)blockDim.x + threadIdx.x;  // (b, z, kx), kx fastest
  if (w >= (long)B * P) return;
  const int b = (int)(w / P), o = (int)(w % P), zb = o / nxh, i = o % nxh;
  if (active && !active[b]) return;
  const size_t bo = (size_t)b * P + o;
  vw_old[bo] = vw[bo];
  if (o == 0) acc[b] = 0.0;
  const double* src = act + ((size_t)b * nz + zb) * nx;
  double2 s = mk(0.0, 0.0);
  int e = 0;  // (i xa) mod nx
#pragma unroll 8
  for (int xa = 0; xa < nx; ++xa) {
    s = s + fmin(fmax(src[xa], -u_tau), u_tau) * cconj(tw_nx[e]);
    e += i;
    if (e >= nx) e -= nx;
  }
  tx[bo] = s;
}

__global__ void __launch_bounds__(128) action_z_kernel(int nx, int nz, int nxh, int B, const double2* tx,
                                                       const double2* tw_nz, double2* vw, const int* active) {
  const int P = nz * nxh;
  const long w = blockIdx.x * (long)blockDim.x + threadIdx.x;  // (b, kz row, kx), kx fastest
  if (w >= (long)B * P) return;
  const int b = (int)(w / P), o = (int)(w % P), row = o / nxh, i = o % nxh;
  if (active && !active[b]) return;
  const double sc = 1.0 / ((double)nx * nz);
  double2 s = mk(0.0, 0.0);
  if (row != nz / 2 && !(row == 0 && i == 0)) {
    const int m = row < nz / 2 ? row : row - nz;
    const int step = m < 0 ? m + nz : m;  // (m zb) mod nz advances by m mod nz
    int e = 0;
#pragma unroll 8
    for (int zb = 0; zb < nz; ++zb) {
      s = s + cmul(tx[(size_t)b * P + (size_t)zb * nxh + i], cconj(tw_nz[e]));
      e += step;
      if (e >= nz) e -= nz;
    }
    s = sc * s;
  }
  vw[(size_t)b * P + o] = s;
}

__global__ void finalize_kernel(int B, const double* acc, double inv_steps, double tau_ref, double* out,
                                size_t out_stride, size_t out_offset, const int* active) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B || (active && !active[b])) return;
  const double tau = acc[b] * inv_steps;
  out[(size_t)b * out_stride + out_offset] = tau;
  out[(size_t)b * out_stride + out_offset + 1] = 1.0 - tau / tau_ref;
}

// ---------------------------------------------------------------------------
// stateless tau problems, one thread per (problem, parity, component): the
// elimination factors and the particular solution in one sweep down, the back
// substitution in one sweep up, a_i and b_i in columns of shared memory.  With
// W_{M-1} = 1, W_i = 1 + b_{i+1} W_{i+1} the sweep down also gives
// sum_i P_i = sum_i W_i a_i and sum_i Q_i = W_0, so f_0 = (s - sum P) / W_0.
// Lanes (component, parity) of a problem read whole 32-byte sectors of r.
//
// What bounds it: the FP64 pipe and, below 4864 problems, the chain of one
// warp per sub-partition (64 cycles per FP64 operation).  The row constants
// come from a table and each row divides once; the former one thread per
// (problem, parity) recomputed the constants with six more divisions per row
// and kept its vectors in local memory.
// ---------------------------------------------------------------------------
struct TauRows {
  double a[kMaxNy + 1] = {}, b[kMaxNy + 1] = {}, c[kMaxNy + 1] = {};  // cA_n, and cB_n, cC_n away from the cut
  constexpr TauRows() {
    for (int n = 2; n <= kMaxNy; ++n) {
      a[n] = (n == 2 ? 2.0 : 1.0) / (4.0 * n * (n - 1));
      b[n] = 1.0 / (2.0 * ((double)n * n - 1.0));
      c[n] = 1.0 / (4.0 * n * (n + 1));
    }
  }
};
static __device__ const TauRows g_tau_rows{};

constexpr int kTauNT = 32;

__global__ void __launch_bounds__(kTauNT) tau_helmholtz_kernel(int ny, int M, const double* __restrict__ lam,
                                                               const double2* r, const double2* __restrict__ top,
                                                               const double2* __restrict__ bot, double2* f) {
  extern __shared__ __align__(16) double tausm[];  // [2][rows][kTauNT]
  const int N = ny - 1, rows = N / 2 + 1;
  const long tid = blockIdx.x * (long)kTauNT + threadIdx.x;
  if (tid >= 4L * M) return;
  const int q = (int)(tid & 1), sig = (int)(tid >> 1 & 1);
  const long m = tid >> 2;
  const int Mp = (N - sig) / 2 + 1;
  const double l = lam[m];
  const double* rr = reinterpret_cast<const double*>(r + m * ny + sig) + q;  // element i at 4 i
  double* ca = tausm + threadIdx.x;
  double* cb = ca + rows * kTauNT;
  double r1 = rr[4 * (Mp - 1)], r2 = 0.0, an = 0.0, bn = 0.0, W = 1.0, sum = 0.0;
#pragma unroll 4
  for (int i = Mp - 1; i >= 1; --i) {
    const int n = 2 * i + sig;
    const double cA = __ldg(&g_tau_rows.a[n]);
    const double cB = n <= N - 2 ? __ldg(&g_tau_rows.b[n]) : 0.0;
    const double cC = n + 2 <= N - 2 ? __ldg(&g_tau_rows.c[n]) : 0.0;
    const double r0 = rr[4 * (i - 1)];
    if (i < Mp - 1) W = fma(bn, W, 1.0);
    const double U = -l * cC;  // zero in the last row
    const double e = 1.0 / fma(U, bn, fma(l, cB, 1.0));
    double R = fma(cA, r0, -(cB * r1));
    if (i + 1 < Mp) R = fma(cC, r2, R);
    const double a = e * fma(-U, an, R);
    const double b = e * (l * cA);
    ca[i * kTauNT] = a;
    cb[i * kTauNT] = b;
    sum = fma(W, a, sum);
    an = a;
    bn = b;
    r2 = r1;
    r1 = r0;
  }
  if (Mp > 1) W = fma(bn, W, 1.0);  // sum Q
  const double t = reinterpret_cast<const double*>(top + m)[q], u = reinterpret_cast<const double*>(bot + m)[q];
  double fp = (0.5 * (sig == 0 ? t + u : t - u) - sum) / W;
  double* out = reinterpret_cast<double*>(f + m * ny + sig) + q;
  out[0] = fp;
#pragma unroll 4
  for (int i = 1; i < Mp; ++i) {
    fp = fma(cb[i * kTauNT], fp, ca[i * kTauNT]);
    out[4 * i] = fp;
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// the FP32 copies of a state that came from the host; mode 0: the mean flow
// (W, U) and its derivatives, summed in FP64 and rounded once
__global__ void round_state_kernel(Grid g, int b, PencilBufs pb) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= (long)g.ny * g.P) return;
  const int n = (int)(i / g.P), p = (int)(i % g.P);
  const size_t o = (size_t)b * g.ny * g.P + i;
  double2 v = pb.V[o], w = pb.G[o];
  if (p == 0) {
    const double *U = pb.UM + (size_t)b * g.ny, *W = pb.WM + (size_t)b * g.ny;
    w = mk(W[n], U[n]);
    v = mk(0.0, 0.0);
    for (int m = g.N - ((g.N - n - 1) & 1); m > n; m -= 2) v = mk(fma(2.0 * m, W[m], v.x), fma(2.0 * m, U[m], v.y));
    if (n == 0) v = 0.5 * v;
  }
  pb.V32[o] = make_float2((float)v.x, (float)v.y);
  pb.G32[o] = make_float2((float)w.x, (float)w.y);
}
cudaError_t launch_round_state(const Grid& g, int b, const PencilBufs& pb, cudaStream_t st) {
  round_state_kernel<<<(unsigned)(((long)g.ny * g.P + 255) / 256), 256, 0, st>>>(g, b, pb);
  return cudaGetLastError();
}

cudaError_t launch_wall_shear(const Grid& g, int B, const double* UM, double nu, double* acc, const int* active,
                              cudaStream_t st) {
  wall_shear_kernel<<<B, 32, 0, st>>>(g.ny, B, UM, nu, acc, active);
  return cudaGetLastError();
}

cudaError_t launch_sense(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, int js, double alpha,
                         int opposition, cudaStream_t st) {
  const long sys = 2L * g.P * B;
  if (sys >= 65536 && g.ny <= 97)
    sense_kernel<1><<<(unsigned)((sys + 127) / 128), 128, 0, st>>>(g, B, pb, t, js, alpha, opposition);
  else if (sys >= 16384)
    sense_kernel<4><<<(unsigned)((4 * sys + 127) / 128), 128, 0, st>>>(g, B, pb, t, js, alpha, opposition);
  else
    sense_kernel<8><<<(unsigned)((8 * sys + 127) / 128), 128, 0, st>>>(g, B, pb, t, js, alpha, opposition);
  return cudaGetLastError();
}

cudaError_t launch_obs(const Grid& g, int B, double2* planes, const DevTables& t, double* out, size_t out_stride,
                       const int* active, cudaStream_t st) {
  if (io_by_lines(g, B)) return launch_obs_lines(g, B, planes, t, out, out_stride, active, st);
  // several output rows per CTA once the batch alone gives 128 or more
  // (environment, field) CTAs; otherwise one row per CTA, its sums split over
  // the CTA's threads
  const int zblk = B >= 64 ? std::max(1, std::min(g.nz, 128 / g.nxh)) : 1;
  const int tpr = 128 / zblk;
  const int nq = std::max(1, tpr / g.nxh), nr = std::max(1, tpr / g.nx);
  const size_t smem = (size_t)zblk * ((nq + 1) * g.nxh * sizeof(double2) + (size_t)nr * g.nx * sizeof(double));
  obs_kernel<<<dim3((g.nz + zblk - 1) / zblk, 2, B), 128, smem, st>>>(g.nx, g.nz, g.nxh, zblk, planes, t.tw_nx,
                                                                       t.tw_nz, out, out_stride, active);
  return cudaGetLastError();
}

cudaError_t launch_action(const Grid& g, int B, const double* act, double u_tau, const DevTables& t,
                          const PencilBufs& pb, cudaStream_t st) {
  if (io_by_lines(g, B)) return launch_action_lines(g, B, act, u_tau, t, pb, st);
  // the sensing-plane buffer is free at this point of the step: it is the scratch plane
  double2* tx = pb.planes;
  const long n = (long)B * g.nz * g.nxh;
  const unsigned blocks = (unsigned)((n + 127) / 128);
  action_x_kernel<<<blocks, 128, 0, st>>>(g.nx, g.nz, g.nxh, B, act, u_tau, t.tw_nx, tx, pb.vw_old, pb.vw_new,
                                          pb.tau_acc, pb.active);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  action_z_kernel<<<blocks, 128, 0, st>>>(g.nx, g.nz, g.nxh, B, tx, t.tw_nz, pb.vw_new, pb.active);
  return cudaGetLastError();
}

cudaError_t launch_finalize(int B, const double* acc, double inv_steps, double tau_ref, double* out,
                            size_t out_stride, size_t out_offset, const int* active, cudaStream_t st) {
  finalize_kernel<<<(B + 127) / 128, 128, 0, st>>>(B, acc, inv_steps, tau_ref, out, out_stride, out_offset, active);
  return cudaGetLastError();
}

cudaError_t launch_tau_helmholtz(int ny, int M, const double* lam, const double2* r, const double2* top,
                                 const double2* bot, double2* f, cudaStream_t st) {
  const size_t smem = (size_t)2 * ((ny - 1) / 2 + 1) * kTauNT * sizeof(double);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(tau_helmholtz_kernel, &lim, smem);
  if (e != cudaSuccess) return e;
  tau_helmholtz_kernel<<<(unsigned)((4L * M + kTauNT - 1) / kTauNT), kTauNT, smem, st>>>(ny, M, lam, r, top, bot, f);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Allocation-free variant of the stateless tau entry point.
//
// Kernels that spill work vectors (6.5 KB per problem and parity at 201 nodes)
// to local memory rely on an allocation of the CUDA driver, which may have to
// grow at launch time.  Some callers cannot let
// anything allocate device memory: a control loop with a fixed real-time
// budget (cudaMalloc and a driver-side resize can block for milliseconds and
// synchronise the device), a process whose device memory is already fully
// handed to another allocator's pool, or a host framework that only lends out
// buffers it owns.  For them the work vectors live in one file-scope array
// below, sized once when the library is loaded.
// ---------------------------------------------------------------------------
}  // namespace chdns

// 16 MiB of doubles, held by every GPU that loads the library until the
// process exits.  Shared by all calls; a call writes every slot it reads, so
// nothing has to start at zero.
constexpr size_t kNoAllocScratchDoubles = (size_t)2 << 20;
static __device__ __align__(256) double g_tau_noalloc_scratch[kNoAllocScratchDoubles];

namespace chdns {

__global__ void tau_helmholtz_noalloc_kernel(int ny, int M, int mpad, const double* lam, const double2* r,
                                             const double2* top, const double2* bot, double2* f,
                                             double* scratch) {
  const long tid = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (tid >= 2L * M) return;
  const int m = (int)(tid / 2), sig = (int)(tid % 2);
  const int N = ny - 1;
  // slot layout: e, h, b, Q (mpad doubles each), then r and f (mpad complex each)
  double* base = scratch + (size_t)tid * 8 * mpad;
  double* e = base;
  double* h = base + mpad;
  double* bb = base + 2 * mpad;
  double* Q = base + 3 * mpad;
  double2* rr = reinterpret_cast<double2*>(base + 4 * mpad);
  double2* ff = reinterpret_cast<double2*>(base + 6 * mpad);
  double isq;
  tau_factor(N, sig, lam[m], e, h, bb, Q, &isq);
  const int Mp = (N - sig) / 2 + 1;
  for (int i = 0; i < Mp; ++i) rr[i] = r[(size_t)m * ny + 2 * i + sig];
  const double2 s = sig == 0 ? 0.5 * (top[m] + bot[m]) : 0.5 * (top[m] - bot[m]);
  tau_solve(N, sig, rr, ff, TabLocal{e, h, bb, Q}, isq, s);
  for (int i = 0; i < Mp; ++i) f[(size_t)m * ny + 2 * i + sig] = ff[i];
}

}  // namespace chdns

namespace {

// Device address of the scratch array, looked up once per device.
using chdns::kMaxDevices;
double* g_noalloc_ptr[kMaxDevices] = {nullptr};
std::mutex g_noalloc_mu;

int noalloc_scratch(double** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return CH_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_tau_noalloc_scratch) != cudaSuccess || !p) return CH_ERR_CUDA;
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return CH_OK;
}

}  // namespace

extern "C" int ch_tau_helmholtz_noalloc(int ny, int M, const double* d_lam, const double* d_r,
                                        const double* d_top, const double* d_bot, double* d_f, void* stream) {
  if (ny < 5 || ny > chdns::kMaxNy || M < 0) return CH_ERR_ARG;
  if (M == 0) return CH_OK;
  if (!d_lam || !d_r || !d_top || !d_bot || !d_f) return CH_ERR_ARG;
  const int mpad = ((ny / 2 + 1) + 1) & ~1;  // even, keeps the complex work vectors 16-byte aligned
  if ((size_t)2 * M * 8 * mpad > kNoAllocScratchDoubles) return CH_ERR_ARG;
  double* scratch = nullptr;
  const int rc = noalloc_scratch(&scratch);
  if (rc != CH_OK) return rc;
  const long n = 2L * M;
  chdns::tau_helmholtz_noalloc_kernel<<<(unsigned)((n + 63) / 64), 64, 0, static_cast<cudaStream_t>(stream)>>>(
      ny, M, mpad, d_lam, reinterpret_cast<const double2*>(d_r), reinterpret_cast<const double2*>(d_top),
      reinterpret_cast<const double2*>(d_bot), reinterpret_cast<double2*>(d_f), scratch);
  return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ERR_CUDA;
}
