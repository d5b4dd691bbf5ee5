// Unpadded transforms between the wall-parallel planes the caller sees
// (actions, observations) and their spectra, FP64, for batches and large grids:
// every line in two register DFTs around one exchange in shared memory
// (fft_reg.cuh), n = A B.
//
// What bounds them: the FP64 pipe.  The direct sums of pencil.cu take
// O(nx nz (nx + nz)) operations per plane, 3.1 M warp operations for the two
// observation planes of 256 x 256 points against 0.2 M here; they remain for
// small planes, whose few sums spread over more threads.
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace chdns {

__host__ __device__ constexpr int io_b(int n) { return n == 8 ? 2 : n <= 96 ? 4 : n <= 192 ? 8 : 16; }
__host__ __device__ constexpr int io_a(int n) { return n / io_b(n); }
// line lengths built
#define CH_IO_LENGTHS(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256)

// columns per single-warp CTA of a z pass and row pairs per CTA of an x pass:
// eight where the batch has CTAs to spare, two for single large planes, whose
// few lines spread over more SMs (the chain of a warp is what their passes take)
constexpr int kIoNT = 64;

// z inverse of the sensing spectra in place: planes [B][2][nz][nxh]
template <int NZ, int CT>
__global__ void __launch_bounds__(32) obs_z_kernel(int nxh, double2* planes, const double2* __restrict__ tw, const int* active) {
  constexpr int A = io_a(NZ), B = io_b(NZ);
  __shared__ double2 T[NZ * CT];
  const int b = blockIdx.y, c0 = blockIdx.x * CT;
  if (active && !active[b]) return;
  double2* F = planes + (size_t)b * 2 * NZ * nxh;
  for (int w = threadIdx.x; w < B * CT; w += 32) {
    const int c = w % CT, kb = w / CT, g = c0 + c;
    if (g >= 2 * nxh) continue;
    const double2* src = F + (size_t)(g / nxh) * NZ * nxh + g % nxh;
    double2 x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) x[p] = B * p + kb == NZ / 2 ? mk(0.0, 0.0) : src[(size_t)(B * p + kb) * nxh];
    dft_reg<+1, false, A, double>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) T[(kb * A + p) * CT + c] = x[p];
  }
  __syncthreads();
  for (int w = threadIdx.x; w < A * CT; w += 32) {
    const int c = w % CT, ka = w / CT, g = c0 + c;
    if (g >= 2 * nxh) continue;
    double2 x[B];
    x[0] = T[ka * CT + c];
#pragma unroll
    for (int s = 1; s < B; ++s) x[s] = cmul(T[(s * A + ka) * CT + c], tw[s * ka]);
    dft_pow2<+1, B, double>(x);
    double2* dst = F + (size_t)(g / nxh) * NZ * nxh + g % nxh;
#pragma unroll
    for (int s = 0; s < B; ++s) dst[(size_t)(ka + A * s) * nxh] = x[s];
  }
}

// x inverse of row pairs of both fields to the observation planes
template <int NX, int NPR>
__global__ void __launch_bounds__(kIoNT) obs_x_kernel(int nz, const double2* __restrict__ planes,
                                                      const double2* __restrict__ tw, double* out, size_t out_stride,
                                                      const int* active) {
  constexpr int A = io_a(NX), B = io_b(NX), A1 = A | 1, LS = B * A1, NXH = NX / 2;
  extern __shared__ __align__(16) double2 iosm[];  // [NPR][B][A1]
  const int b = blockIdx.y, g0 = blockIdx.x * NPR;  // row pair (field, m): rows 2 m, 2 m + 1
  if (active && !active[b]) return;
  const double2* F = planes + (size_t)b * 2 * nz * NXH;
  for (int w = threadIdx.x; w < NPR * B; w += kIoNT) {
    const int kb = w % B, g = g0 + w / B;
    if (g >= nz) continue;
    const double2* r1 = F + (size_t)2 * g * NXH;  // the rows of both fields follow one another
    const double2* r2 = r1 + NXH;
    double2 x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) {
      const int k = B * p + kb;
      if (k == 0) {
        x[p] = mk(r1[0].x, r2[0].x);
      } else if (k < NXH) {
        const double2 u = r1[k], v = r2[k];
        x[p] = mk(u.x - v.y, u.y + v.x);
      } else if (k > NXH) {
        const double2 u = r1[NX - k], v = r2[NX - k];
        x[p] = mk(u.x + v.y, v.x - u.y);
      } else {
        x[p] = mk(0.0, 0.0);
      }
    }
    dft_reg<+1, false, A, double>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) iosm[(w / B) * LS + kb * A1 + p] = x[p];
  }
  __syncthreads();
  for (int w = threadIdx.x; w < NPR * A; w += kIoNT) {
    const int ka = w % A, g = g0 + w / A;
    if (g >= nz) continue;
    const double2* X = iosm + (w / A) * LS + ka;
    double2 x[B];
    x[0] = X[0];
#pragma unroll
    for (int s = 1; s < B; ++s) x[s] = cmul(X[s * A1], tw[s * ka]);
    dft_pow2<+1, B, double>(x);
    double* dst = out + (size_t)b * out_stride + (size_t)2 * g * NX;
#pragma unroll
    for (int s = 0; s < B; ++s) {
      dst[ka + A * s] = x[s].x;
      dst[NX + ka + A * s] = x[s].y;
    }
  }
}

// x forward of the clipped action, row pairs; starts the new action as
// action_x_kernel (pencil.cu)
template <int NX, int NPR>
__global__ void __launch_bounds__(kIoNT) act_x_kernel(int nz, const double* __restrict__ act, double u_tau,
                                                      const double2* __restrict__ tw, double2* tx, double2* vw_old,
                                                      const double2* vw, double* acc, const int* active) {
  constexpr int A = io_a(NX), B = io_b(NX), A1 = A | 1, LS = B * A1, NXH = NX / 2;
  extern __shared__ __align__(16) double2 iosm[];
  const int b = blockIdx.y, g0 = blockIdx.x * NPR, pairs = nz / 2;
  if (active && !active[b]) return;
  const double* src = act + (size_t)b * nz * NX;
  auto clip = [u_tau](double v) { return fmin(fmax(v, -u_tau), u_tau); };
  for (int w = threadIdx.x; w < NPR * A; w += kIoNT) {
    const int ka = w % A, g = g0 + w / A;
    if (g >= pairs) continue;
    const double* r1 = src + (size_t)2 * g * NX;
    double2 x[B];
#pragma unroll
    for (int s = 0; s < B; ++s) x[s] = mk(clip(r1[ka + A * s]), clip(r1[NX + ka + A * s]));
    dft_pow2<-1, B, double>(x);
    double2* X = iosm + (w / A) * LS + ka;
    X[0] = x[0];
#pragma unroll
    for (int s = 1; s < B; ++s) X[s * A1] = cmul(x[s], cconj(tw[s * ka]));
  }
  __syncthreads();
  for (int w = threadIdx.x; w < NPR * B; w += kIoNT) {
    double2* X = iosm + (w / B) * LS + (w % B) * A1;
    if (g0 + w / B >= pairs) continue;
    double2 x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) x[p] = X[p];
    dft_reg<-1, false, A, double>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) X[p] = x[p];  // k = B p + s
  }
  __syncthreads();
  for (int w = threadIdx.x; w < NPR * NXH; w += kIoNT) {
    const int i = w % NXH, g = g0 + w / NXH;
    if (g >= pairs) continue;
    const int im = i == 0 ? 0 : NX - i;
    const double2 zk = iosm[(w / NXH) * LS + (i % B) * A1 + i / B], zm = iosm[(w / NXH) * LS + (im % B) * A1 + im / B];
    const size_t o = ((size_t)b * nz + 2 * g) * NXH + i;
    tx[o] = mk(0.5 * (zk.x + zm.x), 0.5 * (zk.y - zm.y));
    tx[o + NXH] = mk(0.5 * (zk.y + zm.y), 0.5 * (zm.x - zk.x));
    vw_old[o] = vw[o];
    vw_old[o + NXH] = vw[o + NXH];
    if (g == 0 && i == 0) acc[b] = 0.0;
  }
}

// z forward of the action to the wall spectrum
template <int NZ, int CT>
__global__ void __launch_bounds__(32) act_z_kernel(int nx, const double2* __restrict__ tx, const double2* __restrict__ tw,
                                                   double2* vw, const int* active) {
  constexpr int A = io_a(NZ), B = io_b(NZ);
  __shared__ double2 T[NZ * CT];
  const int b = blockIdx.y, c0 = blockIdx.x * CT, nxh = nx / 2;
  if (active && !active[b]) return;
  const size_t o = (size_t)b * NZ * nxh;
  for (int w = threadIdx.x; w < A * CT; w += 32) {
    const int c = w % CT, ka = w / CT, i = c0 + c;
    if (i >= nxh) continue;
    double2 x[B];
#pragma unroll
    for (int s = 0; s < B; ++s) x[s] = tx[o + (size_t)(ka + A * s) * nxh + i];
    dft_pow2<-1, B, double>(x);
    T[ka * CT + c] = x[0];
#pragma unroll
    for (int s = 1; s < B; ++s) T[(s * A + ka) * CT + c] = cmul(x[s], cconj(tw[s * ka]));
  }
  __syncthreads();
  const double sc = 1.0 / ((double)nx * NZ);
  for (int w = threadIdx.x; w < B * CT; w += 32) {
    const int c = w % CT, s = w / CT, i = c0 + c;
    if (i >= nxh) continue;
    double2 x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) x[p] = T[(s * A + p) * CT + c];
    dft_reg<-1, false, A, double>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) {
      const int row = B * p + s;
      const bool zero = row == NZ / 2 || (row == 0 && i == 0);  // zero net mass flux, no Nyquist content
      vw[o + (size_t)row * nxh + i] = zero ? mk(0.0, 0.0) : sc * x[p];
    }
  }
}

}  // namespace chdns
