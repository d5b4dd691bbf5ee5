// Dealiased nonlinear term H = u x omega for planes of 16 x 16 Fourier modes
// (the minimal channel of the paper's first domain; 3/2 rule, padded 24 x 24)
// in batches that supply enough planes to fill the SMs.
//
// Two planes per CTA of 160 threads, one 24-point line per thread in registers
// (fft_reg.cuh), the planes' lines pooled so that few lanes idle:
//   1. z inverse: 96 lines (6 fields x 8 kx columns per plane);
//   2. x inverse: 144 lines (6 fields x 12 pairs of z rows), two real rows of a
//      field packed into one complex line; the rows are read, and after a
//      barrier the transformed lines take their place;
//   3. the three products at the points of every row pair;
//   4. x forward: 72 lines (3 fields x 12 pairs), kept kx in place;
//   5. z forward: 48 lines (3 fields x 8 columns): the two rows of each pair are
//      unpacked as they are read, truncated to |kz| < 8 and scaled.
// One buffer of [6][12][24] points per plane holds every phase (28.8 KB per
// CTA in FP32, 57.6 KB in FP64).
//
// What bounds it: FP64 by the FP64 pipe (the pruned prime-factor lines take 232
// operations where 8 x 3 with twiddles took 320, and pooling fills 90 % of the
// lanes where teams of 96 threads filled 60 %); FP32 by issue and shared memory.
#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace chdns {

namespace {

constexpr int kNxh = 8, kNz = 16, kM = 24, kPairs = 12;
constexpr int kPPB = 2, kNT = 160;
// strides that keep both the line-wise and the point-wise accesses free of
// bank conflicts: z-transformed columns [6][12 pairs][2][8], row pairs [6][12][24]
constexpr int kZPair = 17, kZField = 216, kLine = 25;
constexpr int kX = 6 * kPairs * kLine;
static_assert(6 * kZField <= kX, "the columns fit the buffer");

}  // namespace

template <typename R>
__global__ void __launch_bounds__(kNT, sizeof(R) == 4 ? 6 : 3) plane16_kernel(PlaneArgs<R> a) {
  using C = typename cpx<R>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);  // [planes][kX], at first with the columns of step 1
  const int tid = threadIdx.x, b = blockIdx.y, j0 = blockIdx.x * kPPB;
  if (a.active && !a.active[b]) return;  // whole CTA (same b) returns together
  pdl_wait_then_release();               // the node values come from stage_pre
  const size_t P = a.P;

  // 1. z inverse
  if (tid < kPPB * 6 * kNxh) {
    const int i = tid % kNxh, f = tid / kNxh % 6, pl = tid / (6 * kNxh);
    if (j0 + pl < a.ny) {
      const C* q = a.q + (((size_t)b * 6 + f) * a.ny + j0 + pl) * P + i;
      C x[kM];
#pragma unroll
      for (int u = 0; u < kNz / 2; ++u) x[u] = q[u * kNxh];
      x[kNz] = czero<C>();  // the Nyquist row
#pragma unroll
      for (int u = kNz + 1; u < kM; ++u) x[u] = q[(u - (kM - kNz)) * kNxh];
      dft_reg<+1, true, kM, R>(x);
      C* Z = S + pl * kX + f * kZField + i;
#pragma unroll
      for (int z = 0; z < kM; ++z) Z[(z / 2) * kZPair + (z % 2) * kNxh] = x[z];
    }
  }
  __syncthreads();

  // 2. x inverse on pairs of rows
  {
    const bool on = tid < kPPB * 6 * kPairs;
    C* line = S + (on ? tid : 0) * kLine;
    C x[kM];
    if (on) {
      const int m = tid % kPairs, f = tid / kPairs % 6, pl = tid / (6 * kPairs);
      const C* A = S + pl * kX + f * kZField + m * kZPair;
      const C* B = A + kNxh;
#pragma unroll
      for (int k = 0; k < kNxh; ++k) {
        const C u = A[k], v = B[k];
        if (k == 0) {
          x[0] = mk(u.x, v.x);
          x[2 * kNxh] = czero<C>();
        } else {
          x[k] = mk(u.x - v.y, u.y + v.x);
          x[kM - k] = mk(u.x + v.y, v.x - u.y);
        }
      }
      dft_reg<+1, true, kM, R>(x);
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int k = 0; k < kM; ++k) line[k] = x[k];
    }
  }
  __syncthreads();

  // 3. products: real parts are the first row of a pair, imaginary parts the second
  constexpr int FS = kPairs * kLine;
  for (int w = tid; w < kPPB * kPairs * kM; w += kNT) {
    C* L = S + (w / (kPairs * kM)) * kX + (w / kM % kPairs) * kLine + w % kM;
    const C u = L[0], v = L[FS], ww = L[2 * FS];
    const C ox = L[3 * FS], oy = L[4 * FS], oz = L[5 * FS];
    L[0] = mk(v.x * oz.x - ww.x * oy.x, v.y * oz.y - ww.y * oy.y);
    L[FS] = mk(ww.x * ox.x - u.x * oz.x, ww.y * ox.y - u.y * oz.y);
    L[2 * FS] = mk(u.x * oy.x - v.x * ox.x, u.y * oy.y - v.y * ox.y);
  }
  __syncthreads();

  // 4. x forward, the kept kx in place
  if (tid < kPPB * 3 * kPairs) {
    C* line = S + (tid / (3 * kPairs)) * kX + (tid % (3 * kPairs)) * kLine;
    C x[kM];
#pragma unroll
    for (int k = 0; k < kM; ++k) x[k] = line[k];
    dft_reg<-1, false, kM, R>(x);
#pragma unroll
    for (int k = 0; k < kM; ++k)
      if (k < kNxh || k > kM - kNxh) line[k] = x[k];
  }
  __syncthreads();

  // 5. unpack, z forward, truncation and scaling (the 1/2 of the unpacking folded in)
  if (tid < kPPB * 3 * kNxh) {
    const int i = tid % kNxh, f = tid / kNxh % 3, pl = tid / (3 * kNxh);
    if (j0 + pl < a.ny) {
      const C* X = S + pl * kX + f * FS;
      const int im = i == 0 ? 0 : kM - i;
      C x[kM];
#pragma unroll
      for (int m = 0; m < kPairs; ++m) {
        const C zk = X[m * kLine + i], zm = X[m * kLine + im];
        x[2 * m] = mk(zk.x + zm.x, zk.y - zm.y);
        x[2 * m + 1] = mk(zk.y + zm.y, zm.x - zk.x);
      }
      dft_reg<-1, false, kM, R>(x);
      const R sc = (R)0.5 * a.scale;
      C* h = a.h + (((size_t)b * 3 + f) * a.ny + j0 + pl) * P + i;
#pragma unroll
      for (int row = 0; row < kNz; ++row)
        h[row * kNxh] = row == kNz / 2 ? czero<C>() : sc * x[row < kNz / 2 ? row : row + kM - kNz];
    }
  }
}

bool plane16_shape(int mx, int mz, int nxh, int nz) { return mx == kM && mz == kM && nxh == kNxh && nz == kNz; }

template <typename R>
cudaError_t launch_plane16(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  const size_t smem = (size_t)kPPB * kX * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(plane16_kernel<R>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl_if<sizeof(R) == 4>(plane16_kernel<R>, dim3((a.ny + kPPB - 1) / kPPB, B), dim3(kNT), smem, st, a);
}

template cudaError_t launch_plane16<double>(const PlaneArgs<double>&, int, cudaStream_t);
template cudaError_t launch_plane16<float>(const PlaneArgs<float>&, int, cudaStream_t);

}  // namespace chdns
