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
#include <cooperative_groups.h>

#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

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

  // 1. z inverse
  if (tid < kPPB * 6 * kNxh) {
    const int i = tid % kNxh, f = tid / kNxh % 6, pl = tid / (6 * kNxh);
    if (j0 + pl < a.ny) {
      const C* q = a.q + b * a.qb + f * a.qf + (j0 + pl) * a.qj + i;
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
      C* h = a.h + b * a.hb + f * a.qf + (j0 + pl) * a.qj + i;
#pragma unroll
      for (int row = 0; row < kNz; ++row)
        h[row * kNxh] = row == kNz / 2 ? czero<C>() : sc * x[row < kNz / 2 ? row : row + kM - kNz];
    }
  }
}

// ---------------------------------------------------------------------------
// The same planes in batches that do not fill the SMs (a single minimal channel
// has 65): one plane per cluster of two CTAs, the 24-point lines in two register
// steps of 6 and 4 points so that every phase has 48 to 216 tasks per CTA.
// CTA `rank` transforms the columns of three fields along z, owns six row pairs
// for the x transforms and products, and four kx columns of H; rows and columns
// change hands through distributed shared memory.
//
// What bounds it: the chain of phases.  An FP64 operation holds a warp's
// sub-partition for 64 cycles, so a phase costs the operations of its task
// (28 to 40) times the warps per sub-partition (one or two); four CTAs per plane
// with whole-row tasks took 27 us per launch for 65 planes.
// ---------------------------------------------------------------------------
namespace {
constexpr int kPairNT = 256;
constexpr int kT6 = 28, kA1 = 7;                      // exchange of a 24-point line: [4][7]
constexpr int kPZField = 6 * kZPair, kHCol = 25;      // rows of six pairs per field; a column of H
constexpr int kPairSmem = 24 * kT6 + 6 * kPZField + 36 * kT6 + 12 * kHCol;
}  // namespace

template <typename R>
__global__ void __launch_bounds__(kPairNT) plane16_pair_kernel(PlaneArgs<R> a) {
  using C = typename cpx<R>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* T = reinterpret_cast<C*>(smem_raw);  // [24 columns][4][7]
  C* Z = T + 24 * kT6;                    // [6][6 pairs][2][8]
  C* X = Z + 6 * kPZField;                // [6][6 pairs][4][7]
  C* H = X + 36 * kT6;                    // [3][4 kx][24 z]
  auto cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x, j = blockIdx.y, b = blockIdx.z;
  if (a.active && !a.active[b]) return;  // whole cluster (same b) returns together
  const C* __restrict__ tw = a.tw_x;     // e^{2 pi i k / 24}
  C* Zr = cluster.map_shared_rank(Z, rank ^ 1);
  C* Hr = cluster.map_shared_rank(H, rank ^ 1);

  // z inverse of this CTA's three fields
  if (tid < 96) {
    const int c = tid % 24, kb = tid / 24;
    const C* q = a.q + b * a.qb + (3 * rank + c / 8) * a.qf + j * a.qj + c % 8;
    C x[6];
#pragma unroll
    for (int p = 0; p < 2; ++p) x[p] = q[(4 * p + kb) * kNxh];
#pragma unroll
    for (int p = 4; p < 6; ++p) x[p] = p == 4 && kb == 0 ? czero<C>() : q[(4 * p + kb - 8) * kNxh];
    dft_reg<+1, true, 6, R>(x);
#pragma unroll
    for (int p = 0; p < 6; ++p) T[c * kT6 + kb * kA1 + p] = x[p];
  }
  cluster.sync();  // also: both CTAs are running before either writes to the other
  if (tid < 144) {
    const int c = tid % 24, ka = tid / 24;
    const C w[2] = {tw[ka], tw[2 * ka]};
    C x[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) x[s] = T[c * kT6 + s * kA1 + ka];
    dft_tw<4, R>(x, w);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int z = ka + 6 * s, m = z / 2;
      C* dst = m / 6 == rank ? Z : Zr;
      dst[(3 * rank + c / 8) * kPZField + (m % 6) * kZPair + (z % 2) * kNxh + c % 8] = x[s];
    }
  }
  cluster.sync();

  // x inverse, products, x forward of this CTA's six row pairs
  if (tid < 144) {
    const int kb = tid % 4, line = tid / 4;
    const C* r1 = Z + (line / 6) * kPZField + (line % 6) * kZPair;
    const C* r2 = r1 + kNxh;
    C x[6];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const C u = r1[4 * p + kb], v = r2[4 * p + kb];
      x[p] = p == 0 && kb == 0 ? mk(u.x, v.x) : mk(u.x - v.y, u.y + v.x);
    }
#pragma unroll
    for (int p = 4; p < 6; ++p) {
      if (p == 4 && kb == 0) {
        x[p] = czero<C>();
      } else {
        const C u = r1[kM - (4 * p + kb)], v = r2[kM - (4 * p + kb)];
        x[p] = mk(u.x + v.y, v.x - u.y);
      }
    }
    dft_reg<+1, true, 6, R>(x);
#pragma unroll
    for (int p = 0; p < 6; ++p) X[line * kT6 + kb * kA1 + p] = x[p];
  }
  __syncthreads();
  if (tid < 216) {
    const int ka = tid % 6;
    C* L = X + (tid / 6) * kT6 + ka;
    const C w[2] = {tw[ka], tw[2 * ka]};
    C x[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) x[s] = L[s * kA1];
    dft_tw<4, R>(x, w);
#pragma unroll
    for (int s = 0; s < 4; ++s) L[s * kA1] = x[s];
  }
  __syncthreads();
  if (tid < 144) {
    constexpr int FS = 6 * kT6;
    C* L = X + (tid / 24) * kT6 + (tid / 6 % 4) * kA1 + tid % 6;
    const C u = L[0], v = L[FS], ww = L[2 * FS], ox = L[3 * FS], oy = L[4 * FS], oz = L[5 * FS];
    L[0] = mk(v.x * oz.x - ww.x * oy.x, v.y * oz.y - ww.y * oy.y);
    L[FS] = mk(ww.x * ox.x - u.x * oz.x, ww.y * ox.y - u.y * oz.y);
    L[2 * FS] = mk(u.x * oy.x - v.x * ox.x, u.y * oy.y - v.y * ox.y);
  }
  __syncthreads();
  if (tid < 108) {
    const int ka = tid % 6;
    C* L = X + (tid / 6) * kT6 + ka;
    C x[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) x[s] = L[s * kA1];
    small_dft_ct<-1, 4, C, R>(x);
    L[0] = x[0];
#pragma unroll
    for (int s = 1; s < 4; ++s) L[s * kA1] = cmul(x[s], cconj(tw[s * ka]));
  }
  __syncthreads();
  if (tid < 72) {
    C* L = X + (tid / 4) * kT6 + (tid % 4) * kA1;
    C x[6];
#pragma unroll
    for (int p = 0; p < 6; ++p) x[p] = L[p];
    dft_reg<-1, false, 6, R>(x);
#pragma unroll
    for (int p = 0; p < 6; ++p)
      if (p < 2 || p >= 4) L[p] = x[p];  // k = 4 p + s
  }
  __syncthreads();
  if (tid < 144) {
    const int i = tid % 8, line = tid / 8, f = line / 6, z = 2 * (line % 6 + 6 * rank);
    const int im = i == 0 ? 0 : kM - i;
    const C zk = X[line * kT6 + (i % 4) * kA1 + i / 4], zm = X[line * kT6 + (im % 4) * kA1 + im / 4];
    C* dst = (i / 4 == rank ? H : Hr) + (f * 4 + i % 4) * kHCol + z;
    dst[0] = mk(zk.x + zm.x, zk.y - zm.y);
    dst[1] = mk(zk.y + zm.y, zm.x - zk.x);
  }
  cluster.sync();

  // z forward of this CTA's four kx columns (the 1/2 of the unpacking in the scale)
  if (tid < 72) {
    const int c = tid % 12, ka = tid / 12;
    C x[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) x[s] = H[c * kHCol + ka + 6 * s];
    small_dft_ct<-1, 4, C, R>(x);
    T[c * kT6 + ka] = x[0];
#pragma unroll
    for (int s = 1; s < 4; ++s) T[c * kT6 + s * kA1 + ka] = cmul(x[s], cconj(tw[s * ka]));
  }
  __syncthreads();
  if (tid < 48) {
    const int c = tid % 12, s = tid / 12;
    C x[6];
#pragma unroll
    for (int p = 0; p < 6; ++p) x[p] = T[c * kT6 + s * kA1 + p];
    dft_reg<-1, false, 6, R>(x);
    const R sc = (R)0.5 * a.scale;
    C* h = a.h + b * a.hb + c / 4 * a.qf + j * a.qj + rank * 4 + c % 4;
#pragma unroll
    for (int p = 0; p < 2; ++p) h[(4 * p + s) * kNxh] = sc * x[p];
#pragma unroll
    for (int p = 4; p < 6; ++p) h[(4 * p + s - 8) * kNxh] = p == 4 && s == 0 ? czero<C>() : sc * x[p];
  }
}

template <typename R>
static cudaError_t launch_plane16_pair(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  const size_t smem = (size_t)kPairSmem * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(plane16_pair_kernel<R>, &lim, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2, a.ny, B);
  cfg.blockDim = dim3(kPairNT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, plane16_pair_kernel<R>, a);
}

bool plane16_shape(int mx, int mz, int nxh, int nz) { return mx == kM && mz == kM && nxh == kNxh && nz == kNz; }

template <typename R>
cudaError_t launch_plane16(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  if (a.team16 == 2) return launch_plane16_pair<R>(a, B, st);
  const size_t smem = (size_t)kPPB * kX * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(plane16_kernel<R>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(plane16_kernel<R>, dim3((a.ny + kPPB - 1) / kPPB, B), dim3(kNT), smem, st, a);
}

template cudaError_t launch_plane16<double>(const PlaneArgs<double>&, int, cudaStream_t);
template cudaError_t launch_plane16<float>(const PlaneArgs<float>&, int, cudaStream_t);

}  // namespace chdns
