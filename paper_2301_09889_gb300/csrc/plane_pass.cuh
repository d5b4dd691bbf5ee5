// Dealiased nonlinear term H = u x omega (3/2 rule; paper Sec. 3.1
// pseudo-spectral method) in three passes through global memory, over node
// values y[B][ny][6][mz][nxh] that stay in L2 for all but the largest planes (in
// a step the handle's node array, in place; ch_nonlinear uses it as scratch):
//   1. z inverse: the kept kz rows of a (node, field, kx) column -> mz rows;
//   2. x pass: two physical z rows of a field packed into one complex line,
//      inverse transform, the three products, forward transform, unpacked over
//      fields 0..2 of the same rows;
//   3. z forward: mz rows of H -> the rows |kz| < nz/2, scaled by 1/(mx mz).
// Every line goes through two register DFTs and one exchange in shared memory
// (fft_reg.cuh): no index arithmetic or barrier inside a transform, and the
// padding third of every line costs no operation.
//
// What bounds it: FP64 planes by the FP64 pipe.  On GB300 a warp-wide FP64
// operation holds its sub-partition's pipe for 64 cycles (76 with all four
// sub-partitions busy: 1.06 TFLOP/s per GPU), whatever its active lanes, so
// the passes are shaped for the fewest operations with every lane at work:
// tiles whose task counts are multiples of a warp, small CTAs that even out
// over the SMs.  FP32 planes by L2 and instruction issue.  The twiddles of a
// line of A x B points stand as [B][A], in the order in which the lanes of a
// warp take them (as gathers from one table of roots they took more L1 cycles
// than the exchange: 278 us, 238 in lane order, for the x pass of
// 256x193x256 in FP32, split 24 x 16; 206 split 48 x 8 with the products in
// registers; 128x129x128 48 and 38).
#pragma once

#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace chdns {

// z passes: tiles of 16 (FP32) or 8 (FP64) adjacent columns, one task of the
// first step per thread
template <typename R> constexpr int z_cols() { return sizeof(R) == 4 ? 16 : 8; }
template <typename R> constexpr int z_threads(int m) { return line_b(m) * z_cols<R>() < 32 ? 32 : line_b(m) * z_cols<R>(); }

// x pass: row pairs per CTA (the task counts of its steps are multiples of the
// threads, or nearly), threads and CTAs per SM (bounds the registers)
constexpr int x_pairs(int m) { return m <= 96 ? 8 : m <= 192 ? 4 : 2; }
template <typename R> constexpr int x_threads(int m) { return m <= 24 || (sizeof(R) == 4 && m >= 144) ? 96 : 192; }
template <typename R> constexpr int x_ctas(int m) { return sizeof(R) == 4 && m >= 144 ? 5 : 1; }
// elements between the sub-lines of a line, odd, and between lines: the
// exchanges meet (nearly) no bank twice.  FP32 lines of 48 x 8 and 36 x 8: 50,
// with an odd line, for the unpacking of eight adjacent modes of two sub-lines.
// Lines of sixteen: the second step's lanes run on into the next line, which
// continues the banks of the first.
template <typename R> __host__ __device__ constexpr int x_stride(int m) {
  return sizeof(R) == 4 && m > 192 ? 50 : x_line_a<R>(m) | 1;
}
template <typename R> __host__ __device__ constexpr int x_line(int m) {
  const int b = x_line_b<R>(m), l = b * x_stride<R>(m);
  if (sizeof(R) == 4 && m > 192) return l + 1;
  return b == 16 ? l + ((x_line_a<R>(m) - l) % 8 + 8) % 8 : l;
}

template <typename R, int MZ>
__global__ void __launch_bounds__(z_threads<R>(MZ)) zpass_inverse_kernel(PlaneArgs<R> a) {
  using C = typename cpx<R>::T;
  constexpr int A = line_a(MZ), B = line_b(MZ), CT = z_cols<R>(), NT = z_threads<R>(MZ);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* T = reinterpret_cast<C*>(smem_raw);  // [B][A][CT]
  const int b = blockIdx.y, nxh = a.nxh;
  if (a.active && !a.active[b]) return;
  const int cols = a.ny * 6 * nxh, c0 = blockIdx.x * CT;  // column (j, f, i), i fastest
  for (int w = threadIdx.x; w < B * CT; w += NT) {
    const int c = w % CT, kb = w / CT, g = c0 + c;
    if (g >= cols) continue;
    const int i = g % nxh, jf = g / nxh, f = jf % 6, j = jf / 6;
    const C* src = a.q + b * a.qb + f * a.qf + j * a.qj + i;
    C x[A];
#pragma unroll
    for (int p = 0; p < A / 3; ++p) x[p] = src[(size_t)(B * p + kb) * nxh];
#pragma unroll
    for (int p = 2 * A / 3; p < A; ++p) {
      const int row = B * p + kb - MZ / 3;  // kz = B p + kb - MZ; the row of -nz/2 stays zero
      x[p] = (p == 2 * A / 3 && kb == 0) ? czero<C>() : src[(size_t)row * nxh];
    }
    dft_reg<+1, true, A, R>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) T[(kb * A + p) * CT + c] = x[p];
  }
  __syncthreads();
  C* yb = a.y + (size_t)b * a.ny * 6 * MZ * nxh;
  for (int w = threadIdx.x; w < A * CT; w += NT) {
    const int c = w % CT, ka = w / CT, g = c0 + c;
    if (g >= cols) continue;
    C x[B];
    C tw[log2i(B)];
    load_tw<B, A>(tw, a.tw_mz + ka);
#pragma unroll
    for (int s = 0; s < B; ++s) x[s] = T[(s * A + ka) * CT + c];
    dft_tw<B, R>(x, tw);
    C* dst = yb + (size_t)(g / nxh) * MZ * nxh + g % nxh;
#pragma unroll
    for (int s = 0; s < B; ++s) dst[(size_t)(ka + A * s) * nxh] = x[s];
  }
}

template <typename R, int MX, int NPR, int NT>
__global__ void __launch_bounds__(NT, x_ctas<R>(MX)) xpass_kernel(PlaneArgs<R> a) {
  using C = typename cpx<R>::T;
  constexpr int A = x_line_a<R>(MX), B = x_line_b<R>(MX), A1 = x_stride<R>(MX), LS = x_line<R>(MX), NXH = MX / 3;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* X = reinterpret_cast<C*>(smem_raw);  // [6][NPR][LS]: [B][A1] in use
  const int b = blockIdx.y, hz = a.mz / 2;
  if (a.active && !a.active[b]) return;
  const int npairs = a.ny * hz, g0 = blockIdx.x * NPR;  // row pair (j, m), m fastest
  C* yb = a.y + (size_t)b * a.ny * 6 * a.mz * NXH;
  auto rows = [&](int g, int f) { return yb + ((size_t)(g / hz * 6 + f) * a.mz + 2 * (g % hz)) * NXH; };
  // every read of this CTA's rows happens before the first barrier; the rows
  // of H are written over fields 0..2 of the same rows at the end
  for (int w = threadIdx.x; w < 6 * NPR * B; w += NT) {
    const int kb = w % B, line = w / B, g = g0 + line % NPR;
    if (g >= npairs) continue;
    const C* r1 = rows(g, line / NPR);
    const C* r2 = r1 + NXH;
    C x[A];
#pragma unroll
    for (int p = 0; p < A / 3; ++p) {
      const C u = r1[B * p + kb], v = r2[B * p + kb];
      x[p] = (p == 0 && kb == 0) ? mk(u.x, v.x) : mk(u.x - v.y, u.y + v.x);
    }
#pragma unroll
    for (int p = 2 * A / 3; p < A; ++p) {
      const int k = MX - (B * p + kb);  // Hermitian half; k = nxh (the Nyquist mode) stays zero
      if (p == 2 * A / 3 && kb == 0) {
        x[p] = czero<C>();
      } else {
        const C u = r1[k], v = r2[k];
        x[p] = mk(u.x + v.y, v.x - u.y);
      }
    }
    dft_reg<+1, true, A, R>(x);
#pragma unroll
    for (int p = 0; p < A; ++p) X[line * LS + kb * A1 + p] = x[p];
  }
  __syncthreads();
  if constexpr (B <= 4 || (B == 8 && sizeof(R) == 4)) {
    // second half of the inverse lines, products and first half of the forward
    // lines at the points ka + A kb of one row pair (real parts: first row,
    // imaginary parts: second row); each thread reads and writes its own slots
    for (int w = threadIdx.x; w < NPR * A; w += NT) {
      const int ka = w % A, pp = w / A;
      if (g0 + pp >= npairs) continue;
      C tw[log2i(B)];
      load_tw<B, A>(tw, a.tw_x + ka);
      C* slot = X + pp * LS + ka;
      constexpr int FS = NPR * LS;
      C v[6][B];
#pragma unroll
      for (int f = 0; f < 6; ++f) {
#pragma unroll
        for (int s = 0; s < B; ++s) v[f][s] = slot[f * FS + s * A1];
        dft_tw<B, R>(v[f], tw);
      }
      C h[3][B];
#pragma unroll
      for (int s = 0; s < B; ++s) {
        const C u = v[0][s], vv = v[1][s], ww = v[2][s], ox = v[3][s], oy = v[4][s], oz = v[5][s];
        h[0][s] = mk(vv.x * oz.x - ww.x * oy.x, vv.y * oz.y - ww.y * oy.y);
        h[1][s] = mk(ww.x * ox.x - u.x * oz.x, ww.y * ox.y - u.y * oz.y);
        h[2][s] = mk(u.x * oy.x - vv.x * ox.x, u.y * oy.y - vv.y * ox.y);
      }
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        dft_pow2<-1, B, R>(h[f]);
        slot[f * FS] = h[f][0];
#pragma unroll
        for (int s = 1; s < B; ++s) slot[f * FS + s * A1] = cmul(h[f][s], cconj(a.tw_x[s * A + ka]));
      }
    }
  } else {
    // longer lines: field by field in place, the products point by point (six
    // lines of B points would take 200 registers in FP64)
    constexpr int FS = NPR * LS;
    for (int w = threadIdx.x; w < 6 * NPR * A; w += NT) {
      const int ka = w % A;
      C* slot = X + (w / A) * LS + ka;
      C v[B], tw[log2i(B)];
      load_tw<B, A>(tw, a.tw_x + ka);
#pragma unroll
      for (int s = 0; s < B; ++s) v[s] = slot[s * A1];
      dft_tw<B, R>(v, tw);
#pragma unroll
      for (int s = 0; s < B; ++s) slot[s * A1] = v[s];
    }
    __syncthreads();
    for (int w = threadIdx.x; w < NPR * B * A; w += NT) {
      C* L = X + (w / (A * B)) * LS + (w / A % B) * A1 + w % A;
      const C u = L[0], vv = L[FS], ww = L[2 * FS], ox = L[3 * FS], oy = L[4 * FS], oz = L[5 * FS];
      L[0] = mk(vv.x * oz.x - ww.x * oy.x, vv.y * oz.y - ww.y * oy.y);
      L[FS] = mk(ww.x * ox.x - u.x * oz.x, ww.y * ox.y - u.y * oz.y);
      L[2 * FS] = mk(u.x * oy.x - vv.x * ox.x, u.y * oy.y - vv.y * ox.y);
    }
    __syncthreads();
    for (int w = threadIdx.x; w < 3 * NPR * A; w += NT) {
      const int ka = w % A;
      C* slot = X + (w / A) * LS + ka;
      C v[B];
#pragma unroll
      for (int s = 0; s < B; ++s) v[s] = slot[s * A1];
      dft_pow2<-1, B, R>(v);
      slot[0] = v[0];
#pragma unroll
      for (int s = 1; s < B; ++s) slot[s * A1] = cmul(v[s], cconj(a.tw_x[s * A + ka]));
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < 3 * NPR * B; w += NT) {
    const int s = w % B, line = w / B;
    C* slot = X + line * LS + s * A1;
    C x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) x[p] = slot[p];
    dft_reg<-1, false, A, R>(x);
#pragma unroll
    for (int p = 0; p < A; ++p)
      if (p < A / 3 || p >= 2 * A / 3) slot[p] = x[p];  // k = B p + s
  }
  __syncthreads();
  for (int w = threadIdx.x; w < 3 * NPR * NXH; w += NT) {
    const int i = w % NXH, line = w / NXH, g = g0 + line % NPR;
    if (g >= npairs) continue;
    const int im = i == 0 ? 0 : MX - i;
    const C zk = X[line * LS + (i % B) * A1 + i / B];
    const C zm = X[line * LS + (im % B) * A1 + im / B];
    C* dst = rows(g, line / NPR);
    dst[i] = mk(zk.x + zm.x, zk.y - zm.y);  // twice the rows: the last pass scales by half as much
    dst[NXH + i] = mk(zk.y + zm.y, zm.x - zk.x);
  }
}

template <typename R, int MZ>
__global__ void __launch_bounds__(z_threads<R>(MZ)) zpass_forward_kernel(PlaneArgs<R> a) {
  using C = typename cpx<R>::T;
  constexpr int A = line_a(MZ), B = line_b(MZ), CT = z_cols<R>(), NT = z_threads<R>(MZ);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* T = reinterpret_cast<C*>(smem_raw);  // [B][A][CT]
  const int b = blockIdx.y, nxh = a.nxh;
  if (a.active && !a.active[b]) return;
  const int cols = a.ny * 3 * nxh, c0 = blockIdx.x * CT;  // column (j, f, i), i fastest
  const C* yb = a.y + (size_t)b * a.ny * 6 * MZ * nxh;
  for (int w = threadIdx.x; w < A * CT; w += NT) {
    const int c = w % CT, ka = w / CT, g = c0 + c;
    if (g >= cols) continue;
    const int jf = g / nxh;
    const C* src = yb + (size_t)(jf / 3 * 6 + jf % 3) * MZ * nxh + g % nxh;
    C x[B];
#pragma unroll
    for (int s = 0; s < B; ++s) x[s] = src[(size_t)(ka + A * s) * nxh];
    dft_pow2<-1, B, R>(x);
    T[ka * CT + c] = x[0];
#pragma unroll
    for (int s = 1; s < B; ++s) T[(s * A + ka) * CT + c] = cmul(x[s], cconj(a.tw_mz[s * A + ka]));
  }
  __syncthreads();
  for (int w = threadIdx.x; w < B * CT; w += NT) {
    const int c = w % CT, s = w / CT, g = c0 + c;
    if (g >= cols) continue;
    const int i = g % nxh, jf = g / nxh, f = jf % 3, j = jf / 3;
    C x[A];
#pragma unroll
    for (int p = 0; p < A; ++p) x[p] = T[(s * A + p) * CT + c];
    dft_reg<-1, false, A, R>(x);
    C* dst = a.h + b * a.hb + f * a.qf + j * a.qj + i;
    const R sc = (R)0.5 * a.scale;
#pragma unroll
    for (int p = 0; p < A / 3; ++p) dst[(size_t)(B * p + s) * nxh] = sc * x[p];
#pragma unroll
    for (int p = 2 * A / 3; p < A; ++p) {
      const int row = B * p + s - MZ / 3;
      dst[(size_t)row * nxh] = (p == 2 * A / 3 && s == 0) ? czero<C>() : sc * x[p];
    }
  }
}

template <typename R, int MZ>
cudaError_t zpass_inverse_m(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  constexpr int CT = z_cols<R>(), NT = z_threads<R>(MZ);
  constexpr size_t smem = (size_t)MZ * CT * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(zpass_inverse_kernel<R, MZ>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(zpass_inverse_kernel<R, MZ>, dim3((a.ny * 6 * a.nxh + CT - 1) / CT, B),
                                       dim3(NT), smem, st, a);
}
template <typename R, int MZ>
cudaError_t zpass_forward_m(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  constexpr int CT = z_cols<R>(), NT = z_threads<R>(MZ);
  constexpr size_t smem = (size_t)MZ * CT * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(zpass_forward_kernel<R, MZ>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(zpass_forward_kernel<R, MZ>, dim3((a.ny * 3 * a.nxh + CT - 1) / CT, B),
                                       dim3(NT), smem, st, a);
}
template <typename R, int MX>
cudaError_t xpass_m(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  constexpr int NPR = x_pairs(MX), NT = x_threads<R>(MX);
  constexpr size_t smem = (size_t)6 * NPR * x_line<R>(MX) * sizeof(typename cpx<R>::T);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(xpass_kernel<R, MX, NPR, NT>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(xpass_kernel<R, MX, NPR, NT>, dim3((a.ny * (a.mz / 2) + NPR - 1) / NPR, B),
                                       dim3(NT), smem, st, a);
}

}  // namespace chdns

// explicit instantiations of the three passes for one padded length
#define CH_PASS_INSTANTIATE(R, M)                                                      \
  namespace chdns {                                                                    \
  template cudaError_t zpass_inverse_m<R, M>(const PlaneArgs<R>&, int, cudaStream_t);  \
  template cudaError_t zpass_forward_m<R, M>(const PlaneArgs<R>&, int, cudaStream_t);  \
  template cudaError_t xpass_m<R, M>(const PlaneArgs<R>&, int, cudaStream_t);          \
  }
