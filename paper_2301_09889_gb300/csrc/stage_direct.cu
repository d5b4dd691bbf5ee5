// Launchers of the direct-sum lines (stage_direct.cuh).
#include "stage_direct.cuh"
#include "stage_launch.h"

namespace chdns {

// table pitches: a warp may read up to seven sums beyond the last
int direct_pre_pitch(int N) { return (N / 2 + 1 + 15) / 8 * 8; }
int direct_ana_pitch(int N) { return direct_pre_pitch(N); }

// sums per warp for `count` outputs
template <typename RN>
static int sums_per_warp(int count) {
  if (sizeof(RN) == 4) return 8;
  const int warps = (count + 7) / 8, k = (count + warps - 1) / warps;
  return k < 5 ? 5 : k;
}

template <typename RN, int K>
static cudaError_t pre_k(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q,
                         cudaStream_t st) {
  const int per = (g.N / 2 + 1 + K - 1) / K;  // warps of K node pairs
  const int z = (per + 5) / 6, nw = (per + z - 1) / z;  // up to six share the coefficients of a CTA
  const size_t smem = (size_t)g.ny * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_direct_kernel<RN, K>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(stage_pre_direct_kernel<RN, K>, dim3((g.P + 15) / 16 * 6, B, z), dim3(32 * nw), smem,
                                        st, g, pb, t, q);
}
// The few-mode form, in FP64 where its CTAs find an SM each.  Us per launch, it /
// the transforms or direct sums above: 128 modes N = 32 15.2 / 16.7, N = 48 18.9 /
// 22.5, N = 49 19.1 / 33.2, N = 64 21.1 / 28.1; 32 modes N = 128 33.5 / 49.6.  With
// twice the modes a CTA of four pairs per warp no longer gains (28.6 / 27.0 at
// 256 modes, N = 64).  Its shared memory bounds N.
static unsigned few_groups(const Grid& g) { return (g.N / 2 + kFewPairs) / kFewPairs; }
bool pre_few(const Grid& g, int B) {
  return g.N <= 128 && (long)((g.P + 15) / 16) * 6 * B * few_groups(g) <= 152;
}
cudaError_t launch_pre_few(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, double2* q, cudaStream_t st) {
  const size_t smem = (size_t)g.ny * (4 * 32 + kFewPairs + 1) * sizeof(double);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(stage_pre_few_kernel, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(stage_pre_few_kernel, dim3((g.P + 15) / 16 * 6, B, few_groups(g)), dim3(32 * kFewWarps),
                       smem, st, g, pb, t, q);
}

template <typename RN, int K>
static cudaError_t analysis_k(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, const typename cpx<RN>::T* hn,
                              typename cpx<RN>::T* hc, cudaStream_t st) {
  const int groups = (g.N / 2 + 1 + K * kAnaWarps - 1) / (K * kAnaWarps);
  const size_t smem = (size_t)(g.N / 2 + 1) * 32 * sizeof(RN);
  static SmemLimit lim;
  const cudaError_t e = raise_smem_limit(analysis_direct_kernel<RN, K>, &lim, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(analysis_direct_kernel<RN, K>, dim3((g.P + 15) / 16, B, 6 * groups),
                                        dim3(32 * kAnaWarps), smem, st, g, pb, t, hn, hc, direct_ana_pitch(g.N));
}

template <typename RN>
cudaError_t launch_pre_direct(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q,
                              cudaStream_t st) {
  if constexpr (sizeof(RN) == 8) {
    switch (sums_per_warp<RN>(g.N / 2 + 1)) {
      case 5: return pre_k<RN, 5>(g, B, pb, t, q, st);
      case 6: return pre_k<RN, 6>(g, B, pb, t, q, st);
      case 7: return pre_k<RN, 7>(g, B, pb, t, q, st);
      default: break;
    }
  }
  return pre_k<RN, 8>(g, B, pb, t, q, st);
}

template <typename RN>
cudaError_t launch_analysis_direct(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                                   const typename cpx<RN>::T* hn, typename cpx<RN>::T* hc, cudaStream_t st) {
  if constexpr (sizeof(RN) == 8) {
    switch (sums_per_warp<RN>(g.N / 2 + 1)) {
      case 5: return analysis_k<RN, 5>(g, B, pb, t, hn, hc, st);
      case 6: return analysis_k<RN, 6>(g, B, pb, t, hn, hc, st);
      case 7: return analysis_k<RN, 7>(g, B, pb, t, hn, hc, st);
      default: break;
    }
  }
  return analysis_k<RN, 8>(g, B, pb, t, hn, hc, st);
}

template cudaError_t launch_pre_direct<double>(const Grid&, int, const PencilBufs&, const DevTables&, double2*, cudaStream_t);
template cudaError_t launch_pre_direct<float>(const Grid&, int, const PencilBufs&, const DevTables&, float2*, cudaStream_t);
template cudaError_t launch_analysis_direct<double>(const Grid&, int, const PencilBufs&, const DevTables&, const double2*,
                                                    double2*, cudaStream_t);
template cudaError_t launch_analysis_direct<float>(const Grid&, int, const PencilBufs&, const DevTables&, const float2*,
                                                   float2*, cudaStream_t);

}  // namespace chdns
