// Per-MH and per-order launchers of the stage kernels.  MH bounds the
// per-thread register arrays (unknowns of one parity); each bucket and each
// group of Chebyshev orders is compiled in its own translation unit
// (stage_mh*.cu, stage_dct_*.cu) so that the instantiations build in parallel.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"

namespace chdns {

template <typename RN, int MH>
cudaError_t post_mh(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, const typename cpx<RN>::T* h,
                    const StageCoef& sc, int ppc, size_t smem, cudaStream_t st);
// direct sums (stage_direct.cu); pitches of their cosine tables
template <typename RN>
cudaError_t launch_pre_direct(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q,
                              cudaStream_t st);
cudaError_t launch_pre_few(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, double2* q, cudaStream_t st);
template <typename RN>
cudaError_t launch_analysis_direct(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                                   const typename cpx<RN>::T* hn, typename cpx<RN>::T* hc, cudaStream_t st);
// register cosine transforms (stage_dct.cuh)
template <typename RN, int N>
cudaError_t pre_dct_n(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, typename cpx<RN>::T* q,
                      cudaStream_t st);
template <typename RN, int N>
cudaError_t analysis_dct_n(const Grid& g, int B, const PencilBufs& pb, typename cpx<RN>::T* h, cudaStream_t st);
// implicit solves of handles with many modes (stage_solve.cu)
template <typename RN>
cudaError_t launch_stage_solve(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                               const typename cpx<RN>::T* h, const StageCoef& sc, cudaStream_t st);

}  // namespace chdns
