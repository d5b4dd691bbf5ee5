// Dispatch of the fused stage kernels (stage_kernels.cuh) to the register-array
// bucket MH that covers one parity of the Chebyshev unknowns, and their
// shared-memory sizes.
#include "dct_reg.cuh"
#include "stage_launch.h"

namespace chdns {

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
#define CH_MH_BUCKETS(X) X(5) X(9) X(17) X(33) X(49) X(65) X(97) X(101)
static int mh_bucket(int need) {
#define X(v) if (need <= v) return v;
  CH_MH_BUCKETS(X)
#undef X
  return 0;
}

// register cosine transforms are built for this Chebyshev order
static bool dct_order(int N) {
  switch (N) {
#define X(n) case n:
    CH_DCT_ORDERS(X)
#undef X
    return true;
    default: return false;
  }
}

bool stage_direct(const Grid& g) { return !dct_order(g.N); }
// (three fields of H, the state and the previous right-hand sides of a tile of
// modes, their tables, and six complex values per mode)
size_t stage_post_smem(const Grid& g, int Mh, int ppc) {
  return ((size_t)7 * g.ny + 6) * ppc * sizeof(double2) + ((size_t)18 * Mh * ppc + 6 * ppc) * sizeof(double);
}
int stage_post_launches(int top, bool batched) { return (batched || top) ? 2 : 1; }

template <typename RN>
cudaError_t launch_stage_pre(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                             typename cpx<RN>::T* q, cudaStream_t st) {
  if constexpr (sizeof(RN) == 8) {
    if (pre_few(g, B)) return launch_pre_few(g, B, pb, t, q, st);
  }
  switch (g.N) {
#define X(n) case n: return pre_dct_n<RN, n>(g, B, pb, t, q, st);
    CH_DCT_ORDERS(X)
#undef X
    default: return launch_pre_direct<RN>(g, B, pb, t, q, st);
  }
}

// The implicit half: handles with few modes under the no-slip top run one
// kernel on tiles of modes (stage_post_kernel), all others the analysis of H
// and the solves in two launches.
template <typename RN>
cudaError_t launch_stage_post(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                              typename cpx<RN>::T* h, const StageCoef& sc, int ppc, bool batched, cudaStream_t st) {
  if (!batched && !t.tau.top_bc) {
    const size_t smem = stage_post_smem(g, t.tau.Mh, ppc);
    switch (mh_bucket(g.N / 2 + 1)) {
#define X(m) case m: return post_mh<RN, m>(g, B, pb, t, h, sc, ppc, smem, st);
      CH_MH_BUCKETS(X)
#undef X
      default: return cudaErrorInvalidValue;
    }
  }
  // the coefficients of H: over its nodal values, or (direct sums) over the node
  // values of the vorticity, which no kernel reads any more
  typename cpx<RN>::T* hc = h;
  cudaError_t e;
  switch (g.N) {
#define X(n) case n: e = analysis_dct_n<RN, n>(g, B, pb, h, st); break;
    CH_DCT_ORDERS(X)
#undef X
    default:
      hc = h + 3 * g.qf;
      e = launch_analysis_direct<RN>(g, B, pb, t, h, hc, st);
  }
  if (e != cudaSuccess) return e;
  return launch_stage_solve<RN>(g, B, pb, t, hc, sc, st);
}

template cudaError_t launch_stage_pre<double>(const Grid&, int, const PencilBufs&, const DevTables&, double2*,
                                              cudaStream_t);
template cudaError_t launch_stage_post<double>(const Grid&, int, const PencilBufs&, const DevTables&, double2*,
                                               const StageCoef&, int, bool, cudaStream_t);
template cudaError_t launch_stage_pre<float>(const Grid&, int, const PencilBufs&, const DevTables&, float2*,
                                             cudaStream_t);
template cudaError_t launch_stage_post<float>(const Grid&, int, const PencilBufs&, const DevTables&, float2*,
                                              const StageCoef&, int, bool, cudaStream_t);

}  // namespace chdns
