// Implicit solves of handles with many modes (stage_solve.cuh), both node
// precisions and both upper boundaries.
#include "stage_solve.cuh"

namespace chdns {

template <typename RN>
cudaError_t launch_stage_solve(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                               const typename cpx<RN>::T* h, const StageCoef& sc, cudaStream_t st) {
  return t.tau.top_bc ? solve_top<RN, 1>(g, B, pb, t, h, sc, st) : solve_top<RN, 0>(g, B, pb, t, h, sc, st);
}

template cudaError_t launch_stage_solve<double>(const Grid&, int, const PencilBufs&, const DevTables&, const double2*,
                                                const StageCoef&, cudaStream_t);
template cudaError_t launch_stage_solve<float>(const Grid&, int, const PencilBufs&, const DevTables&, const float2*,
                                               const StageCoef&, cudaStream_t);

}  // namespace chdns
