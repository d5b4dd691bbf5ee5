// Dispatch of the three-pass nonlinear term (plane_pass.cuh) by padded length.
// Each length is compiled for the z passes and the x pass, in both
// precisions, in plane_pass_*.cu.
#include "common.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace chdns {

template <typename R, int MZ> cudaError_t zpass_inverse_m(const PlaneArgs<R>&, int, cudaStream_t);
template <typename R, int MZ> cudaError_t zpass_forward_m(const PlaneArgs<R>&, int, cudaStream_t);
template <typename R, int MX> cudaError_t xpass_m(const PlaneArgs<R>&, int, cudaStream_t);

// Planes whose padded lengths are both built run in passes, but for planes
// of 16 x 16 modes, which fit one CTA (plane_small.cu, plane.cu).
bool passes_built(int mx, int mz) {
  auto built = [](int m) {
    switch (m) {
#define X(M) case M:
      CH_LINE_LENGTHS(X)
#undef X
      return true;
      default: return false;
    }
  };
  return built(mx) && built(mz) && !(mx == 24 && mz == 24);
}

template <typename R>
cudaError_t launch_plane_passes(const PlaneArgs<R>& a, int B, cudaStream_t st) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (a.mz) {
#define X(M) case M: e = zpass_inverse_m<R, M>(a, B, st); break;
    CH_LINE_LENGTHS(X)
#undef X
  }
  if (e != cudaSuccess) return e;
  switch (a.mx) {
#define X(M) case M: e = xpass_m<R, M>(a, B, st); break;
    CH_LINE_LENGTHS(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  switch (a.mz) {
#define X(M) case M: return zpass_forward_m<R, M>(a, B, st);
    CH_LINE_LENGTHS(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

template cudaError_t launch_plane_passes<double>(const PlaneArgs<double>&, int, cudaStream_t);
template cudaError_t launch_plane_passes<float>(const PlaneArgs<float>&, int, cudaStream_t);

}  // namespace chdns
