// Launchers of the unpadded transforms (plane_io.cuh).
#include "plane_io.cuh"

namespace chdns {

// Transforms by lines where both lengths are built and the planes of the
// batch give them enough lines; small planes keep the direct sums, whose
// single launch and shorter chains win there.
bool io_by_lines(const Grid& g, int B) {
  auto built = [](int n) {
    switch (n) {
#define X(N) case N:
      CH_IO_LENGTHS(X)
#undef X
      return true;
      default: return false;
    }
  };
  return built(g.nx) && built(g.nz) && (long)B * g.nx * g.nz >= 8192;
}

static size_t pairs_smem(int n) { return (size_t)kIoPairs * io_b(n) * (io_a(n) | 1) * sizeof(double2); }

cudaError_t launch_obs_lines(const Grid& g, int B, double2* planes, const DevTables& t, double* out, size_t out_stride,
                             const int* active, cudaStream_t st) {
  const dim3 gz((2 * g.nxh + kIoCols - 1) / kIoCols, B), gx((g.nz + kIoPairs - 1) / kIoPairs, B);
  switch (g.nz) {
#define X(N) case N: obs_z_kernel<N><<<gz, 32, 0, st>>>(g.nxh, planes, t.tw_nz, active); break;
    CH_IO_LENGTHS(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  switch (g.nx) {
#define X(N) case N: obs_x_kernel<N><<<gx, kIoNT, pairs_smem(N), st>>>(g.nz, planes, t.tw_nx, out, out_stride, active); break;
    CH_IO_LENGTHS(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_action_lines(const Grid& g, int B, const double* act, double u_tau, const DevTables& t,
                                const PencilBufs& pb, cudaStream_t st) {
  double2* tx = pb.planes;  // free at this point of the step
  const dim3 gx((g.nz / 2 + kIoPairs - 1) / kIoPairs, B), gz((g.nxh + kIoCols - 1) / kIoCols, B);
  switch (g.nx) {
#define X(N)                                                                                                     \
  case N:                                                                                                        \
    act_x_kernel<N><<<gx, kIoNT, pairs_smem(N), st>>>(g.nz, act, u_tau, t.tw_nx, tx, pb.vw_old, pb.vw_new,        \
                                                      pb.tau_acc, pb.active);                                    \
    break;
    CH_IO_LENGTHS(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  switch (g.nz) {
#define X(N) case N: act_z_kernel<N><<<gz, 32, 0, st>>>(g.nx, tx, t.tw_nz, pb.vw_new, pb.active); break;
    CH_IO_LENGTHS(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace chdns
