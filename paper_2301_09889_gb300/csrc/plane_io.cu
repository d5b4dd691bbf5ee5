// Launchers of the unpadded transforms (plane_io.cuh).
#include "plane_io.cuh"

namespace chdns {

// Transforms by lines where both lengths are built and the planes of the batch
// give them enough lines; small planes keep the direct sums, whose single launch
// and shorter chains win there (us of a step's small kernels, sums / lines:
// 16x16 49.4 / 51.5 at 16 environments and 60.0 / 54.5 at 64, 8x12 49.8 / 50.3 at
// 64 and 51.3 / 52.4 at 100; 32x32 61.9 / 56.9 at eight, 128x64 114 / 77).
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

template <int N, int W>
static cudaError_t obs_z(const Grid& g, int B, double2* planes, const DevTables& t, const int* active, cudaStream_t st) {
  obs_z_kernel<N, W><<<dim3((2 * g.nxh + W - 1) / W, B), 32, 0, st>>>(g.nxh, planes, t.tw_nz, active);
  return cudaGetLastError();
}
template <int N, int W>
constexpr size_t pairs_smem() { return (size_t)W * io_b(N) * (io_a(N) | 1) * sizeof(double2); }
template <int N, int W>
static cudaError_t obs_x(const Grid& g, int B, const double2* planes, const DevTables& t, double* out, size_t out_stride,
                         const int* active, cudaStream_t st) {
  obs_x_kernel<N, W><<<dim3((g.nz + W - 1) / W, B), kIoNT, pairs_smem<N, W>(), st>>>(g.nz, planes, t.tw_nx, out, out_stride,
                                                                                    active);
  return cudaGetLastError();
}
template <int N, int W>
static cudaError_t act_x(const Grid& g, int B, const double* act, double u_tau, const DevTables& t, const PencilBufs& pb,
                         cudaStream_t st) {
  // pb.planes is free at this point of the step: the scratch plane
  act_x_kernel<N, W><<<dim3((g.nz / 2 + W - 1) / W, B), kIoNT, pairs_smem<N, W>(), st>>>(
      g.nz, act, u_tau, t.tw_nx, pb.planes, pb.vw_old, pb.vw_new, pb.tau_acc, pb.active);
  return cudaGetLastError();
}
template <int N, int W>
static cudaError_t act_z(const Grid& g, int B, const DevTables& t, const PencilBufs& pb, cudaStream_t st) {
  act_z_kernel<N, W><<<dim3((g.nxh + W - 1) / W, B), 32, 0, st>>>(g.nx, pb.planes, t.tw_nz, pb.vw_new, pb.active);
  return cudaGetLastError();
}

// eight lines per CTA once the batch has as many tiles as SMs
#define CH_IO_LAUNCH(len, wide, call, ...)                                   \
  switch (len) {                                                             \
    CH_IO_CASES(wide, call, __VA_ARGS__)                                     \
    default: return cudaErrorInvalidValue;                                   \
  }
#define CH_IO_CASE(N, wide, call, ...) \
  case N: e = (wide) ? call<N, 8>(__VA_ARGS__) : call<N, 2>(__VA_ARGS__); break;
#define CH_IO_CASES(w, c, ...)                                                                                     \
  CH_IO_CASE(8, w, c, __VA_ARGS__) CH_IO_CASE(12, w, c, __VA_ARGS__) CH_IO_CASE(16, w, c, __VA_ARGS__)             \
  CH_IO_CASE(24, w, c, __VA_ARGS__) CH_IO_CASE(32, w, c, __VA_ARGS__) CH_IO_CASE(48, w, c, __VA_ARGS__)            \
  CH_IO_CASE(64, w, c, __VA_ARGS__) CH_IO_CASE(96, w, c, __VA_ARGS__) CH_IO_CASE(128, w, c, __VA_ARGS__)           \
  CH_IO_CASE(192, w, c, __VA_ARGS__) CH_IO_CASE(256, w, c, __VA_ARGS__)

cudaError_t launch_obs_lines(const Grid& g, int B, double2* planes, const DevTables& t, double* out, size_t out_stride,
                             const int* active, cudaStream_t st) {
  cudaError_t e;
  CH_IO_LAUNCH(g.nz, (long)B * 2 * g.nxh >= 8 * 152, obs_z, g, B, planes, t, active, st)
  if (e != cudaSuccess) return e;
  CH_IO_LAUNCH(g.nx, (long)B * g.nz >= 8 * 152, obs_x, g, B, planes, t, out, out_stride, active, st)
  return e;
}

cudaError_t launch_action_lines(const Grid& g, int B, const double* act, double u_tau, const DevTables& t,
                                const PencilBufs& pb, cudaStream_t st) {
  cudaError_t e;
  CH_IO_LAUNCH(g.nx, (long)B * g.nz / 2 >= 8 * 152, act_x, g, B, act, u_tau, t, pb, st)
  if (e != cudaSuccess) return e;
  CH_IO_LAUNCH(g.nz, (long)B * g.nxh >= 8 * 152, act_z, g, B, t, pb, st)
  return e;
}

}  // namespace chdns
