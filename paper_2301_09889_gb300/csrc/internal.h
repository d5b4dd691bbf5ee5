// Host-side declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace chdns {

template <typename R>
cudaError_t launch_plane(const PlaneArgs<R>& a, int B, size_t smem, cudaStream_t st);
template <typename R>
cudaError_t plane_max_clusters(const PlaneArgs<R>& a, size_t smem, int* clusters);
// nonlinear term of planes of 16 x 16 modes, line transforms in registers (plane_small.cu)
bool plane16_shape(int mx, int mz, int nxh, int nz);
template <typename R>
cudaError_t launch_plane16(const PlaneArgs<R>& a, int B, cudaStream_t st);
// nonlinear term in three passes through global memory (plane_pass.cu)
bool passes_built(int mx, int mz);
template <typename R>
cudaError_t launch_plane_passes(const PlaneArgs<R>& a, int B, cudaStream_t st);

struct PencilBufs {
  double2 *V, *G;               // [B][ny][P]
  double2 *HVP, *HGP;           // [B][ny][P] complex in the node precision (FP32 pairs in mixed mode)
  float2 *V32, *G32;            // [B][ny][P] V and G rounded to FP32 (mixed precision): what stage_pre reads;
                                // mode 0 of G32 holds the mean flow (W, U), that of V32 (DW, DU)
  double *UM, *WM, *HXP, *HZP;  // [B][ny]
  // node values of u, v, w, ox, oy, oz in the node precision, then those of H (or
  // its coefficients) over the first three: strides Grid.qf, qj, qb.  Where the
  // nonlinear term runs in passes a node's fields are [6][mz][nxh], the
  // first nz rows of each in use, so that the z transforms run in place;
  // otherwise [6][ny][P].  (A step so holds no array beside the six fields:
  // 9 ny P values with passes, 6 ny P without)
  double2* Q;
  double2 *vw_old, *vw_new;     // [B][P] wall-velocity spectra
  double2* planes;              // [B][2][P] u, v spectra at the sensing node
  double* tau_acc;              // [B]
  const int* active;            // [B] slots advanced by this step (nullptr: all)
};

struct DevTables {
  const double* kx;    // [nxh]
  const double* kz;    // [nz]
  const double* cheb;  // [ny][ny] cos(pi j n / N)
  const float* cheb_f; // the same table in FP32 (mixed precision)
  const double* dts;   // [ny] T_n'(y_js) at the sensing node
  // direct sums, in the node precision (cos_ana for orders without a register
  // transform, cos_pre for these and the few-mode form): cos(pi j n / N) as
  // [n][j <= N/2, padded] and as [j <= N/2][parity of n][i, padded], n = 2 i + parity
  const double *cos_pre, *cos_ana;
  const float *cos_pre_f, *cos_ana_f;
  TauTables tau;
  const double2* tw_nx;  // [nx]
  const double2* tw_nz;  // [nz]
};

// wall-normal halves of a stage (stage.cu)
size_t stage_post_smem(const Grid& g, int Mh, int ppc);  // per-tile implicit half, ppc modes per CTA
// direct Chebyshev sums (no register cosine transform for this order): the
// handle needs their tables, of these pitches
bool stage_direct(const Grid& g);
// FP64 handles whose explicit half runs as direct sums spread over the GPU
bool pre_few(const Grid& g, int B);
int direct_pre_pitch(int N);
int direct_ana_pitch(int N);
// kernels one launch_stage_post issues
int stage_post_launches(int top, bool batched);
template <typename RN>
cudaError_t launch_stage_pre(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                             typename cpx<RN>::T* q, cudaStream_t st);
// batched (and every handle under a free-slip top): the analysis of H over its
// nodal values h in place, then one thread per (mode, class, component,
// equation); otherwise sixteen lanes per system on a shared-memory tile of ppc modes
template <typename RN>
cudaError_t launch_stage_post(const Grid& g, int B, const PencilBufs& pb, const DevTables& t,
                              typename cpx<RN>::T* h, const StageCoef& sc, int ppc, bool batched,
                              cudaStream_t st);
// V32, G32 of one environment from V, G (after its state has been set)
cudaError_t launch_round_state(const Grid& g, int b, const PencilBufs& pb, cudaStream_t st);
cudaError_t launch_wall_shear(const Grid& g, int B, const double* UM, double nu, double* acc,
                              const int* active, cudaStream_t st);
cudaError_t launch_sense(const Grid& g, int B, const PencilBufs& pb, const DevTables& t, int js,
                         double alpha, int opposition, cudaStream_t st);
cudaError_t launch_obs(const Grid& g, int B, double2* planes, const DevTables& t, double* out,
                       size_t out_stride, const int* active, cudaStream_t st);
cudaError_t launch_action(const Grid& g, int B, const double* act, double u_tau, const DevTables& t,
                          const PencilBufs& pb, cudaStream_t st);
// the unpadded transforms by lines (plane_io.cu), chosen by size in launch_obs
// and launch_action: two launches each
bool io_by_lines(const Grid& g, int B);
cudaError_t launch_obs_lines(const Grid& g, int B, double2* planes, const DevTables& t, double* out, size_t out_stride,
                             const int* active, cudaStream_t st);
cudaError_t launch_action_lines(const Grid& g, int B, const double* act, double u_tau, const DevTables& t,
                                const PencilBufs& pb, cudaStream_t st);
cudaError_t launch_finalize(int B, const double* acc, double inv_steps, double tau_ref, double* out,
                            size_t out_stride, size_t out_offset, const int* active, cudaStream_t st);
cudaError_t launch_tau_helmholtz(int ny, int M, const double* lam, const double2* r, const double2* top,
                                 const double2* bot, double2* f, cudaStream_t st);

// on-device policy (policy.cu): a multilayer perceptron shared by every agent
constexpr int kPolicyMaxWidth = 64;
constexpr int kPolicyMaxWindow = 7;
// weights of the largest network: 2 (7 x 7) inputs, two hidden layers of 64
constexpr int kPolicyMaxWeights =
    kPolicyMaxWidth * 2 * kPolicyMaxWindow * kPolicyMaxWindow + kPolicyMaxWidth +
    kPolicyMaxWidth * kPolicyMaxWidth + kPolicyMaxWidth + kPolicyMaxWidth + 1;
struct PolicyDesc {
  int wz, wx;      // observation window (odd)
  int n_hidden;    // 0, 1 or 2 ReLU layers
  int h1, h2;      // hidden widths
  int out_tanh;    // 1: action = u_tau tanh(y)
  int n_weights;   // FP32 values at w
};
int policy_weight_count(const PolicyDesc& d);
// plane [B][2][nz][nx] (u, v on the sensing plane) -> act [B][nz][nx]
cudaError_t launch_policy(int nx, int nz, int B, const PolicyDesc& d, const float* w, const double* plane,
                          double* act, double u_tau, const int* active, cudaStream_t st);

}  // namespace chdns

struct ch_env;
namespace chdns {
// internal entry points of api.cu used by the serving layer
int step_masked(ch_env* env, const double* d_action, const int* d_active, const int* h_active);
double* env_dout(ch_env* env);
double* env_dact(ch_env* env);
size_t env_out_stride(const ch_env* env);
cudaStream_t env_stream(const ch_env* env);
int env_slot_seed(ch_env* env, int e, uint64_t seed, double amplitude, int kmax);
size_t env_footprint(const struct ch_params* p);
}  // namespace chdns
