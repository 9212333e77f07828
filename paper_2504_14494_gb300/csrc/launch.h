// Internal launchers shared between the kernel files and the C ABI layer.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace lbmgnn {

// Launch that, with `early`, may start before the preceding kernel on `st` has
// completed; the kernel waits for it in dep_wait() (common.cuh).  Early only
// while the kernels of a call need one CTA per SM: the shared-memory split of
// an SM cannot change under a running CTA, so the CTAs of a kernel that wants
// two per SM, started early, ran one per SM (1024^2 GNN-LBM step 599 us
// against 546; 64^2, one CTA per SM: 23 against 35).
template <typename... Params, typename... Args>
inline cudaError_t launch_after(bool early, void (*kern)(Params...), unsigned grid, unsigned block,
                                size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

// SMs of the current device; 0: unknown.
int sm_count();

// Blocks of a single step of these buffers (each ends in 5 atomics with totals).
int64_t bgk_step_blocks(const float* fin, const float* fout, const Shape& s);
cudaError_t launch_bgk_step(const float* fin, float* fout, const Shape& s, float tau,
                            const float* taus, double* totals, cudaStream_t st);
// The step restricted to lattice rows row0 .. row1-1 (of the nb*ny rows).
cudaError_t launch_bgk_step_rows(const float* fin, float* fout, const Shape& s, float tau,
                                 const float* taus, double* totals, int64_t row0, int64_t row1,
                                 cudaStream_t st);
// nsteps >= 2 BGK steps with the state kept on chip between steps
// (multi_step.cu); ftmp: ping-pong buffer as in lbm_step_bgk; totals of the last
// state (cleared by the caller) or NULL.
cudaError_t launch_bgk_steps(const float* fin, float* fout, float* ftmp, const Shape& s, float tau,
                             const float* taus, int nsteps, double* totals, cudaStream_t st);
// The same for the channel step, for calls that channel_steps_fit() accepts.
bool channel_steps_fit(const Shape& s, int nsteps, cudaStream_t st);
cudaError_t launch_channel_steps(const float* fin, float* fout, const Shape& s, float tau,
                                 const float* taus, float gx, int nsteps, cudaStream_t st);
cudaError_t launch_moments(const float* f, const Shape& s, float* rho, float* ux, float* uy,
                           double* totals, cudaStream_t st);
cudaError_t launch_tgv_init(float* f, const Shape& s, double rho0, double u0, double kx,
                            double ky, int pc, cudaStream_t st);

cudaError_t launch_channel_step(const float* fin, float* fout, const Shape& s, float tau,
                                const float* taus, float gx, double* totals, cudaStream_t st);
cudaError_t launch_stream(const float* fin, float* fout, const Shape& s, cudaStream_t st);
cudaError_t launch_restrict(const float* ff, const Shape& fs, float* fc, const Shape& cs, int m,
                            float tau_f, const float* taus_f, float tau_c, const float* taus_c,
                            cudaStream_t st);
cudaError_t launch_tgv_init_batch(float* f, const Shape& s, const double* prm, int pc,
                                  cudaStream_t st);

}  // namespace lbmgnn
