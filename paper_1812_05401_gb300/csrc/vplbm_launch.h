// Host-side launchers of the per-storage kernel instantiations.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "vplbm_params.h"

namespace vplbm {

// Launch that may start while the previous kernel on the stream still runs:
// the kernel calls pdl_wait() before its first access to memory that earlier
// work writes, and pdl_trigger() to let its own successor start. Behind other
// stream work (a copy, a kernel without a trigger) it is an ordinary launch.
template <class... Params, class... Args>
cudaError_t launch_pdl_smem(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                            Args&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <class... Params, class... Args>
cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t st, Args&&... args) {
  return launch_pdl_smem(kernel, grid, block, 0, st, std::forward<Args>(args)...);
}

#define VPLBM_DECLARE_LAUNCHERS(SUFFIX)                                                         \
  cudaError_t launch_fused_##SUFFIX(int coll, const StepParams& p, cudaStream_t st);            \
  cudaError_t launch_node_##SUFFIX(int coll, const StepParams& p, cudaStream_t st);             \
  cudaError_t launch_group_##SUFFIX(const StepParams* d_params,                                 \
                                    const GroupTile* d_table, int n_blocks, long long k,         \
                                    int mode, cudaStream_t st);                                 \
  cudaError_t launch_moments_##SUFFIX(const StepParams& p, double* rho, double* ux, double* uy, \
                                      cudaStream_t st);                                         \
  cudaError_t launch_momentum_exchange_##SUFFIX(const StepParams& p, const MeArgs& m,            \
                                                cudaStream_t st);                               \
  cudaError_t launch_init_##SUFFIX(const StepParams& p, void* dst, const double* u, double rho0, \
                                   double u0x, double u0y, cudaStream_t st);                    \
  cudaError_t launch_ghost_init_##SUFFIX(const StepParams& p, const void* src, void* ghost,     \
                                        void* z, cudaStream_t st);                              \
  cudaError_t launch_export_##SUFFIX(const StepParams& p, const void* src, double* f,           \
                                     cudaStream_t st);                                          \
  cudaError_t launch_import_##SUFFIX(const StepParams& p, void* dst, const double* f,           \
                                     cudaStream_t st);

VPLBM_DECLARE_LAUNCHERS(f64)
VPLBM_DECLARE_LAUNCHERS(f32)
VPLBM_DECLARE_LAUNCHERS(f16)
VPLBM_DECLARE_LAUNCHERS(bf16)

// Two steps in one launch (FP32, two-rate collision, tiles of kPairRows rows);
// prepare: once per device before the first launch.
cudaError_t prepare_pair_f32();
cudaError_t launch_pair_f32(const PairParams& pp, cudaStream_t st);

}  // namespace vplbm
