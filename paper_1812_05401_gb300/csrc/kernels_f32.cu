// Kernels for f32 population storage.
#define VPLBM_STORE vplbm::kF32
#define VPLBM_SUFFIX f32
#include "vplbm_kernels_impl.cuh"
#include "vplbm_pair.cuh"

namespace vplbm {

cudaError_t prepare_pair_f32() {
  return prepare_pair(reinterpret_cast<const void*>(pair_step_kernel<kF32>), int(sizeof(PairTile<kF32>)));
}

cudaError_t launch_pair_f32(const PairParams& pp, cudaStream_t st) {
  return launch_pdl_smem(pair_step_kernel<kF32>, dim3(pp.a.n_tiles), dim3(kLanes, warps_per_block(kF32)),
                         sizeof(PairTile<kF32>), st, pp);
}

}  // namespace vplbm
