// Launchers of the step-kernel instantiations, shared by their translation units.
#pragma once

#include "corde_step.cuh"
#include "corde_variants.cuh"

namespace corde {

template <int EPT, int NT>
cudaError_t launch_step(const StepArgs& a, int n_blocks, cudaStream_t s) {
  constexpr int smem = step_smem_bytes<EPT, NT>();
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(step_kernel<EPT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(step_kernel<EPT, NT>, dim3(n_blocks), dim3(NT), smem, s, a.pdl, 0, a.rods, a.work, a.x4,
                       a.v4, a.q4, a.o4, a.u4, a.k4, a.drive, a.n_steps, a.traj, a.n_elem, a.mb, a.pos_out);
}

template <int EPT, int NT>
cudaError_t preload_step() {
  cudaFuncAttributes at;
  return cudaFuncGetAttributes(&at, step_kernel<EPT, NT>);
}

template <int EPT, int NT>
constexpr StepVariant step_variant() {
  return {EPT, NT, step_smem_bytes<EPT, NT>(), &launch_step<EPT, NT>, &preload_step<EPT, NT>};
}

}  // namespace corde
