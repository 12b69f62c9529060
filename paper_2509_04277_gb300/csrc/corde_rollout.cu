// Recorded rollouts (rod_rollout) on the adjoint's two-element layout: all steps and their
// checkpoints in one launch.  A launch and a state copy per checkpoint segment cost 7 us each: 200
// steps of 256 nodes with a checkpoint every 20 took 0.66 ms for one rod and 0.68 ms for 256.
#include "corde_step.cuh"
#include "corde_variants.cuh"

namespace corde {

template <int NT>
static cudaError_t launch_t(const StepArgs& a, int n_blocks, cudaStream_t s) {
  constexpr int smem = step_smem_bytes<2, NT>();
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(rollout_kernel<2, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(rollout_kernel<2, NT>, dim3(n_blocks), dim3(NT), smem, s, a.pdl, 0, a.rods, a.work, a.x4, a.v4, a.q4,
                       a.o4, a.u4, a.k4, a.drive, a.n_steps, a.traj, a.n_elem, CkptDev{a.ckpt, a.ckpt_every});
}

cudaError_t launch_rollout(int nt, const StepArgs& a, int n_blocks, cudaStream_t s) {
  switch (nt) {
    case 32: return launch_t<32>(a, n_blocks, s);
    case 64: return launch_t<64>(a, n_blocks, s);
    case 128: return launch_t<128>(a, n_blocks, s);
    case 256: return launch_t<256>(a, n_blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace corde
