// FP64 reference-path kernels for lattice D1Q3 (compiled with -fmad=false).
#include "lbm_ref_launch.cuh"
#include "lbm_ref_1d.cuh"
LBM_DEFINE_REF_LAUNCHERS(1)

namespace lbm {
cudaError_t launch_ref_steps_1d(const Ref1DArgs &r, cudaStream_t st) {
  const int core = r1_core(r.steps);
  k_steps_ref_1d<<<(r.a.n[0] + r.shift + core - 1) / core, 8 * R1_NODES, 0, st>>>(r);
  return cudaGetLastError();
}
}  // namespace lbm
