// The fused step on D3Q19 (Sec. II-C, "Lattice-agnostic construction and the D3Q19
// example"): instantiations of the kernels of step_kernels.cuh with the collision of d3q19.cuh.
#include "step_kernels.cuh"

namespace flbm {

cudaError_t launch_step_d3q19(int storage, int variant, int parity, bool noise, bool shear, const StepArgs &a,
                              cudaStream_t s) {
  if (storage == 0) return launch_rates<19, float, false>(variant, parity, noise, shear, a, s);
  if (storage == 1) return launch_rates<19, __nv_bfloat16, false>(variant, parity, noise, shear, a, s);
  return launch_rates<19, __half, false>(variant, parity, noise, shear, a, s);
}

}  // namespace flbm
